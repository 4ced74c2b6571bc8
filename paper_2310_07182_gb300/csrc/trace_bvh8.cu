// trace_bvh8.cu -- closest-hit and any-hit traversal of the BVH8-Q (8-wide nodes whose
// child boxes are quantised to 8 bits, after Ylitie, Karras and Laine 2017).  Same
// primitives and closest-hit rule as the BVH2 kernels (trace_common.cuh), so both layouts
// return the same hit bit for bit.
#include <cuda_runtime.h>

#include "cr_internal.h"
#include "launch_next.cuh"
#include "trace_common.cuh"

namespace cr {
namespace {

// ------------------------------------------------------------------------------------
// BVH8-Q traversal with hit-mask node groups (the scheme of Ylitie, Karras and Laine 2017).
// Node layout (80 bytes, five 16-byte loads): w0 = origin xyz | exponent bytes + inner mask,
// w1 = first inner child, first triangle, 8 meta bytes, w2..w4 = the children's 8-bit
// low / high planes per axis.  Children sit in slots by the octant of their centroid, so
// visiting slot i ^ octant(d) for i = 0..7 goes roughly near to far without sorting.
//
// One iteration intersects one node: the 8 children are slab-tested straight from their
// bytes (one FMA per plane, with error bounds that keep the test conservative; the near and far
// words of each axis are picked by the ray's signs, so a box needs no minima and maxima of its plane
// distances); hit inner children form a bit mask in slot order, taken to visiting order by the
// ray's octant, hit leaves a mask of their triangles, which
// are tested at once.  The nearest inner child is visited next and the rest of the mask is
// pushed as one (first child, mask) entry, so the stack holds at most one entry per tree
// level.  Inner children are stored in slot order: the child in slot s is first child +
// popc(inner mask below s).
constexpr int kStack8 = (int)kBvh8StackCapacity; // >= the tree depth (checked at scene creation)

// byte i of the 8-byte field (lo, hi) as a float (exact)
template <int i>
__device__ __forceinline__ float qbyte(uint32_t lo, uint32_t hi) {
    return __uint2float_rn(((i < 4 ? lo : hi) >> (8 * (i & 3))) & 0xffu);
}

// Bit i of the result is bit i ^ oct of the 8-bit mask m; s0, s1, s2 = oct & 1, oct & 2, oct & 4.
__device__ __forceinline__ uint32_t visiting_order(uint32_t m, uint32_t s0, uint32_t s1, uint32_t s2) {
    m = ((m << s0) & 0xaau) | ((m >> s0) & 0x55u); // s = 0 leaves m as it is
    m = ((m << s1) & 0xccu) | ((m >> s1) & 0x33u);
    m = ((m << s2) & 0xf0u) | ((m >> s2) & 0x0fu);
    return m;
}

// Traversal of a warp's rays, one ray per lane; all 32 lanes call it together.
//
// What bounds it: the instructions of a node visit (eight box tests), times lanes that wait.  With
// kMore, lanes whose ray has ended take the next rays, and a lane that has hit leaves waits with
// their triangles until no more than three quarters of the warp's lanes are without (a half and a
// quarter cost 0 and 12%; not waiting 7%).  Camera rays do neither: their warps run together
// (0.51 against 0.58 ms for the interior's).
// Interior (1280x720, 4 bounces, one sample with light samples): secondary trace 4.42 ms at the start,
// 2.85 with lanes refilled, near and far words picked once per node instead of minima and maxima per
// child, and no byte reordering of the node, 2.65 with the wait; shadow rays 2.67 -> 1.39 ->
// 1.29 ms; primary 0.68 -> 0.51 ms.  Landscape secondary trace 1.75 -> 1.03 ms.
template <bool kCount, bool kAny, bool kWide, class Src>
__device__ __forceinline__ void trace_bvh8_warp(const SceneDev* __restrict__ scenes, Src& src,
                                                unsigned long long& n_node, unsigned long long& n_tri) {
    constexpr bool kWait = Src::kMore;
    const SceneDev* sc = scenes;
    const uint4* __restrict__ nodes = scenes->nodes8;
    const float4* __restrict__ tris = scenes->tris;
    RayPre r;
    uint32_t s0 = 0, s1 = 0, s2 = 0; // the octant's bits (bit set: that direction component is negative)
    int skip = -1, key = -1;
    Best best{0.0f, -1};
    float tcull = 0.0f;
    uint2 stack[kStack8];
    int sp = 0;
    uint32_t node = 0, trimask = 0, tri_base = 0;
    bool live = false, last = false;
    auto fill = [&](uint32_t alive) {
        const uint32_t i = src.take(~alive);
        if (!live) {
            if (Src::kMore && key >= 0) src.store(key, best.leaf, best.t, tris);
            key = -1;
            float4 ro, rd;
            if (i < src.n && src.load(i, key, ro, rd)) {
                sc = scenes + src.scene(key);
                nodes = sc->nodes8;
                tris = sc->tris;
                r = prep_ray(ro, rd);
                skip = __float_as_int(ro.w);
                s0 = rd.x < 0.0f ? 1u : 0u;
                s1 = rd.y < 0.0f ? 2u : 0u;
                s2 = rd.z < 0.0f ? 4u : 0u;
                best = Best{rd.w, -1};
                tcull = __fmul_rn(best.t, kCullWiden);
                sp = 0;
                node = 0;
                trimask = 0;
                live = true;
            }
        }
    };
    if (!Src::kMore) fill(0u);
    int refill = 32; // idle lanes at which rays are taken; 33: none are left
    while (true) {
        uint32_t alive = __ballot_sync(0xffffffffu, live);
        if (Src::kMore && 32 - __popc(alive) >= refill) {
            fill(alive);
            alive = __ballot_sync(0xffffffffu, live);
            if (Src::kProbe) src.probe(live, s0 | s1 | s2);
            refill = !src.more() ? 33 : alive == 0u ? 32 : src.idle;
            if (alive == 0u && refill == 32) continue; // the positions taken held no rays
        }
        if (alive == 0u) {
            if (key >= 0) src.store(key, best.leaf, best.t, tris);
            return;
        }
        const int most = (3 * __popc(alive)) >> 2;
        do {
            if (live && (!kWait || !trimask)) {
                if (kCount) ++n_node;
                CR_DBG(if (!dbg_in_range(sc, (uint32_t)node, kDbgNode, sc->n_nodes)) {
                    live = false;
                    continue;
                })
                const uint4 w0 = __ldg(&nodes[5 * (size_t)node + 0]);
                const uint4 w1 = __ldg(&nodes[5 * (size_t)node + 1]);
                const uint4 w2 = __ldg(&nodes[5 * (size_t)node + 2]);
                const uint4 w3 = __ldg(&nodes[5 * (size_t)node + 3]);
                const uint4 w4 = __ldg(&nodes[5 * (size_t)node + 4]);
                const float ox = __uint_as_float(w0.x), oy = __uint_as_float(w0.y), oz = __uint_as_float(w0.z);
                const float sx = __uint_as_float((w0.w & 0xffu) << 23);
                const float sy = __uint_as_float(((w0.w >> 8) & 0xffu) << 23);
                const float sz = __uint_as_float(((w0.w >> 16) & 0xffu) << 23);
                const uint32_t imask = w0.w >> 24;
                const uint32_t child_base = w1.x;
                tri_base = w1.y;
                const bool gx = r.ix < 0.0f, gy = r.iy < 0.0f, gz = r.iz < 0.0f; // the upper plane is the near one
                const uint32_t nx_lo = gx ? w3.z : w2.x, nx_hi = gx ? w3.w : w2.y, fx_lo = gx ? w2.x : w3.z, fx_hi = gx ? w2.y : w3.w;
                const uint32_t ny_lo = gy ? w4.x : w2.z, ny_hi = gy ? w4.y : w2.w, fy_lo = gy ? w2.z : w4.x, fy_hi = gy ? w2.w : w4.y;
                const uint32_t nz_lo = gz ? w4.z : w3.x, nz_hi = gz ? w4.w : w3.y, fz_lo = gz ? w3.x : w4.z, fz_hi = gz ? w3.y : w4.w;
                // Plane distances straight from the bytes: a plane at origin + q * step meets the ray
                // at fma(q, a, b) with a = step / d (exact, step is a power of two) and
                // b = (origin - o) / d.  Against the decoded plane fl(origin + q * step), whose box
                // the builder makes contain the child, this is off by at most a relative 2^-23 plus
                // 2^-23 |1/d| (|origin| + 255 step + |origin - o|).  b is biased, down for the entry plane
                // and up for the exit plane, by 2^-20 |1/d| times the same sum: twice that error and the
                // relative 2^-21 by which the BVH2 test used to widen the exit (a distance is at most
                // |1/d| (255 step + |origin - o|)), so no child box the decoded form would enter is
                // rejected (2^-100 more covers a step / d that falls into the subnormal range).
                const auto offsets = [](float org, float step, float o, float i, float& a, float& bn, float& bf) {
                    const float d = __fsub_rn(org, o);
                    a = __fmul_rn(step, i);
                    const float b = __fmul_rn(d, i);
                    const float e = __fmul_rn(__fmul_rn(__fadd_rn(__fadd_rn(fabsf(org), __fmul_rn(255.0f, step)), fabsf(d)),
                                                        fabsf(i)), 0x1.0p-20f) + 0x1.0p-100f;
                    bn = __fsub_rn(b, e);
                    bf = __fadd_rn(b, e);
                };
                float ax, ay, az, bnx, bfx, bny, bfy, bnz, bfz;
                offsets(ox, sx, r.ox, r.ix, ax, bnx, bfx);
                offsets(oy, sy, r.oy, r.iy, ay, bny, bfy);
                offsets(oz, sz, r.oz, r.iz, az, bnz, bfz);
                uint32_t hits = 0;
#define CR_BVH8_CHILD(i)                                                                                  \
            {                                                                                                     \
                const float tn = fmaxf(max3f(fmaf(qbyte<i>(nx_lo, nx_hi), ax, bnx), fmaf(qbyte<i>(ny_lo, ny_hi), ay, bny), \
                                             fmaf(qbyte<i>(nz_lo, nz_hi), az, bnz)), 0.0f);                       \
                const float tf = min3f(fmaf(qbyte<i>(fx_lo, fx_hi), ax, bfx), fmaf(qbyte<i>(fy_lo, fy_hi), ay, bfy), \
                                       fmaf(qbyte<i>(fz_lo, fz_hi), az, bfz));                                    \
                if (tn <= tf && tn <= tcull) { /* empty slots: no bit of the inner mask, no triangles */          \
                    const uint32_t meta = ((i < 4 ? w1.z : w1.w) >> (8 * (i & 3))) & 0xffu;                       \
                    hits |= 1u << (i);                                                                            \
                    trimask |= ((1u << (meta >> 5)) - 1u) << (meta & 31u); /* inner children: no triangles */     \
                }                                                                                                 \
            }
                CR_BVH8_CHILD(0)
                CR_BVH8_CHILD(1)
                CR_BVH8_CHILD(2)
                CR_BVH8_CHILD(3)
                CR_BVH8_CHILD(4)
                CR_BVH8_CHILD(5)
                CR_BVH8_CHILD(6)
                CR_BVH8_CHILD(7)
#undef CR_BVH8_CHILD
                hits = visiting_order(hits & imask, s0, s1, s2);
                // next node: the nearest hit inner child of this node, else the next of a pushed group
                uint32_t base = child_base, im = imask;
                if (!hits && sp > 0) {
                    --sp;
                    base = stack[sp].x;
                    hits = stack[sp].y & 0xffu;
                    im = stack[sp].y >> 8;
                }
                last = !hits; // nothing is left to visit
                if (hits) {
                    const uint32_t i = (uint32_t)__ffs(hits) - 1u;
                    hits &= hits - 1u;
                    node = base + __popc(im & ((1u << (i ^ (s0 | s1 | s2))) - 1u));
                    if (hits) {
                        stack[sp] = make_uint2(base, hits | (im << 8));
                        sp = sp < kStack8 - 1 ? sp + 1 : sp; // scene creation checks depth < kStack8
                    }
                } else if (!trimask) {
                    live = false;
                }
            }
        } while (kWait && __popc(__ballot_sync(0xffffffffu, live && !trimask)) > most);
        // the hit leaves' triangles
        if (trimask) {
            do {
                const uint32_t j = (uint32_t)__ffs(trimask) - 1u;
                trimask &= trimask - 1u;
                CR_DBG(if (!dbg_in_range(sc, tri_base + j, kDbgTri, sc->n_tris)) break;)
                test_leaf<kWide>(tris, r, r.ix, r.iy, r.iz, skip, tri_base + j, 1u, best, n_tri);
            } while (trimask);
            trimask = 0;
            tcull = __fmul_rn(best.t, kCullWiden);
            if (last || (kAny && best.leaf >= 0)) live = false;
        }
    }
}

#ifndef CR_BVH8_MIN_BLOCKS
#define CR_BVH8_MIN_BLOCKS 8 // resident 128-thread blocks per SM the register budget is sized for
#endif

template <bool kCount, bool kAny, bool kWide, RangeKind kKind>
__global__ void __launch_bounds__(128, CR_BVH8_MIN_BLOCKS) k_trace_bvh8(const SceneDev* __restrict__ scenes,
                             const uint16_t* slot_scene, const float4* ray_o, const float4* ray_d,
                             const int32_t* queue, const uint32_t* queue_count,
                             uint32_t n_max, int2* __restrict__ hit, unsigned long long* counters, uint32_t* work) {
    start_of_step();
    const uint32_t n = queue_count ? min(*queue_count, n_max) : n_max;
    unsigned long long n_node = 0, n_tri = 0;
    QueueSrc<kKind> src(n, work, slot_scene, ray_o, ray_d, queue, hit, blockIdx.x, gridDim.x);
    if (src.more()) trace_bvh8_warp<kCount, kAny, kWide>(scenes, src, n_node, n_tri);
    if (kCount) add_counts(counters, n_node, n_tri);
}

template <bool kCount, bool kAny, bool kWide, RangeKind kKind>
__global__ void __launch_bounds__(128, CR_BVH8_MIN_BLOCKS) k_trace_bvh8_user(const SceneDev* __restrict__ scene,
                                                                             UserRays rays, uint32_t n,
                                                                             unsigned long long* counters, uint32_t* work) {
    unsigned long long n_node = 0, n_tri = 0;
    UserSrc<kKind> src(n, work, rays);
    if (src.more()) trace_bvh8_warp<kCount, kAny, kWide>(scene, src, n_node, n_tri);
    if (kCount) add_counts(counters, n_node, n_tri);
}

// Shadow rays of next-event estimation over the BVH8-Q (see k_trace_shadow).
template <bool kWide, RangeKind kKind>
__global__ void __launch_bounds__(128, CR_BVH8_MIN_BLOCKS) k_trace_shadow8(
    const SceneDev* __restrict__ scenes, const uint16_t* slot_scene, const float4* sh_o, const float4* sh_d,
    const float4* sh_c, const int32_t* group_queue, const uint32_t* group_count, uint32_t n_groups_max, uint32_t K, float4* __restrict__ radiance,
    unsigned long long* __restrict__ n_traced, uint32_t* work) {
    start_of_step();
    const uint32_t n = (group_queue ? min(*group_count, n_groups_max) : n_groups_max) * K;
    ShadowSrc<kKind> src(n, work, slot_scene, sh_o, sh_d, sh_c, group_queue, radiance, K, blockIdx.x, gridDim.x);
    if (!src.more()) return;
    unsigned long long dn = 0, dt = 0;
    trace_bvh8_warp<false, true, kWide>(scenes, src, dn, dt);
    src.add_traced(n_traced);
}

// Closest hits (blocks below `first`) and light samples in one launch (see k_trace_both).
template <bool kWide, RangeKind kKind>
__global__ void __launch_bounds__(128, CR_BVH8_MIN_BLOCKS) k_trace_both8(
    const SceneDev* __restrict__ scenes, const uint16_t* slot_scene, const float4* ray_o, const float4* ray_d,
    const int32_t* queue, const uint32_t* queue_count, uint32_t n_max, int2* __restrict__ hit, uint32_t* work,
    const float4* sh_o, const float4* sh_d, const float4* sh_c, const int32_t* group_queue, const uint32_t* group_count,
    uint32_t n_groups_max, uint32_t K, float4* __restrict__ radiance, unsigned long long* __restrict__ n_traced,
    uint32_t* sh_work, uint32_t first) {
    start_of_step();
    unsigned long long dn = 0, dt = 0;
    if (blockIdx.x < first) {
        const uint32_t n = queue_count ? min(*queue_count, n_max) : n_max;
        QueueSrc<kKind> src(n, work, slot_scene, ray_o, ray_d, queue, hit, blockIdx.x, first);
        if (src.more()) trace_bvh8_warp<false, false, kWide>(scenes, src, dn, dt);
    } else {
        const uint32_t n = (group_queue ? min(*group_count, n_groups_max) : n_groups_max) * K;
        ShadowSrc<kKind> src(n, sh_work, slot_scene, sh_o, sh_d, sh_c, group_queue, radiance, K, blockIdx.x - first,
                             gridDim.x - first);
        if (!src.more()) return;
        trace_bvh8_warp<false, true, kWide>(scenes, src, dn, dt);
        src.add_traced(n_traced);
    }
}

} // namespace

// As for the BVH2: rays handed out lane by lane where the launch may hold more than lanes are
// resident at once.
template <bool kCount, bool kAny, bool kWide>
static void launch_bvh8(const TraceArgs& a, cudaStream_t st, LaunchCount& lc) {
    const uint32_t need = blocks_for(a.n_max, a.block);
    if (a.user.rays) {
        const uint32_t most = a.work ? resident_blocks<k_trace_bvh8_user<kCount, kAny, kWide, kMore>>(a.block, 0) : 0u;
        if (most && need > most)
            k_trace_bvh8_user<kCount, kAny, kWide, kMore><<<most, a.block, 0, st>>>(a.scenes, a.user, a.n_max, a.counters, a.work);
        else
            k_trace_bvh8_user<kCount, kAny, kWide, kPlain><<<need, a.block, 0, st>>>(a.scenes, a.user, a.n_max, a.counters, nullptr);
    } else {
        const uint32_t most = a.work ? resident_blocks<k_trace_bvh8<kCount, kAny, kWide, kMore>>(a.block, 0) : 0u;
        if (most && need > most)
            launch_step(a.chained, k_trace_bvh8<kCount, kAny, kWide, kMore>, most, a.block, 0, st, a.scenes, a.slot_scene, a.ray_o,
                        a.ray_d, a.queue, a.queue_count, a.n_max, a.hit, a.counters, a.work);
        else
            launch_step(a.chained, k_trace_bvh8<kCount, kAny, kWide, kPlain>, need, a.block, 0, st, a.scenes, a.slot_scene, a.ray_o,
                        a.ray_d, a.queue, a.queue_count, a.n_max, a.hit, a.counters, nullptr);
    }
    lc.n++;
}

template <bool kWide>
static void launch_bvh8_both(const TraceArgs& a, cudaStream_t st, LaunchCount& lc) {
    const ShadowArgs& s = *a.shadow;
    const uint32_t need = blocks_for(a.n_max, a.block), need_sh = blocks_for(s.n_groups_max * s.K, a.block);
    const uint32_t most = a.work && s.work ? resident_blocks<k_trace_both8<kWide, kMore>>(a.block, 0) : 0u;
    auto run = [&](auto kernel, uint32_t first, uint32_t rest, bool more) {
        launch_step(a.chained, kernel, first + rest, a.block, 0, st, a.scenes, a.slot_scene, a.ray_o, a.ray_d, a.queue,
                    a.queue_count, a.n_max, a.hit, more ? a.work : nullptr, s.sh_o, s.sh_d, s.sh_c, s.group_queue,
                    s.group_count, s.n_groups_max, s.K, s.radiance, s.n_traced, more ? s.work : nullptr, first);
    };
    if (most && (need > most || need_sh > most))
        run(k_trace_both8<kWide, kMore>, need < most ? need : most, need_sh < most ? need_sh : most, true);
    else run(k_trace_both8<kWide, kPlain>, need, need_sh, false);
    lc.n++;
}

template <bool kWide>
static void launch_bvh8(const TraceArgs& a, cudaStream_t st, LaunchCount& lc) {
    if (a.shadow && !a.any_hit && !a.counters && !a.user.rays) {
        launch_bvh8_both<kWide>(a, st, lc);
        return;
    }
    if (a.shadow) launch_shadow(*a.shadow, st, lc);
    if (a.any_hit) launch_bvh8<false, true, kWide>(a, st, lc);
    else if (a.counters) launch_bvh8<true, false, kWide>(a, st, lc);
    else launch_bvh8<false, false, kWide>(a, st, lc);
}

void launch_trace_bvh8(const TraceArgs& a, cudaStream_t st, LaunchCount& lc) {
    if (a.wide) launch_bvh8<true>(a, st, lc);
    else launch_bvh8<false>(a, st, lc);
}

template <bool kWide>
static void launch_shadow8(const ShadowArgs& a, cudaStream_t st, LaunchCount& lc) {
    const int block = 128;
    const uint32_t need = blocks_for(a.n_groups_max * a.K, block);
    const uint32_t most = a.work ? resident_blocks<k_trace_shadow8<kWide, kMore>>(block, 0) : 0u;
    auto run = [&](auto kernel, uint32_t grid, uint32_t* work) {
        launch_step(a.chained, kernel, grid, block, 0, st, a.scenes, a.slot_scene, a.sh_o, a.sh_d, a.sh_c, a.group_queue,
                    a.group_count, a.n_groups_max, a.K, a.radiance, a.n_traced, work);
    };
    if (most && need > most) run(k_trace_shadow8<kWide, kMore>, most, a.work);
    else run(k_trace_shadow8<kWide, kPlain>, need, nullptr);
    lc.n++;
}

void launch_shadow_bvh8(const ShadowArgs& a, cudaStream_t st, LaunchCount& lc) {
    if (a.wide) launch_shadow8<true>(a, st, lc);
    else launch_shadow8<false>(a, st, lc);
}

} // namespace cr
