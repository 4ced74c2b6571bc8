// trace.cu -- closest-hit BVH2 traversal (the intersection step, which dominates path
// tracing time, Sec. 1), one ray per lane.
//
// Stackful traversal of the 32-byte two-child records (DevBVH2): one 256-bit load fetches both
// child boxes, the nearer hit child is visited first and the farther one pushed.  The stack
// lives in shared memory (kSmemStack entries per lane, a warp's entries of one level in one
// 128-byte line) and older entries move to local memory when it fills.  Leaves hold
// up to four triangles tested with the watertight test of Woop, Benthin and Wald (2013).
// The primitives and the closest-hit rule shared with the BVH8-Q kernels (trace_bvh8.cu)
// are in trace_common.cuh.
#include <cuda_runtime.h>

#include <type_traits>

#include "cr_internal.h"
#include "launch_next.cuh"
#include "trace_common.cuh"

namespace cr {
namespace {


__device__ __forceinline__ void sts(uint32_t a, uint32_t v) {
    asm volatile("st.shared.u32 [%0], %1;" ::"r"(a), "r"(v) : "memory");
}
__device__ __forceinline__ uint32_t lds(uint32_t a) {
    uint32_t v;
    asm volatile("ld.shared.u32 %0, [%1];" : "=r"(v) : "r"(a) : "memory");
    return v;
}

constexpr int kNoNode = (int)0x80000000; // no traversal left (leaf codes are all above kRefill)
constexpr int kRefill = (int)0x80000001; // the stack's older entries wait in local memory
constexpr int kSteps = 2;                // node visits between two votes of the warp
constexpr int kStealIdle = 16;           // idle lanes of a warp at which they take over parts of other lanes' rays
// Shared-memory bytes of one warp: the lanes' stacks, three or four more words each.
__host__ __device__ constexpr uint32_t warp_smem(int entries, bool wide) { return (uint32_t)(entries + (wide ? 4 : 3)) * 128u; }
// Whether a link leads into or out of a grid (DevBVH2).
__device__ __forceinline__ bool grid_link(int node) { return node < (int)~(kGridLink - 1u) && node > kRefill; }

// Traversal of a warp's rays, one ray per lane; all 32 lanes call it together.
//
// What bounds it: issue slots and the latency of the record loads, both multiplied by lanes
// that wait (at the start 8 of 32 lanes were busy on secondary rays).  Three rules keep lanes busy:
//  - The descent ends as soon as no more than half of the warp's unfinished lanes are still in it,
//    and the leaves reached are tested while the others wait (half is the best of 3/8 to 3/4, a
//    vote every second visit the best of 1 to 4).
//  - kMore: once kTraceIdle lanes have finished their rays they take the next ones of the queue
//    (6 to 10 are alike, 16 costs 2%, 24 15%; ranges of 32 positions beat 16 and 64 by 2%).  Neighbours of
//    the queue stay together, and the records are small enough for the wider spread of
//    addresses.  Camera rays are traced without: a warp's rays are one pixel block, which
//    ends together, and taking rays one by one mixes blocks (0.35 to 0.40 ms against 0.28).
//  - kSteal: once the queue is empty and 16 lanes of the warp have nothing to do (8 to 24 are alike),
//    each of them takes the oldest stack entry of a lane that has one, with a copy of its ray, and
//    hands its hit back at the end; a word per ray carries the smallest distance found so far, by
//    which all of its lanes cull.  The closest hit does not depend on the order of visits, so it
//    stays the same.  Short launches spread their rays over the whole device first (two to a
//    warp or more): their time is that of their longest ray, one dependent load after another.
//  - kWide: some subtrees may be on grids of their own (DevBVH2).  A lane that comes to a link into or out
//    of one crosses within the descent, the link out waits on its stack below the subtree's entries.
//    A 1M-triangle sphere on a ground plane 500 times its size: 1M rays at it 0.89 ms with exact boxes (the
//    64-byte nodes), 2.18 in one grid, 0.34 so; a 1280x720 frame of 3 bounces 0.98, 7.1, 0.74 ms.  (Crossing
//    in the leaves' turn costs 4% more; without giving away what lies outside 1,000 rays take 115 us, not 76.)
// Landscape frame (1920x1080, 1.93M secondary rays): secondary trace 1.059 ms at the start (64-byte
// records in four loads, none of the rules), 0.74 with 32-byte records and the first rule, 0.63 with the
// second; primary trace 0.357 -> 0.280 ms.  Interior (3.35M secondary, 1.68M shadow rays): 2.46 ->
// 1.84 -> 1.52 ms and 1.75 -> 1.39 -> 0.92, 0.89 ms with the third.  A 500x333 frame of 4 samples and 8
// bounces (17,600 rays per launch): secondary trace 2.03 ms without the third rule, 1.26 with it;
// the two traces of 4,096 and 1,987 rays of a 64x64 frame 26 and 33 us (with 6 us of events
// each), 21 and 24 with it.
//
// kAny: visibility only; a lane is done at the first triangle hit before its ray's tmax.
// kSmemS: stack entries per lane kept in shared memory (8, 16 or 32), a launch-shape knob of
// the autotuner.
// kOne: every ray is in scenes[0], whose pointers then take no registers per lane.
template <bool kCount, bool kAny, int kSmemS, bool kOne, bool kWide, bool kSteal, class Src>
__device__ __forceinline__ void trace_bvh2_warp(const SceneDev* __restrict__ scenes, Src& src, uint32_t* smem,
                                                unsigned long long& n_node, unsigned long long& n_tri) {
    constexpr uint32_t kLevel = 128u; // bytes between a lane's entries
    constexpr int kHalf = kSmemS / 2;
    const SceneDev* sc = scenes;
    const uint32_t* __restrict__ nodes = scenes->nodes2;
    const float4* __restrict__ tris = scenes->tris;
    RayPre r;
    GridRay g;
    Best best{0.0f, -1};
    float tcull = 0.0f; // changes only after a leaf
    int skip = -1, key = -1;
    // entry 0 holds kNoNode (or kRefill while older entries are in lstack), so a pop needs no
    // test for an empty stack
    const uint32_t lane = threadIdx.x & 31u;
    const uint32_t base = (uint32_t)__cvta_generic_to_shared(smem) + (threadIdx.x >> 5) * warp_smem(kSmemS, kWide) + lane * 4u;
    // kSteal: more words per lane
    const uint32_t lent = base + kSmemS * kLevel;      // lanes that trace part of this lane's ray
    const uint32_t bound = lent + kLevel;              // the smallest distance found for this lane's ray
    const uint32_t list = bound + kLevel - lane * 4u;  // scratch list of the warp
    const uint32_t inside = bound + 2u * kLevel;       // kWide: count << 29 | last, the grids that the lane has gone into
    const uint32_t lim = base + (uint32_t)(kSmemS - kSteps + 1) * kLevel; // below it there is room for kSteps pushes
    uint32_t top = base + kLevel;                                         // next free entry
    int lstack[kStackTotal];
    int lsp = 0;
    uint32_t bot = base; // the entry that holds kNoNode or kRefill
    uint32_t owner = lane; // kSteal: the lane whose ray this lane traces (part of)
    int node = kNoNode;
    auto step = [&]() {
        if (kCount) ++n_node;
        CR_DBG(if (!dbg_in_range(sc, (uint32_t)node, kDbgNode, sc->n_nodes)) {
            node = kNoNode;
            return;
        })
        const NodeTest q = node_test(g, nodes, node);
        // the nearer hit child is next; with both hit the farther one is pushed, with none an
        // entry is popped (predicated: branches here cost 10% of the trace)
        asm volatile("{\n\t"
                     ".reg .pred p0, p1, q, s, b, n;\n\t"
                     ".reg .b32 far;\n\t"
                     "setp.le.f32 p0, %2, %4;\n\t"
                     "setp.le.and.f32 p0, %2, %6, p0;\n\t"
                     "setp.le.f32 p1, %3, %5;\n\t"
                     "setp.le.and.f32 p1, %3, %6, p1;\n\t"
                     "setp.le.f32 q, %2, %3;\n\t"
                     "not.pred n, p1;\n\t"
                     "or.pred s, q, n;\n\t"
                     "and.pred s, s, p0;\n\t"
                     "and.pred b, p0, p1;\n\t"
                     "or.pred n, p0, p1;\n\t"
                     "not.pred n, n;\n\t"
                     "selp.b32 %1, %7, %8, s;\n\t"
                     "selp.b32 far, %8, %7, s;\n\t"
                     "@b st.shared.u32 [%0], far;\n\t"
                     "@b add.u32 %0, %0, %9;\n\t"
                     "@n sub.u32 %0, %0, %9;\n\t"
                     "@n ld.shared.u32 %1, [%0];\n\t}"
                     : "+r"(top), "+r"(node)
                     : "f"(q.t0), "f"(q.t1), "f"(q.f0), "f"(q.f1), "f"(tcull), "r"(q.c0), "r"(q.c1), "n"(kLevel)
                     : "memory");
    };
    // a step into or out of a grid
    auto cross = [&]() {
        const uint32_t code = (uint32_t)(~node) & ~kGridLink;
        const uint4* rec = reinterpret_cast<const uint4*>(nodes + kDevNode2Words * (size_t)code);
        const uint4 a = __ldg(rec), b = __ldg(rec + 1);
        const bool in = !(code & 1u);
        cross_grid(r, a, b, g);
        if (in && top == bot + kLevel && lsp == 0) { // nothing is left outside
            node = (int)b.w;
            return;
        }
        if (kSteal) {
            const uint32_t n_in = (lds(inside) >> 29) + (in ? 1u : 0xffffffffu);
            sts(inside, n_in ? n_in << 29 | (in ? code : b.w) : 0u);
        }
        if (in) { // the link out waits on the stack
            sts(top, (uint32_t)(node - 1)); // ~(kGridLink | r + 1)
            top += kLevel;
            node = (int)b.w;
        } else {
            top -= kLevel;
            node = (int)lds(top);
        }
    };
    // the idle lanes hand in their hits and get new rays
    auto fill = [&](uint32_t alive) {
        const uint32_t i = src.take(~alive);
        if (node == kNoNode) {
            if (Src::kMore && key >= 0) src.store(key, best.leaf, best.t, tris);
            key = -1;
            float4 ro, rd;
            if (i < src.n && src.load(i, key, ro, rd)) {
                if (!kOne) {
                    sc = scenes + src.scene(key);
                    nodes = sc->nodes2;
                    tris = sc->tris;
                }
                r = prep_ray(ro, rd);
                g = grid_ray(ro, rd, *sc);
                skip = __float_as_int(ro.w);
                best = Best{rd.w, -1};
                tcull = __fmul_rn(best.t, kCullWiden);
                bot = base;
                sts(bot, (uint32_t)kNoNode);
                top = base + kLevel;
                if (kSteal) {
                    sts(lent, 0u);
                    sts(bound, __float_as_uint(rd.w));
                    if (kWide) sts(inside, 0u);
                }
                node = 0;
            }
        }
    };
    if (!Src::kMore) fill(0u);
    int refill = Src::kMore ? 32 : 33; // idle lanes at which rays are taken; 33: none are left
    while (true) {
        if (kSteal && refill == 33) {
            // a lane that has finished its part of another lane's ray hands its hit over
            uint32_t done = __ballot_sync(0xffffffffu, node == kNoNode && owner != lane);
            while (done) {
                const int h = __ffs(done) - 1;
                done &= done - 1u;
                const uint32_t o = __shfl_sync(0xffffffffu, owner, h);
                const float t = __shfl_sync(0xffffffffu, best.t, h);
                const int leaf = __shfl_sync(0xffffffffu, best.leaf, h);
                if (lane == o) {
                    sts(lent, lds(lent) - 1u);
                    if (leaf >= 0 && (best.leaf < 0 || t < best.t ||
                                      (t == best.t && __float_as_int(__ldg(&tris[3 * leaf]).w) <
                                                          __float_as_int(__ldg(&tris[3 * best.leaf]).w))))
                        best = Best{t, leaf};
                }
                if (lane == (uint32_t)h) owner = lane;
            }
            if (node == kNoNode && key >= 0 && lds(lent) == 0u) {
                src.store(key, best.leaf, best.t, tris);
                key = -1;
            }
        }
        uint32_t alive = __ballot_sync(0xffffffffu, node != kNoNode);
        if (Src::kMore && 32 - __popc(alive) >= refill) {
            fill(alive);
            alive = __ballot_sync(0xffffffffu, node != kNoNode);
            if (Src::kProbe) {
                const uint32_t oct = (g.ix < 0.0f ? 1u : 0u) | (g.iy < 0.0f ? 2u : 0u) | (g.iz < 0.0f ? 4u : 0u);
                src.probe(node != kNoNode, oct);
            }
            refill = !src.more() ? 33 : alive == 0u ? 32 : src.idle;
            if (alive == 0u && refill == 32) continue; // the positions taken held no rays
        }
        if (alive == 0u) {
            if (key >= 0) src.store(key, best.leaf, best.t, tris);
            return;
        }
        if (kSteal && refill == 33 && 32 - __popc(alive) >= kStealIdle) {
            // lanes without a ray take the oldest stack entry of a lane that has one
            const bool free = node == kNoNode && key < 0;
            bool gives = node != kNoNode && node != kRefill && lsp == 0 && top > bot + kLevel;
            if (kWide && gives) {
                // the oldest entry is in the grid that the lane started in: it gives only from there or from
                // one step away, and drops a link out that has nothing below it
                const uint32_t in = lds(inside), oldest = lds(bot + kLevel);
                gives = in < 2u << 29;
                if (gives && in && grid_link((int)oldest) && (~oldest & 1u)) {
                    bot += kLevel;
                    sts(bot, (uint32_t)kNoNode);
                    sts(inside, 0u);
                    gives = top > bot + kLevel;
                }
            }
            const uint32_t takers = __ballot_sync(0xffffffffu, free), givers = __ballot_sync(0xffffffffu, gives);
            const int n_moves = min(__popc(takers), __popc(givers));
            if (n_moves) {
                const uint32_t below = (1u << lane) - 1u;
                const int rank = __popc((gives ? givers : takers) & below);
                if (gives && rank < n_moves) {
                    sts(list + 4u * rank, lane);
                    asm volatile("red.shared.min.s32 [%0], %1;" ::"r"(bound + (owner - lane) * 4u), "r"(__float_as_int(best.t)) : "memory");
                }
                __syncwarp();
                const bool takes = free && rank < n_moves;
                const uint32_t from = takes ? lds(list + 4u * rank) : lane;
                const uint32_t their_bot = __shfl_sync(0xffffffffu, bot, from);
                const uint32_t their_owner = __shfl_sync(0xffffffffu, owner, from);
                r.ox = __shfl_sync(0xffffffffu, r.ox, from);
                r.oy = __shfl_sync(0xffffffffu, r.oy, from);
                r.oz = __shfl_sync(0xffffffffu, r.oz, from);
                r.sx = __shfl_sync(0xffffffffu, r.sx, from);
                r.sy = __shfl_sync(0xffffffffu, r.sy, from);
                r.sz = __shfl_sync(0xffffffffu, r.sz, from);
                r.kz = __shfl_sync(0xffffffffu, r.kz, from);
                g.ix = __shfl_sync(0xffffffffu, g.ix, from);
                g.iy = __shfl_sync(0xffffffffu, g.iy, from);
                g.iz = __shfl_sync(0xffffffffu, g.iz, from);
                g.nx = __shfl_sync(0xffffffffu, g.nx, from);
                g.ny = __shfl_sync(0xffffffffu, g.ny, from);
                g.nz = __shfl_sync(0xffffffffu, g.nz, from);
                g.fx = __shfl_sync(0xffffffffu, g.fx, from);
                g.fy = __shfl_sync(0xffffffffu, g.fy, from);
                g.fz = __shfl_sync(0xffffffffu, g.fz, from);
                g.snx = __shfl_sync(0xffffffffu, g.snx, from);
                g.sny = __shfl_sync(0xffffffffu, g.sny, from);
                g.snz = __shfl_sync(0xffffffffu, g.snz, from);
                g.sfx = __shfl_sync(0xffffffffu, g.sfx, from);
                g.sfy = __shfl_sync(0xffffffffu, g.sfy, from);
                g.sfz = __shfl_sync(0xffffffffu, g.sfz, from);
                skip = __shfl_sync(0xffffffffu, skip, from);
                const float their_t = __shfl_sync(0xffffffffu, best.t, from);
                if (!kOne) {
                    const unsigned long long their_sc = __shfl_sync(0xffffffffu, (unsigned long long)sc, from);
                    if (takes) {
                        sc = (const SceneDev*)their_sc;
                        nodes = sc->nodes2;
                        tris = sc->tris;
                    }
                }
                if (takes) {
                    const uint32_t in = kWide ? lds(inside + (from - lane) * 4u) & 0x1fffffffu : 0u;
                    if (kWide && in) { // out of the giver's grid, into the entry's
                        const uint4* rec = reinterpret_cast<const uint4*>(nodes + kDevNode2Words * (size_t)(in + 1u));
                        cross_grid(r, __ldg(rec), __ldg(rec + 1), g);
                    }
                    node = (int)lds(their_bot + kLevel);
                    owner = their_owner;
                    asm volatile("red.shared.add.u32 [%0], 1;" ::"r"(lent + (owner - lane) * 4u) : "memory");
                    best = Best{their_t, -1};
                    bot = base;
                    sts(bot, (uint32_t)kNoNode);
                    if (kWide) sts(inside, 0u);
                    top = base + kLevel;
                    lsp = 0;
                }
                __syncwarp();
                if (gives && rank < n_moves) {
                    bot += kLevel;
                    sts(bot, (uint32_t)kNoNode);
                }
                alive = __ballot_sync(0xffffffffu, node != kNoNode);
            }
        }
        if (kSteal && refill == 33) { // what the other lanes of this ray have found
            const float b = __uint_as_float(lds(bound + (owner - lane) * 4u));
            tcull = __fmul_rn(fminf(best.t, b), kCullWiden);
            if (kAny && b < 0.0f) { // one of them was blocked
                node = kNoNode;
                lsp = 0;
            }
        }
        const int half = __popc(alive) >> 1;
        bool run;
        do {
            run = (node >= 0 || (kWide && grid_link(node))) && top < lim;
            if (kWide && run && node < 0) {
                cross();
                run = node >= 0;
            }
#pragma unroll
            for (int e = 0; e < kSteps; ++e) {
                if (run) {
                    step();
                    run = node >= 0;
                }
            }
            run = (run || (kWide && grid_link(node))) && top < lim;
        } while (__popc(__ballot_sync(0xffffffffu, run)) > half);
        const bool full = top >= lim && (node >= 0 || (kWide && grid_link(node))); // room for a push is needed
        if (kSteal && full && bot != base) { // the room of entries given away
            const uint32_t by = bot - base;
            for (uint32_t a = bot; a < top; a += kLevel) sts(a - by, lds(a));
            bot = base;
            top -= by;
        } else if (full) { // rare: the older half of the stack moves to local memory
            for (int k = 0; k < kHalf; ++k) lstack[lsp + k] = (int)lds(base + (1 + k) * kLevel);
            for (uint32_t a = base + (1 + kHalf) * kLevel; a < top; a += kLevel) sts(a - kHalf * kLevel, lds(a));
            sts(base, (uint32_t)kRefill);
            lsp += kHalf;
            top -= kHalf * kLevel;
        }
        if (node < 0 && node != kNoNode && !(kWide && grid_link(node))) {
            if (node == kRefill) { // the stack is empty: its next entries come back
                lsp -= kHalf;
                for (int k = 0; k < kHalf; ++k) sts(base + (1 + k) * kLevel, (uint32_t)lstack[lsp + k]);
                top = base + (1 + kHalf) * kLevel;
                if (lsp == 0) sts(base, (uint32_t)kNoNode);
            } else { // a leaf
                const uint32_t code = (uint32_t)(~node);
                CR_DBG(if (!dbg_in_range(sc, (code >> 2) + (code & 3u), kDbgTri, sc->n_tris)) {
                    node = kNoNode;
                    lsp = 0;
                    continue;
                })
                test_leaf<kWide>(tris, r, g.ix, g.iy, g.iz, skip, code >> 2, (code & 3u) + 1u, best, n_tri);
                tcull = __fmul_rn(best.t, kCullWiden);
                if (kSteal && refill == 33 && best.leaf >= 0)
                    asm volatile("red.shared.min.s32 [%0], %1;" ::"r"(bound + (owner - lane) * 4u),
                                 "r"(__float_as_int(kAny ? -1.0f : best.t))
                                 : "memory");
            }
            top -= kLevel;
            node = (int)lds(top);
            if (kAny && best.leaf >= 0) {
                node = kNoNode;
                lsp = 0;
            }
        }
    }
}

#ifndef CR_TRACE_MAXNREG
// 36 warps resident per SM; 48 and 64 are within 1%, 40 costs 4%.  Variants for one scene spill up to 32 bytes
// per lane (44 where k_trace_both takes new rays), those for several 8 to 172.
#define CR_TRACE_MAXNREG 56
#endif

template <bool kCount, bool kAny, int kSmemS, bool kOne, bool kWide, RangeKind kKind>
__global__ void __maxnreg__(CR_TRACE_MAXNREG) k_trace_bvh2(const SceneDev* __restrict__ scenes,
                                                           chained_ptr<kOne, uint16_t> slot_scene,
                                                           chained_ptr<kOne, float4> ray_o,
                                                           chained_ptr<kOne, float4> ray_d,
                                                           chained_ptr<kOne, int32_t> queue,
                                                           chained_ptr<kOne, uint32_t> queue_count, uint32_t n_max,
                                                           int2* __restrict__ hit, unsigned long long* counters,
                                                           uint32_t* work) {
    if (kOne) start_of_step();
    extern __shared__ uint32_t smem_stack[];
    const uint32_t n = queue_count ? min(*queue_count, n_max) : n_max;
    unsigned long long n_node = 0, n_tri = 0;
    QueueSrc<kKind> src(n, work, slot_scene, ray_o, ray_d, queue, hit, blockIdx.x, gridDim.x);
    if (src.more()) trace_bvh2_warp<kCount, kAny, kSmemS, kOne, kWide, !kCount && !kAny && kKind != kPlain>(scenes, src, smem_stack, n_node, n_tri);
    if (kCount) add_counts(counters, n_node, n_tri);
}

// A caller's rays and hit arrays, no scratch between: cr_trace_rays used to copy the rays into the
// render path's records, trace, and copy the hits out, in buffers allocated per call (1M surface
// rays 952 us against 503, 300k camera rays 456 against 146, 1,000 rays 69 against 51).
template <bool kCount, bool kAny, bool kWide, RangeKind kKind>
__global__ void __maxnreg__(CR_TRACE_MAXNREG) k_trace_bvh2_user(const SceneDev* __restrict__ scene, UserRays rays,
                                                                uint32_t n, unsigned long long* counters,
                                                                uint32_t* work) {
    extern __shared__ uint32_t smem_stack[];
    unsigned long long n_node = 0, n_tri = 0;
    UserSrc<kKind> src(n, work, rays);
    if (src.more()) trace_bvh2_warp<kCount, kAny, kSmemStack, true, kWide, !kCount && !kAny && kKind != kPlain>(scene, src, smem_stack, n_node, n_tri);
    if (kCount) add_counts(counters, n_node, n_tri);
}

// Two-phase variant: phase 1 traverses every ray for at most `budget` node and leaf visits;
// a ray that runs out saves its traversal state (next node, stack, best hit) and is flagged.
// The flagged rays are compacted in queue order (so neighbours stay neighbours) and phase 2
// resumes them in full warps, so short rays no longer leave most lanes of a warp idle while
// its long rays finish.  Suspension only happens with at most kSaveStack entries on the
// stack (deeper rays run to completion in phase 1).  The visit order is the single-ray
// kernel's, so the hits are identical.
constexpr int kSaveStack = 24;

__device__ __forceinline__ int2 trace_bvh2_resumable(const SceneDev& sc, float4 ro, float4 rd, uint32_t* sstack,
                                                     uint32_t budget, TraceState* st, bool resume, bool& suspended) {
    constexpr int kSmemS = kSmemStack;
    const uint32_t* __restrict__ nodes = sc.nodes2;
    const float4* __restrict__ tris = sc.tris;
    const RayPre r = prep_ray(ro, rd);
    const GridRay g = grid_ray(ro, rd, sc);
    const int skip = __float_as_int(ro.w);
    Best best{rd.w, -1};
    int lstack[kStackTotal - kSmemStack];
    const int stride = blockDim.x;
    int sp = 0, node = 0;
    if (resume) {
        node = st->node;
        sp = st->sp;
        best = Best{st->t, st->leaf};
        for (int k = 0; k < sp; ++k) {
            const int v = st->stack[k];
            if (k < kSmemStack) sstack[k * stride] = (uint32_t)v;
            else lstack[k - kSmemStack] = v;
        }
    }
    uint32_t visits = 0;
    suspended = false;
    while (true) {
        while (node >= 0) {
            if (++visits > budget && sp <= kSaveStack) {
                suspended = true;
                break;
            }
            const float tcull = __fmul_rn(best.t, kCullWiden);
            const NodeTest q = node_test(g, nodes, node);
            const float t0 = q.t0, t1 = q.t1;
            const int c0 = q.c0, c1 = q.c1;
            const bool h0 = q.hit0(tcull), h1 = q.hit1(tcull);
            if (h0 && h1) {
                const bool first0 = t0 <= t1;
                const int near = first0 ? c0 : c1, far = first0 ? c1 : c0;
                STACK_PUSH(far);
                node = near;
            } else if (h0 || h1) {
                node = h0 ? c0 : c1;
            } else {
                if (sp == 0) { node = 0x7fffffff; break; }
                STACK_POP(node);
            }
        }
        if (suspended || node == 0x7fffffff) break;
        const uint32_t code = (uint32_t)(~node);
        unsigned long long dummy = 0;
        test_leaf<false>(tris, r, g.ix, g.iy, g.iz, skip, code >> 2, (code & 3u) + 1u, best, dummy);
        ++visits;
        if (sp == 0) break;
        STACK_POP(node);
    }
    if (suspended) {
        st->node = node;
        st->sp = sp;
        st->t = best.t;
        st->leaf = best.leaf;
        for (int k = 0; k < sp; ++k) st->stack[k] = k < kSmemStack ? (int)sstack[k * stride] : lstack[k - kSmemStack];
    }
    return make_int2(best.leaf, __float_as_int(best.t));
}

__global__ void __maxnreg__(CR_TRACE_MAXNREG) k_trace_bvh2_phase(
    const SceneDev* __restrict__ scenes, const uint16_t* __restrict__ slot_scene, const float4* __restrict__ ray_o,
    const float4* __restrict__ ray_d, const int32_t* __restrict__ queue, const uint32_t* __restrict__ queue_count,
    uint32_t n_max, int2* __restrict__ hit, TraceState* __restrict__ state, uint8_t* __restrict__ susp,
    uint32_t budget, int resume) {
    extern __shared__ uint32_t smem_stack[];
    const uint32_t n = queue_count ? min(*queue_count, n_max) : n_max;
    const uint32_t i = blockIdx.x * blockDim.x + threadIdx.x;
    if (i >= n) return;
    const int slot = queue ? queue[i] : (int)i;
    const float4 ro = ray_o[slot];
    const float4 rd = ray_d[slot];
    bool suspended = false;
    int2 h = make_int2(-1, __float_as_int(INFINITY));
    if (rd.w >= 0.0f) {
        const SceneDev& sc = scenes[slot_scene ? slot_scene[slot] : 0];
        h = trace_bvh2_resumable(sc, ro, rd, smem_stack + threadIdx.x, budget, &state[slot],
                                 resume != 0, suspended);
    }
    if (!suspended) hit[slot] = h;
    if (susp) susp[i] = suspended ? 1 : 0;
}

// Order-preserving compaction of the suspended rays' queue entries (count, scan, scatter).
__global__ void __launch_bounds__(256) k_susp_count(const uint8_t* __restrict__ susp, const uint32_t* __restrict__ count,
                                                    uint32_t n_max, uint32_t* __restrict__ block_counts) {
    __shared__ uint32_t s_w[8];
    const uint32_t n = min(*count, n_max);
    const uint32_t i = blockIdx.x * 256 + threadIdx.x;
    const uint32_t f = (i < n && susp[i]) ? 1u : 0u;
    const uint32_t b = __ballot_sync(0xffffffffu, f);
    if ((threadIdx.x & 31) == 0) s_w[threadIdx.x >> 5] = __popc(b);
    __syncthreads();
    if (threadIdx.x == 0) {
        uint32_t t = 0;
        for (int w = 0; w < 8; ++w) t += s_w[w];
        block_counts[2 * blockIdx.x] = t;
        block_counts[2 * blockIdx.x + 1] = 0;
    }
}

__global__ void __launch_bounds__(256) k_susp_scatter(const uint8_t* __restrict__ susp, const int32_t* __restrict__ queue,
                                                      const uint32_t* __restrict__ count, uint32_t n_max,
                                                      const uint32_t* __restrict__ block_offsets,
                                                      int32_t* __restrict__ out_queue) {
    __shared__ uint32_t s_w[8];
    const uint32_t n = min(*count, n_max);
    const uint32_t i = blockIdx.x * 256 + threadIdx.x;
    const uint32_t f = (i < n && susp[i]) ? 1u : 0u;
    const uint32_t lane = threadIdx.x & 31, w = threadIdx.x >> 5;
    const uint32_t b = __ballot_sync(0xffffffffu, f);
    if (lane == 0) s_w[w] = __popc(b);
    __syncthreads();
    uint32_t before = 0;
    for (uint32_t k = 0; k < w; ++k) before += s_w[k];
    if (f) out_queue[block_offsets[2 * blockIdx.x] + before + __popc(b & ((1u << lane) - 1u))] = queue[i];
}

// Warp-packet variant: the 32 lanes of a warp traverse ONE node sequence.  At each inner
// node every lane tests both child boxes against its own ray (with its own culling
// distance); a child is entered if any lane's ray reaches it, nearer-first by majority.
// Leaves are tested by every lane against its own ray.  Each lane therefore visits a
// superset of the boxes its own ray enters, with the same triangle test and tie rule, so
// the hits are the single-ray kernel's bit for bit.  Control flow is warp-uniform, which
// pays off when the rays of a warp are coherent (primary rays, reused directions) and
// costs extra box and triangle tests when they are not.  Every ray is in scenes[0].
__global__ void __maxnreg__(CR_TRACE_MAXNREG) k_trace_bvh2_packet(
    const SceneDev* __restrict__ scenes, const float4* __restrict__ ray_o,
    const float4* __restrict__ ray_d, const int32_t* __restrict__ queue, const uint32_t* __restrict__ queue_count,
    uint32_t n_max, int2* __restrict__ hit) {
    extern __shared__ uint32_t smem_stack[];
    uint32_t* sstack = smem_stack + threadIdx.x;
    const int stride = blockDim.x;
    const uint32_t n = queue_count ? min(*queue_count, n_max) : n_max;
    const uint32_t i = blockIdx.x * blockDim.x + threadIdx.x;
    if (__all_sync(0xffffffffu, i >= n)) return;
    int slot = -1;
    bool valid = false;
    RayPre r;
    int skip = -1;
    Best best{-1.0f, -1}; // t < 0: a lane without a ray never enters a box
    if (i < n) {
        slot = queue ? queue[i] : (int)i;
        const float4 ro = ray_o[slot];
        const float4 rd = ray_d[slot];
        if (rd.w >= 0.0f) {
            r = prep_ray(ro, rd);
            skip = __float_as_int(ro.w);
            best = Best{rd.w, -1};
            valid = true;
        } else {
            hit[slot] = make_int2(-1, __float_as_int(INFINITY));
        }
    }
    const SceneDev& sc = scenes[0];
    const uint32_t* nodes = sc.nodes2;
    const float4* tris = sc.tris;
    unsigned long long dummy = 0;
    constexpr int kSmemS = kSmemStack;
#if CR_TRACE_LOCAL_STACK
    int lstack_all[kStackTotal];
#else
    int lstack[kStackTotal - kSmemStack];
#endif
    int sp = 0;
    int node = 0;
    if (!valid) r = prep_ray(make_float4(0, 0, 0, 0), make_float4(0, 0, 1, -1)); // inert ray
    const GridRay g = grid_ray(make_float4(r.ox, r.oy, r.oz, 0), make_float4(r.dx, r.dy, r.dz, 0), sc);
    while (true) {
        if (node >= 0) {
            const float tcull = __fmul_rn(best.t, kCullWiden);
            const NodeTest q = node_test(g, nodes, node);
            const float t0 = q.t0, t1 = q.t1;
            const int c0 = q.c0, c1 = q.c1;
            const bool h0 = q.hit0(tcull), h1 = q.hit1(tcull);
            const uint32_t v0 = __ballot_sync(0xffffffffu, h0 && (!h1 || t0 <= t1));
            const uint32_t v1 = __ballot_sync(0xffffffffu, h1 && (!h0 || t1 < t0));
            const bool any0 = __any_sync(0xffffffffu, h0), any1 = __any_sync(0xffffffffu, h1);
            if (any0 && any1) {
                const bool first0 = __popc(v0) >= __popc(v1);
                STACK_PUSH(first0 ? c1 : c0);
                node = first0 ? c0 : c1;
                continue;
            } else if (any0 || any1) {
                node = any0 ? c0 : c1;
                continue;
            }
        } else {
            const uint32_t code = (uint32_t)(~node);
            if (valid) test_leaf<false>(tris, r, g.ix, g.iy, g.iz, skip, code >> 2, (code & 3u) + 1u, best, dummy);
        }
        if (sp == 0) break;
        STACK_POP(node);
    }
    if (valid) hit[slot] = make_int2(best.leaf, __float_as_int(best.t));
}

// Speculative variant: lanes keep one reached leaf pending and go on descending inner
// nodes until every lane of the warp holds a leaf or has finished; then all lanes test
// their pending leaves together.  Inner-node and leaf phases thus run with more active
// lanes.  The loops are warp-synchronous: every lane (finished or not) executes each
// iteration, and every iteration either visits a node, parks a leaf or tests one.
constexpr int kEmpty = 0x7fffffff; // stack exhausted

__global__ void __maxnreg__(CR_TRACE_MAXNREG) k_trace_bvh2_spec(
    const SceneDev* __restrict__ scenes, const uint16_t* __restrict__ slot_scene, const float4* __restrict__ ray_o,
    const float4* __restrict__ ray_d, const int32_t* __restrict__ queue, const uint32_t* __restrict__ queue_count,
    uint32_t n_max, int2* __restrict__ hit) {
    extern __shared__ uint32_t smem_stack[];
    uint32_t* sstack = smem_stack + threadIdx.x;
    const int stride = blockDim.x;
    const uint32_t n = queue_count ? min(*queue_count, n_max) : n_max;
    const uint32_t i = blockIdx.x * blockDim.x + threadIdx.x;
    // whole warps past the end leave together; the others run every iteration
    if (__all_sync(0xffffffffu, i >= n)) return;
    int slot = -1;
    bool done = true;
    RayPre r;
    GridRay g;
    int skip = -1;
    Best best{0.0f, -1};
    const uint32_t* nodes = nullptr;
    const float4* tris = nullptr;
    if (i < n) {
        slot = queue ? queue[i] : (int)i;
        const float4 ro = ray_o[slot];
        const float4 rd = ray_d[slot];
        if (rd.w >= 0.0f) {
            const SceneDev& sc = scenes[slot_scene ? slot_scene[slot] : 0];
            nodes = sc.nodes2;
            tris = sc.tris;
            r = prep_ray(ro, rd);
            g = grid_ray(ro, rd, sc);
            skip = __float_as_int(ro.w);
            best = Best{rd.w, -1};
            done = false;
        } else {
            hit[slot] = make_int2(-1, __float_as_int(INFINITY));
        }
    }
    int lstack[kStackTotal - kSmemStack];
    int sp = 0, node = done ? kEmpty : 0, leaf = 0;
    unsigned long long dummy = 0;
    auto pop = [&]() -> int {
        if (sp == 0) return kEmpty;
        --sp;
        return sp < kSmemStack ? (int)sstack[sp * stride] : lstack[sp - kSmemStack];
    };
    while (true) {
        // inner phase
        while (true) {
            if (node >= 0 && node != kEmpty) {
                const float tcull = __fmul_rn(best.t, kCullWiden);
                const NodeTest q = node_test(g, nodes, node);
                const float t0 = q.t0, t1 = q.t1;
                const int c0 = q.c0, c1 = q.c1;
                const bool h0 = q.hit0(tcull), h1 = q.hit1(tcull);
                if (h0 && h1) {
                    const bool first0 = t0 <= t1;
                    const int far = first0 ? c1 : c0;
                    node = first0 ? c0 : c1;
                    if (sp < kSmemStack) sstack[sp * stride] = (uint32_t)far;
                    else if (sp < kStackTotal) lstack[sp - kSmemStack] = far;
                    sp = sp < kStackTotal ? sp + 1 : sp; // the builder keeps depth < kStackTotal
                } else if (h0 || h1) {
                    node = h0 ? c0 : c1;
                } else {
                    node = pop();
                }
            }
            if (node < 0 && leaf == 0) { // park the reached leaf and keep descending
                leaf = node;
                node = pop();
            }
            const bool searching = leaf == 0 && node != kEmpty;
            if (!__any_sync(0xffffffffu, searching)) break;
        }
        // leaf phase: the parked leaf, then any leaf the descent stopped on
        while (leaf < 0) {
            const uint32_t code = (uint32_t)(~leaf);
            test_leaf<false>(tris, r, g.ix, g.iy, g.iz, skip, code >> 2, (code & 3u) + 1u, best, dummy);
            leaf = 0;
            if (node < 0) {
                leaf = node;
                node = pop();
            }
        }
        if (!done && node == kEmpty) {
            hit[slot] = make_int2(best.leaf, __float_as_int(best.t));
            done = true;
        }
        if (__all_sync(0xffffffffu, done)) break;
    }
}

template <bool kOne, bool kWide, RangeKind kKind>
__global__ void __maxnreg__(CR_TRACE_MAXNREG) k_trace_shadow(
    const SceneDev* __restrict__ scenes, chained_ptr<kOne, uint16_t> slot_scene, chained_ptr<kOne, float4> sh_o,
    chained_ptr<kOne, float4> sh_d, chained_ptr<kOne, float4> sh_c, chained_ptr<kOne, int32_t> group_queue,
    chained_ptr<kOne, uint32_t> group_count, uint32_t n_groups_max, uint32_t K, float4* __restrict__ radiance,
    unsigned long long* __restrict__ n_traced, uint32_t* work) {
    if (kOne) start_of_step();
    extern __shared__ uint32_t smem_stack[];
    const uint32_t n = (group_queue ? min(*group_count, n_groups_max) : n_groups_max) * K;
    ShadowSrc<kKind> src(n, work, slot_scene, sh_o, sh_d, sh_c, group_queue, radiance, K, blockIdx.x, gridDim.x);
    if (!src.more()) return;
    unsigned long long dn = 0, dt = 0;
    trace_bvh2_warp<false, true, kSmemStack, kOne, kWide, kKind != kPlain>(scenes, src, smem_stack, dn, dt);
    src.add_traced(n_traced);
}

// The next closest-hit rays of a bounce and its light samples in one launch: neither trace needs the
// other's results, and each alone spends about 80 us filling the device and draining it to its longest
// rays.  Blocks below `first` trace the closest hits, which take longer; the others come in as these end
// (the other way round: 24 requests 5780 us against 5550, a batch of 16 jobs 5358 against 5314, single
// renders alike).  Against a launch for each: an interior of 96 x 64 pixels 480 -> 350 us, 1280 x 720
// 2965 -> 2805, with 16 samples 36.9 -> 36.5 ms, 24 requests 6390 -> 5550 us.
template <int kSmemS, bool kOne, bool kWide, RangeKind kKind>
__global__ void __maxnreg__(CR_TRACE_MAXNREG) k_trace_both(
    const SceneDev* __restrict__ scenes, chained_ptr<kOne, uint16_t> slot_scene, chained_ptr<kOne, float4> ray_o,
    chained_ptr<kOne, float4> ray_d, chained_ptr<kOne, int32_t> queue, chained_ptr<kOne, uint32_t> queue_count,
    uint32_t n_max, int2* __restrict__ hit, uint32_t* work, chained_ptr<kOne, float4> sh_o,
    chained_ptr<kOne, float4> sh_d, chained_ptr<kOne, float4> sh_c, chained_ptr<kOne, int32_t> group_queue,
    chained_ptr<kOne, uint32_t> group_count, uint32_t n_groups_max, uint32_t K, float4* __restrict__ radiance,
    unsigned long long* __restrict__ n_traced, uint32_t* sh_work, uint32_t first) {
    if (kOne) start_of_step();
    extern __shared__ uint32_t smem_stack[];
    unsigned long long dn = 0, dt = 0;
    if (blockIdx.x < first) {
        const uint32_t n = queue_count ? min(*queue_count, n_max) : n_max;
        QueueSrc<kKind> src(n, work, slot_scene, ray_o, ray_d, queue, hit, blockIdx.x, first);
        if (src.more()) trace_bvh2_warp<false, false, kSmemS, kOne, kWide, kKind != kPlain>(scenes, src, smem_stack, dn, dt);
    } else {
        const uint32_t n = (group_queue ? min(*group_count, n_groups_max) : n_groups_max) * K;
        ShadowSrc<kKind> src(n, sh_work, slot_scene, sh_o, sh_d, sh_c, group_queue, radiance, K, blockIdx.x - first,
                             gridDim.x - first);
        if (!src.more()) return;
        trace_bvh2_warp<false, true, kSmemS, kOne, kWide, kKind != kPlain>(scenes, src, smem_stack, dn, dt);
        src.add_traced(n_traced);
    }
}

__global__ void k_hits_to_user(const float4* __restrict__ tris, const int2* __restrict__ hit, uint32_t n,
                               int32_t* __restrict__ prim, float* __restrict__ t) {
    const uint32_t i = blockIdx.x * blockDim.x + threadIdx.x;
    if (i >= n) return;
    const int2 h = hit[i];
    prim[i] = h.x >= 0 ? __float_as_int(__ldg(&tris[3 * h.x]).w) : -1;
    t[i] = h.x >= 0 ? __int_as_float(h.y) : INFINITY; // a miss of a bounded ray reports inf, not tmax
}

__global__ void k_rays_from_user(const float* __restrict__ rays, const int32_t* __restrict__ skip, uint32_t n,
                                 float4* __restrict__ ray_o, float4* __restrict__ ray_d) {
    const uint32_t i = blockIdx.x * blockDim.x + threadIdx.x;
    if (i >= n) return;
    const float* r = rays + 8 * (size_t)i;
    ray_o[i] = make_float4(r[0], r[1], r[2], __int_as_float(skip ? skip[i] : -1));
    ray_d[i] = make_float4(r[4], r[5], r[6], r[7]);
}

} // namespace

void launch_shadow(const ShadowArgs& a, cudaStream_t st, LaunchCount& lc) {
    const uint32_t n_pos = a.n_groups_max * a.K;
    if (n_pos == 0) return;
    if (a.bvh8) {
        launch_shadow_bvh8(a, st, lc);
        return;
    }
    const int block = kSecondaryBlock;
    const uint32_t need = blocks_for(n_pos, block); // the kinds of range as below
    auto go = [&](auto one, auto wide) {
        constexpr bool kOne = decltype(one)::value, kWide = decltype(wide)::value;
        const size_t smem = (size_t)warp_smem(kSmemStack, kWide) * (block / 32);
        const uint32_t most = resident_blocks<k_trace_shadow<kOne, kWide, kMore>>(block, smem);
        auto run = [&](auto kernel, uint32_t grid) {
            launch_step(kOne && a.chained, kernel, grid, block, smem, st, a.scenes, a.slot_scene, a.sh_o, a.sh_d, a.sh_c,
                        a.group_queue, a.group_count, a.n_groups_max, a.K, a.radiance, a.n_traced, a.work);
        };
        if (need <= most && a.alone) run(k_trace_shadow<kOne, kWide, kFew>, spread_blocks(n_pos, block, most));
        else if (a.work && most && need > most) run(k_trace_shadow<kOne, kWide, kMore>, most);
        else run(k_trace_shadow<kOne, kWide, kPlain>, need);
    };
    if (a.wide) go(std::false_type(), std::true_type());
    else if (a.one_scene) go(std::true_type(), std::false_type());
    else go(std::false_type(), std::false_type());
    lc.n++;
}

bool user_rays_apart(const float* rays, const int32_t* skip, uint32_t n, const int32_t* prim, const float* t) {
    const auto apart = [](const void* a, size_t na, const void* b, size_t nb) {
        const uintptr_t x = (uintptr_t)a, y = (uintptr_t)b;
        return x + na <= y || y + nb <= x;
    };
    const size_t w = 4 * (size_t)n;
    return apart(rays, 8 * w, prim, w) && apart(rays, 8 * w, t, w) && apart(prim, w, t, w) &&
           (!skip || (apart(skip, w, prim, w) && apart(skip, w, t, w)));
}

void launch_rays_from_user(const float* rays, const int32_t* skip, uint32_t n, float4* ray_o, float4* ray_d,
                           cudaStream_t st, LaunchCount& lc) {
    if (n == 0) return;
    k_rays_from_user<<<(n + 255) / 256, 256, 0, st>>>(rays, skip, n, ray_o, ray_d);
    lc.n++;
}

SceneDev scene_entry(const DevScene& s, bool bvh8) {
    SceneDev e;
    e.nodes2 = s.nodes2;
    for (int k = 0; k < 3; ++k) {
        e.grid_lo[k] = s.grid_lo[k];
        e.grid_scale[k] = s.grid_scale[k];
    }
    e.nodes8 = s.nodes8;
    e.nodes4 = s.nodes4;
    e.tris = bvh8 ? s.tris8 : s.tris;
    e.mats = s.mats;
    for (int k = 0; k < 3; ++k) {
        e.env[k] = s.env[k];
        e.lo[k] = s.lo[k];
        e.hi[k] = s.hi[k];
    }
    e.env[3] = e.lo[3] = e.hi[3] = 0.0f;
    e.light_cdf = s.light_cdf;
    e.lights = s.lights;
    e.n_lights = s.n_lights;
    e.light_total = s.light_total;
    e.n_nodes = bvh8 ? s.n_nodes8 : s.n_nodes2;
    e.n_tris = s.n_tri;
    e.n_mats = s.n_mat;
    e.err = s.err;
    return e;
}

template <bool kOne, bool kWide, auto kKernel, int kSmemS>
static void launch_bvh2_kernel(const TraceArgs& a, uint32_t grid, cudaStream_t st, LaunchCount& lc) {
    const size_t smem = (size_t)warp_smem(kSmemS, kWide) * (a.block / 32);
    allow_smem<kKernel>(smem); // blocks of 352 threads or more with 32 entries
    launch_step(kOne && a.chained, kKernel, grid, a.block, smem, st, a.scenes, a.slot_scene, a.ray_o, a.ray_d, a.queue,
                a.queue_count, a.n_max, a.hit, a.counters, a.work);
    lc.n++;
}

// The kind of range.  A launch that may hold more rays than lanes are resident at once hands them
// out lane by lane where a.work allows it (kMore), else one per lane of as many blocks as it takes
// (kPlain).  With fewer rays they are spread over all resident warps (kFew), unless other launches
// share the device (a server's lanes): 24 requests took 6.65 ms against 6.54.
template <bool kOne, bool kWide, bool kCount, bool kAny, int kSmemS>
static void launch_bvh2_scenes(const TraceArgs& a, cudaStream_t st, LaunchCount& lc) {
    constexpr auto kM = k_trace_bvh2<kCount, kAny, kSmemS, kOne, kWide, kMore>;
    constexpr auto kF = k_trace_bvh2<kCount, kAny, kSmemS, kOne, kWide, kFew>;
    constexpr auto kP = k_trace_bvh2<kCount, kAny, kSmemS, kOne, kWide, kPlain>;
    const uint32_t need = blocks_for(a.n_max, a.block);
    const uint32_t most = resident_blocks<kM>(a.block, (size_t)warp_smem(kSmemS, kWide) * (a.block / 32));
    if (need <= most && a.alone) launch_bvh2_kernel<kOne, kWide, kF, kSmemS>(a, spread_blocks(a.n_max, a.block, most), st, lc);
    else if (a.work && most && need > most) launch_bvh2_kernel<kOne, kWide, kM, kSmemS>(a, most, st, lc);
    else launch_bvh2_kernel<kOne, kWide, kP, kSmemS>(a, need, st, lc);
}

template <auto kKernel>
using kernel_of = std::integral_constant<decltype(kKernel), kKernel>;

// One launch for a.shadow's rays too (k_trace_both): the kind of range that the longer list asks for.
template <bool kOne, bool kWide, int kSmemS>
static void launch_bvh2_both(const TraceArgs& a, cudaStream_t st, LaunchCount& lc) {
    const ShadowArgs& s = *a.shadow;
    const size_t smem = (size_t)warp_smem(kSmemS, kWide) * (a.block / 32);
    const uint32_t n_sh = s.n_groups_max * s.K;
    const uint32_t need = blocks_for(a.n_max, a.block), need_sh = blocks_for(n_sh, a.block);
    const uint32_t most = resident_blocks<k_trace_both<kSmemS, kOne, kWide, kMore>>(a.block, smem);
    auto run = [&](auto kernel, uint32_t first, uint32_t rest) {
        constexpr auto kKernel = decltype(kernel)::value;
        allow_smem<kKernel>(smem);
        launch_step(kOne && a.chained, kKernel, first + rest, a.block, smem, st, a.scenes, a.slot_scene, a.ray_o, a.ray_d,
                    a.queue, a.queue_count, a.n_max, a.hit, a.work, s.sh_o, s.sh_d, s.sh_c, s.group_queue, s.group_count,
                    s.n_groups_max, s.K, s.radiance, s.n_traced, s.work, first);
    };
    if (need <= most && need_sh <= most && a.alone)
        run(kernel_of<k_trace_both<kSmemS, kOne, kWide, kFew>>(), spread_blocks(a.n_max, a.block, most), spread_blocks(n_sh, a.block, most));
    else if (a.work && s.work && most && (need > most || need_sh > most))
        run(kernel_of<k_trace_both<kSmemS, kOne, kWide, kMore>>(), need < most ? need : most, need_sh < most ? need_sh : most);
    else run(kernel_of<k_trace_both<kSmemS, kOne, kWide, kPlain>>(), need, need_sh);
    lc.n++;
}

// kOneScene: whether launches over a single scene have a variant of their own.  Only these are set up
// while the launch before ends: the plain pointers that this takes make launches over several scenes
// 1% slower (16-job batch 5424 -> 5472 us) and those over one scene 1% faster (1024 x 1024 1185 -> 1175).
// Launches with a wide scene have kernels of their own (what these do more costs the others 2 to 3%).
template <bool kOneScene, bool kCount, bool kAny, int kSmemS>
static void launch_bvh2(const TraceArgs& a, cudaStream_t st, LaunchCount& lc) {
    const bool one = kOneScene && a.one_scene && !a.wide;
    if constexpr (!kCount && !kAny) {
        if (a.shadow) {
            if (a.wide) launch_bvh2_both<false, true, kSmemS>(a, st, lc);
            else if (one) launch_bvh2_both<kOneScene, false, kSmemS>(a, st, lc);
            else launch_bvh2_both<false, false, kSmemS>(a, st, lc);
            return;
        }
    }
    if (a.shadow) launch_shadow(*a.shadow, st, lc);
    if (a.wide) launch_bvh2_scenes<false, true, kCount, kAny, kSmemS>(a, st, lc);
    else if (one) launch_bvh2_scenes<kOneScene, false, kCount, kAny, kSmemS>(a, st, lc);
    else launch_bvh2_scenes<false, false, kCount, kAny, kSmemS>(a, st, lc);
}

template <bool kCount, bool kAny, bool kWide>
static void launch_bvh2_user(const TraceArgs& a, cudaStream_t st, LaunchCount& lc) {
    const size_t smem = (size_t)warp_smem(kSmemStack, kWide) * (a.block / 32);
    const uint32_t need = blocks_for(a.n_max, a.block);
    const uint32_t most = resident_blocks<k_trace_bvh2_user<kCount, kAny, kWide, kMore>>(a.block, smem);
    auto run = [&](auto kernel, uint32_t grid) {
        kernel<<<grid, a.block, smem, st>>>(a.scenes, a.user, a.n_max, a.counters, a.work);
    };
    if (need <= most) run(k_trace_bvh2_user<kCount, kAny, kWide, kFew>, spread_blocks(a.n_max, a.block, most));
    else if (a.work && most) run(k_trace_bvh2_user<kCount, kAny, kWide, kMore>, most);
    else run(k_trace_bvh2_user<kCount, kAny, kWide, kPlain>, need);
    lc.n++;
}

template <bool kWide>
static void launch_bvh2_user(const TraceArgs& a, cudaStream_t st, LaunchCount& lc) {
    if (a.any_hit) launch_bvh2_user<false, true, kWide>(a, st, lc);
    else if (a.counters) launch_bvh2_user<true, false, kWide>(a, st, lc);
    else launch_bvh2_user<false, false, kWide>(a, st, lc);
}

void launch_trace(const TraceArgs& a, cudaStream_t st, LaunchCount& lc) {
    if (a.n_max == 0) {
        if (a.shadow) launch_shadow(*a.shadow, st, lc);
        return;
    }
    if (a.user.rays && !a.bvh8 && !(a.bvh4 && !a.any_hit)) { // a caller's rays through the BVH2
        if (a.wide) launch_bvh2_user<true>(a, st, lc);
        else launch_bvh2_user<false>(a, st, lc);
        return;
    }
    const int block = a.block;
    const size_t smem = (size_t)warp_smem(kSmemStack, false) * (block / 32); // of the variants
    if (a.bvh8) { // BVH8-Q kernels (trace_bvh8.cu)
        launch_trace_bvh8(a, st, lc);
        return;
    }
    // the BVH4 and the BVH2's variants trace closest hits only
    const bool variants = !a.wide && !a.counters && !a.any_hit;
    const bool two_phase = variants && a.two_phase && a.phase.state && a.queue && a.queue_count;
    const bool packet = variants && a.packet && a.one_scene, speculative = variants && a.speculative;
    if (a.shadow && ((a.bvh4 && !a.any_hit) || two_phase || packet || speculative)) launch_shadow(*a.shadow, st, lc);
    if (a.bvh4 && !a.any_hit) { // BVH4 kernel (trace_bvh4.cu)
        launch_trace_bvh4(a, st, lc);
        return;
    }
    if (a.any_hit) { // visibility queries (cr_trace_rays with CR_OPT_ANY_HIT)
        launch_bvh2<false, false, true, kSmemStack>(a, st, lc);
        return;
    }
    if (two_phase) {
        const uint32_t grid = (a.n_max + block - 1) / block;
        const uint32_t nb = (a.n_max + 255) / 256;
        k_trace_bvh2_phase<<<grid, block, smem, st>>>(a.scenes, a.slot_scene, a.ray_o, a.ray_d, a.queue, a.queue_count,
                                                      a.n_max, a.hit, a.phase.state, a.phase.susp, a.phase.budget, 0);
        k_susp_count<<<nb, 256, 0, st>>>(a.phase.susp, a.queue_count, a.n_max, a.phase.block_counts);
        launch_scan_counts(a.phase.block_counts, nb, a.phase.count2, st);
        k_susp_scatter<<<nb, 256, 0, st>>>(a.phase.susp, a.queue, a.queue_count, a.n_max, a.phase.block_counts,
                                          a.phase.queue2);
        k_trace_bvh2_phase<<<grid, block, smem, st>>>(a.scenes, a.slot_scene, a.ray_o, a.ray_d, a.phase.queue2,
                                                      a.phase.count2, a.n_max, a.hit, a.phase.state, nullptr,
                                                      0xffffffffu, 1);
        lc.n += 5;
        return;
    }
    if (packet) {
        const uint32_t grid = (a.n_max + block - 1) / block;
        k_trace_bvh2_packet<<<grid, block, smem, st>>>(a.scenes, a.ray_o, a.ray_d, a.queue,
                                                       a.queue_count, a.n_max, a.hit);
        lc.n++;
        return;
    }
    if (speculative) {
        const uint32_t grid = (a.n_max + block - 1) / block;
        k_trace_bvh2_spec<<<grid, block, smem, st>>>(a.scenes, a.slot_scene, a.ray_o, a.ray_d, a.queue, a.queue_count,
                                                     a.n_max, a.hit);
        lc.n++;
        return;
    }
    if (a.counters) launch_bvh2<false, true, false, kSmemStack>(a, st, lc);
    else if (a.stack == 8) launch_bvh2<true, false, false, 8>(a, st, lc);
    else if (a.stack == 32) launch_bvh2<true, false, false, 32>(a, st, lc);
    else launch_bvh2<true, false, false, kSmemStack>(a, st, lc);
}

void launch_hits_to_user(const float4* tris, const int2* hit, uint32_t n, int32_t* prim, float* t, cudaStream_t st,
                         LaunchCount& lc) {
    if (n == 0) return;
    k_hits_to_user<<<(n + 255) / 256, 256, 0, st>>>(tris, hit, n, prim, t);
    lc.n++;
}

} // namespace cr
