// trace_common.cuh -- traversal primitives shared by the BVH2 kernels (trace.cu) and the
// BVH8-Q kernels (trace_bvh8.cu): ray set-up, the conservative slab tests, the watertight
// ray/triangle test, the closest-hit rule and the short traversal stack.
//
// Closest-hit rule, identical for every kernel: accept t > 0 if t < t_best, or t == t_best
// and the original triangle index is smaller.  Boxes are culled only if their entry distance
// exceeds t_best (1 + 2^-16), and no slab test rejects a box that a ray enters:
//   BVH2    records enlarged by kGridSlack, entry and exit offsets moved apart (grid_axis)
//   BVH8-Q  entry and exit offsets of each node moved apart (trace_bvh8.cu)
//   BVH4    offsets moved apart by 2^-22 |o / d|, the exit widened by 1 + 2^-21 (box_hit_nf)
// so every layout returns the same hit bit for bit, up to triangles that a ray misses and the
// triangle test accepts by rounding (behind() keeps out the ones that matter).
#pragma once
#include <cuda_runtime.h>

#include <atomic>

#include "cr_internal.h"
#include "debug_checks.cuh"

namespace cr {
namespace {

constexpr int kSmemStack = 16;  // entries per thread in shared memory
constexpr int kStackTotal = (int)kBvh2StackCapacity; // > BVH2 depth (checked at scene creation)
constexpr float kCullWiden = 1.0f + 0x1.0p-16f;

struct RayPre {
    float ox, oy, oz;
    float ix, iy, iz; // 1 / d (zero components replaced by +-1e-20 first)
    int kz;           // axis of the largest direction component; kx, ky follow it cyclically
    float sx, sy, sz; // shear constants of the watertight test
    float dx, dy, dz;
    // slab offsets for t = fma(plane, 1/d, offset): -o/d biased outward by 2^-22 |o/d|, which
    // bounds the rounding of o/d and of the offset, so the FMA interval contains the one the
    // exact (plane - o) / d form gives (see box_hit_nf in trace_bvh4.cu)
    float lox, loy, loz, hix, hiy, hiz;
};

// component kz, kx = kz + 1, ky = kz + 2 (mod 3) of (x, y, z)
__device__ __forceinline__ float sel_z(float x, float y, float z, int kz) { return kz == 0 ? x : (kz == 1 ? y : z); }
__device__ __forceinline__ float sel_x(float x, float y, float z, int kz) { return kz == 0 ? y : (kz == 1 ? z : x); }
__device__ __forceinline__ float sel_y(float x, float y, float z, int kz) { return kz == 0 ? z : (kz == 1 ? x : y); }

__device__ __forceinline__ RayPre prep_ray(float4 o, float4 d) {
    RayPre r;
    r.ox = o.x;
    r.oy = o.y;
    r.oz = o.z;
    r.dx = d.x;
    r.dy = d.y;
    r.dz = d.z;
    const float tiny = 1e-20f;
    r.ix = 1.0f / (fabsf(d.x) > tiny ? d.x : copysignf(tiny, d.x));
    r.iy = 1.0f / (fabsf(d.y) > tiny ? d.y : copysignf(tiny, d.y));
    r.iz = 1.0f / (fabsf(d.z) > tiny ? d.z : copysignf(tiny, d.z));
    const float ax = fabsf(d.x), ay = fabsf(d.y), az = fabsf(d.z);
    const int kz = ax > ay ? (ax > az ? 0 : 2) : (ay > az ? 1 : 2);
    const float dkz = sel_z(d.x, d.y, d.z, kz);
    r.kz = kz;
    r.sx = sel_x(d.x, d.y, d.z, kz) / dkz;
    r.sy = sel_y(d.x, d.y, d.z, kz) / dkz;
    r.sz = 1.0f / dkz;
    // plane of the lower bound enters first when 1/d >= 0; bias each offset so that the
    // entry distance can only decrease and the exit distance only increase
    const float oix = __fmul_rn(r.ox, r.ix), oiy = __fmul_rn(r.oy, r.iy), oiz = __fmul_rn(r.oz, r.iz);
    const float ex = __fmul_rn(fabsf(oix), 0x1.0p-22f), ey = __fmul_rn(fabsf(oiy), 0x1.0p-22f),
                ez = __fmul_rn(fabsf(oiz), 0x1.0p-22f);
    r.lox = r.ix >= 0.0f ? -oix - ex : -oix + ex;
    r.hix = r.ix >= 0.0f ? -oix + ex : -oix - ex;
    r.loy = r.iy >= 0.0f ? -oiy - ey : -oiy + ey;
    r.hiy = r.iy >= 0.0f ? -oiy + ey : -oiy - ey;
    r.loz = r.iz >= 0.0f ? -oiz - ez : -oiz + ez;
    r.hiz = r.iz >= 0.0f ? -oiz + ez : -oiz - ez;
    return r;
}

#ifndef CR_TRACE_MINMAX3
#define CR_TRACE_MINMAX3 1
#endif
// three-input min / max (one instruction each on sm_100 and later)
__device__ __forceinline__ float min3f(float a, float b, float c) {
#if CR_TRACE_MINMAX3
    float r;
    asm("min.f32 %0, %1, %2, %3;" : "=f"(r) : "f"(a), "f"(b), "f"(c));
    return r;
#else
    return fminf(fminf(a, b), c);
#endif
}
__device__ __forceinline__ float max3f(float a, float b, float c) {
#if CR_TRACE_MINMAX3
    float r;
    asm("max.f32 %0, %1, %2, %3;" : "=f"(r) : "f"(a), "f"(b), "f"(c));
    return r;
#else
    return fmaxf(fmaxf(a, b), c);
#endif
}

// ------------------------------------------------------------------------------------
// The BVH2's 32-byte records (DevBVH2 in cr_internal.h).
//
// A ray against boxes in grid coordinates (the same distances t): a plane at g is met at
// fma(g, i, -og * i) with og the origin in the grid and i = 1 / (d * scale).  With
// u = 2^-24, per axis and as a shift of the plane: og is off by 3 u |og|, i by a relative 2 u,
// the offset by 2 u |og| and the fma by u (|og| + 2); the triangle test adds about
// 8 u (|og| + 2).  Boxes are stored 2^-18 = 64 u larger on every side, and the entry and exit
// offsets move apart by 2^-19 |og| = 32 u |og| each, which covers all of it for any origin, so
// no box that holds a candidate triangle is rejected.  (NaN plane distances, from 1/d that
// overflows, drop out of the minima and maxima: that axis then rejects nothing.)
struct GridRay {
    float ix, iy, iz; // 1 / (d * scale) (zero components of d replaced by +-1e-20 first)
    float nx, ny, nz; // offsets of the entry distances
    float fx, fy, fz; // offsets of the exit distances
    // byte selectors that decode the near and the far plane: the plane of the lower bound is
    // entered first when 1/d >= 0, so a box needs no minima and maxima of its plane distances
    uint32_t snx, sny, snz, sfx, sfy, sfz;
};

__device__ __forceinline__ void grid_axis(float o, float d, float lo, float scale, float& i, float& n, float& f,
                                          uint32_t& sn, uint32_t& sf) {
    const float tiny = 1e-20f;
    const float og = fmaf(o - lo, scale, 0.5f);
    i = 1.0f / ((fabsf(d) > tiny ? d : copysignf(tiny, d)) * scale);
    const float oi = __fmul_rn(og, i), e = __fmul_rn(fabsf(oi), 0x1.0p-19f);
    n = -oi - e;
    f = -oi + e;
    sn = i < 0.0f ? 0x7324u : 0x7104u;
    sf = i < 0.0f ? 0x7104u : 0x7324u;
}

__device__ __forceinline__ GridRay grid_ray(float4 o, float4 d, const SceneDev& sc) {
    GridRay g;
    grid_axis(o.x, d.x, sc.grid_lo[0], sc.grid_scale[0], g.ix, g.nx, g.fx, g.snx, g.sfx);
    grid_axis(o.y, d.y, sc.grid_lo[1], sc.grid_scale[1], g.iy, g.ny, g.fy, g.sny, g.sfy);
    grid_axis(o.z, d.z, sc.grid_lo[2], sc.grid_scale[2], g.iz, g.nz, g.fz, g.snz, g.sfz);
    return g;
}

// A ray's way into another grid, by the record of that step (DevBVH2; a, b its words): the offsets are
// made anew and the reciprocals scaled by powers of two, which is exact, so the errors are those above.
__device__ __forceinline__ void cross_axis(float o, uint32_t lo, uint32_t scale, uint32_t two, float& i, float& n, float& f) {
    const float og = fmaf(o - __uint_as_float(lo), __uint_as_float(scale), 0.5f);
    i = __fmul_rn(i, __uint_as_float(two << 23));
    const float oi = __fmul_rn(og, i), e = __fmul_rn(fabsf(oi), 0x1.0p-19f);
    n = -oi - e;
    f = -oi + e;
}
__device__ __forceinline__ void cross_grid(const RayPre& r, const uint4& a, const uint4& b, GridRay& g) {
    cross_axis(r.ox, a.x, a.w, b.z & 0xffu, g.ix, g.nx, g.fx);
    cross_axis(r.oy, a.y, b.x, b.z >> 8 & 0xffu, g.iy, g.ny, g.fy);
    cross_axis(r.oz, a.z, b.y, b.z >> 16, g.iz, g.nz, g.fz);
}

struct NodeTest {
    float t0, t1; // entry distances of the boxes of child 0, 1 (0 from inside)
    float f0, f1; // exit distances
    int c0, c1;   // links
    // whether the ray enters the box before tcull
    __device__ __forceinline__ bool hit0(float tcull) const { return t0 <= f0 && t0 <= tcull; }
    __device__ __forceinline__ bool hit1(float tcull) const { return t1 <= f1 && t1 <= tcull; }
};

// The float of one 16-bit plane code (bytes: 0, code, 0x3f).
__device__ __forceinline__ float plane_at(uint32_t w, uint32_t sel) {
    return __uint_as_float(__byte_perm(w, 0x3f000000u, sel));
}

// Both child boxes of record `node`.  One 256-bit load fetches the record: half the L1
// wavefronts of a 64-byte record, which set the speed before (measured beside the kernel).
__device__ __forceinline__ NodeTest node_test(const GridRay& g, const uint32_t* __restrict__ nodes, int node) {
    const uint32_t* rec = nodes + kDevNode2Words * (size_t)(uint32_t)node;
    uint32_t w0, w1, w2, w3, w4, w5, w6, w7;
    asm("ld.global.nc.v8.b32 {%0, %1, %2, %3, %4, %5, %6, %7}, [%8];"
        : "=r"(w0), "=r"(w1), "=r"(w2), "=r"(w3), "=r"(w4), "=r"(w5), "=r"(w6), "=r"(w7)
        : "l"(rec));
    NodeTest r;
    r.t0 = fmaxf(max3f(fmaf(plane_at(w0, g.snx), g.ix, g.nx), fmaf(plane_at(w1, g.sny), g.iy, g.ny),
                       fmaf(plane_at(w2, g.snz), g.iz, g.nz)), 0.0f);
    r.t1 = fmaxf(max3f(fmaf(plane_at(w3, g.snx), g.ix, g.nx), fmaf(plane_at(w4, g.sny), g.iy, g.ny),
                       fmaf(plane_at(w5, g.snz), g.iz, g.nz)), 0.0f);
    r.f0 = min3f(fmaf(plane_at(w0, g.sfx), g.ix, g.fx), fmaf(plane_at(w1, g.sfy), g.iy, g.fy),
                           fmaf(plane_at(w2, g.sfz), g.iz, g.fz));
    r.f1 = min3f(fmaf(plane_at(w3, g.sfx), g.ix, g.fx), fmaf(plane_at(w4, g.sfy), g.iy, g.fy),
                           fmaf(plane_at(w5, g.sfz), g.iz, g.fz));
    r.c0 = (int)w6;
    r.c1 = (int)w7;
    return r;
}

// Watertight ray/triangle test (Woop, Benthin, Wald 2013) without the double-precision
// fallback: edge functions of exactly zero count as inside, so shared edges are covered.
// kx and ky are not exchanged for rays that run down the kz axis: that negates U, V, W, det
// and T exactly, which leaves the sign test and t = T / det as they are.
// near (kNear): the hit is nearer than 1/16 of the farthest vertex (along kz), where rounding may have moved it
// past the origin (the error is some 2^-22 of that distance unless the ray all but lies in the plane).
template <bool kNear>
__device__ __forceinline__ bool tri_test(const RayPre& r, float4 a4, float4 b4, float4 c4, float& t_out, bool& near) {
    const float Ax3 = a4.x - r.ox, Ay3 = a4.y - r.oy, Az3 = a4.z - r.oz;
    const float Bx3 = b4.x - r.ox, By3 = b4.y - r.oy, Bz3 = b4.z - r.oz;
    const float Cx3 = c4.x - r.ox, Cy3 = c4.y - r.oy, Cz3 = c4.z - r.oz;
    const float Akx = sel_x(Ax3, Ay3, Az3, r.kz), Aky = sel_y(Ax3, Ay3, Az3, r.kz), Akz = sel_z(Ax3, Ay3, Az3, r.kz);
    const float Bkx = sel_x(Bx3, By3, Bz3, r.kz), Bky = sel_y(Bx3, By3, Bz3, r.kz), Bkz = sel_z(Bx3, By3, Bz3, r.kz);
    const float Ckx = sel_x(Cx3, Cy3, Cz3, r.kz), Cky = sel_y(Cx3, Cy3, Cz3, r.kz), Ckz = sel_z(Cx3, Cy3, Cz3, r.kz);
    const float Ax = __fsub_rn(Akx, __fmul_rn(r.sx, Akz)), Ay = __fsub_rn(Aky, __fmul_rn(r.sy, Akz));
    const float Bx = __fsub_rn(Bkx, __fmul_rn(r.sx, Bkz)), By = __fsub_rn(Bky, __fmul_rn(r.sy, Bkz));
    const float Cx = __fsub_rn(Ckx, __fmul_rn(r.sx, Ckz)), Cy = __fsub_rn(Cky, __fmul_rn(r.sy, Ckz));
    const float U = __fsub_rn(__fmul_rn(Cx, By), __fmul_rn(Cy, Bx));
    const float V = __fsub_rn(__fmul_rn(Ax, Cy), __fmul_rn(Ay, Cx));
    const float W = __fsub_rn(__fmul_rn(Bx, Ay), __fmul_rn(By, Ax));
    if ((U < 0.0f || V < 0.0f || W < 0.0f) && (U > 0.0f || V > 0.0f || W > 0.0f)) return false;
    const float det = __fadd_rn(__fadd_rn(U, V), W);
    if (det == 0.0f) return false;
    const float Az = __fmul_rn(r.sz, Akz), Bz = __fmul_rn(r.sz, Bkz), Cz = __fmul_rn(r.sz, Ckz);
    const float T = __fadd_rn(__fadd_rn(__fmul_rn(U, Az), __fmul_rn(V, Bz)), __fmul_rn(W, Cz));
    const float t = __fdiv_rn(T, det);
    if (!(t > 0.0f)) return false;
    if (kNear) near = t < 0.0625f * max3f(fabsf(Az), fabsf(Bz), fabsf(Cz));
    t_out = t;
    return true;
}

struct Best {
    float t;
    int leaf; // triangle in leaf order, -1 none
};

// Whether a triangle lies behind the origin along an axis, by more than 2^-22 of the origin's coordinate
// (i: any value with the direction component's sign).  Such a triangle is not hit, but the test above can
// say so when it is large and the origin lies just off its plane: a ray that leaves a ground of a
// kilometre met the coplanar triangle beside its own at t = 3e-5.  Exact boxes keep most of these from
// the test; enlarged ones do not.  The vertices are read again (this is rare, see tri_test; kept in
// registers since the test, they cost the traces 4 to 9%, read again 2%), and only the kernels for wide
// scenes look (kWideTri).
__device__ __forceinline__ float4 reload(const float4* p) {
    float4 v;
    asm volatile("ld.global.nc.v4.f32 {%0, %1, %2, %3}, [%4];" : "=f"(v.x), "=f"(v.y), "=f"(v.z), "=f"(v.w) : "l"(p));
    return v;
}
__device__ __forceinline__ bool behind_axis(float o, float i, float a, float b, float c) {
    const float e = __fmul_rn(fabsf(o), 0x1.0p-22f);
    return __float_as_int(i) < 0 ? min3f(a, b, c) > __fadd_rn(o, e) : max3f(a, b, c) < __fsub_rn(o, e);
}
__device__ __forceinline__ bool behind(const RayPre& r, float ix, float iy, float iz, const float4* tri) {
    const float4 a = reload(tri), b = reload(tri + 1), c = reload(tri + 2);
    return behind_axis(r.ox, ix, a.x, b.x, c.x) || behind_axis(r.oy, iy, a.y, b.y, c.y) || behind_axis(r.oz, iz, a.z, b.z, c.z);
}

// kWide: look for triangles behind the origin; ix, iy, iz: values with the signs of the direction's components.
template <bool kWide>
__device__ __forceinline__ void test_leaf(const float4* __restrict__ tris, const RayPre& r, float ix, float iy, float iz,
                                          int skip, uint32_t first,
                                          uint32_t count, Best& best, unsigned long long& n_tri) {
    for (uint32_t i = 0; i < count; ++i) {
        const uint32_t tri = first + i;
        const float4 a = __ldg(&tris[3 * tri + 0]);
        const int orig = __float_as_int(a.w);
        if (orig == skip) continue;
        const float4 b = __ldg(&tris[3 * tri + 1]);
        const float4 c = __ldg(&tris[3 * tri + 2]);
        ++n_tri;
        float t;
        bool near = false;
        // a tie goes to the smaller original index (any hit at exactly tmax is taken)
        if (tri_test<kWide>(r, a, b, c, t, near) &&
            (t < best.t || (t == best.t && (best.leaf < 0 || orig < __float_as_int(__ldg(&tris[3 * best.leaf]).w))))) {
            if constexpr (kWide) {
                if (near && behind(r, ix, iy, iz, &tris[3 * tri])) continue;
            }
            best.t = t;
            best.leaf = (int)tri;
        }
    }
}

#ifndef CR_TRACE_LOCAL_STACK
#define CR_TRACE_LOCAL_STACK 0
#endif
#if CR_TRACE_LOCAL_STACK
// whole stack in a per-thread local array (L1-resident); depth < kStackTotal by construction
#define STACK_PUSH(v) (lstack_all[sp++] = (v))
#define STACK_POP(v) ((v) = lstack_all[--sp])
#else
// first kSmemS entries (the user's constant: kSmemStack, or a template parameter) in shared
// memory, the rest in a local array
// (a push never exceeds the tree depth, which scene creation checks is below kStackTotal)
#define STACK_PUSH(v)                                                                \
    do {                                                                             \
        if (sp < kSmemS) sstack[sp * stride] = (uint32_t)(v);                        \
        else lstack[sp - kSmemS] = (v);                                              \
        ++sp;                                                                        \
    } while (0)
#define STACK_POP(v)                                                                 \
    do {                                                                             \
        --sp;                                                                        \
        (v) = sp < kSmemS ? (int)sstack[sp * stride] : lstack[sp - kSmemS];          \
    } while (0)
#endif


// The same stack with a pointer to the next free shared-memory entry, which saves the index
// arithmetic of every push and pop (1% on the secondary trace); used by the BVH4 kernel.
#define STACK_PUSH_TOP(v)                                                            \
    do {                                                                             \
        if (sp < kSmemS) {                                                           \
            *top = (uint32_t)(v);                                                    \
            top += stride;                                                           \
        } else {                                                                     \
            lstack[sp - kSmemS] = (v);                                               \
        }                                                                            \
        ++sp;                                                                        \
    } while (0)
#define STACK_POP_TOP(v)                                                             \
    do {                                                                             \
        --sp;                                                                        \
        if (sp < kSmemS) {                                                           \
            top -= stride;                                                           \
            (v) = (int)*top;                                                         \
        } else {                                                                     \
            (v) = lstack[sp - kSmemS];                                               \
        }                                                                            \
    } while (0)

// ------------------------------------------------------------------------------------
// Ray sources of the trace kernels.
constexpr uint32_t kTraceChunk = 32; // positions a warp takes at a time
constexpr uint32_t kTraceShare = 2;  // positions of a warp at least (below, warps are spread over the device)
constexpr int kTraceIdle = 8;        // idle lanes of a warp at which they get new rays

// Where a warp's rays come from: positions of a list of n.  A source adds
// load() (the ray at a position; false: none there) and store() (its hit).
//   kPlain  kTraceChunk positions, one per lane, are all a warp traces (grids of any size).
//   kMore   lanes whose ray has ended get further positions of the warp's range, and the warp takes
//           another kTraceChunk from `work` (a device counter, zero before the launch) when its own
//           run out (resident grids, more positions than lanes).
//   kFew    the n positions are spread evenly over the warps of a resident grid, which has more lanes.
enum RangeKind { kPlain, kMore, kFew };

template <RangeKind kKind>
struct WarpRange {
    static constexpr bool kMore = kKind == RangeKind::kMore;
    uint32_t n, next, end;
    uint32_t* work;
    uint32_t first_free; // the first position that `work` hands out
    // block, blocks: this block's place among those that share the list
    __device__ __forceinline__ WarpRange(uint32_t n_, uint32_t* work_, uint32_t block, uint32_t blocks) : n(n_), work(work_) {
        const uint32_t w = (block * blockDim.x + threadIdx.x) >> 5, warps = blocks * blockDim.x >> 5;
        // fewer positions than lanes: the same share for every warp
        const uint32_t each = kKind == RangeKind::kPlain ? kTraceChunk : min(max((n + warps - 1u) / warps, kTraceShare), kTraceChunk);
        next = min(w * each, n);
        end = min(next + each, n);
        first_free = warps * each;
    }
    __device__ __forceinline__ bool more() const { return next < n; }
    // The idle lanes (a mask) get the next positions in lane order, n where the range ends.
    __device__ __forceinline__ uint32_t take(uint32_t idle) {
        const uint32_t lane = threadIdx.x & 31u;
        const uint32_t i = next + __popc(idle & ((1u << lane) - 1u)), e = end;
        if (kMore) {
            next += __popc(idle);
            if (next >= e) {
                next = n;
                if (first_free < n) { // else the first ranges were all there is (a short queue)
                    uint32_t got = 0;
                    if (lane == 0) got = atomicAdd(work, kTraceChunk);
                    got = __shfl_sync(0xffffffffu, got, 0);
                    next = min(got + first_free, n);
                    end = min(next + kTraceChunk, n);
                }
            }
        }
        return i < e ? i : n;
    }
};

// Rays of a queue of slots (or of the slots in order), hits per slot.
template <RangeKind kKind>
struct QueueSrc : WarpRange<kKind> {
    const uint16_t* slot_scene;
    const float4* ray_o;
    const float4* ray_d;
    const int32_t* queue;
    int2* __restrict__ hit;
    static constexpr int idle = kTraceIdle;
    static constexpr bool kProbe = false;
    __device__ __forceinline__ void probe(bool, uint32_t) {}
    __device__ __forceinline__ QueueSrc(uint32_t n, uint32_t* work, const uint16_t* ss, const float4* o, const float4* d,
                                        const int32_t* q, int2* h, uint32_t block, uint32_t blocks)
        : WarpRange<kKind>(n, work, block, blocks), slot_scene(ss), ray_o(o), ray_d(d), queue(q), hit(h) {}
    __device__ __forceinline__ bool load(uint32_t i, int& key, float4& ro, float4& rd) const {
        const int slot = queue ? queue[i] : (int)i;
        ro = ray_o[slot];
        rd = ray_d[slot];
        if (!(rd.w >= 0.0f)) {
            hit[slot] = make_int2(-1, __float_as_int(INFINITY));
            return false;
        }
        key = slot;
        return true;
    }
    __device__ __forceinline__ uint32_t scene(int key) const { return slot_scene ? slot_scene[key] : 0u; }
    __device__ __forceinline__ void store(int key, int leaf, float t, const float4*) const {
        hit[key] = make_int2(leaf, __float_as_int(t));
    }
};

// A caller's rays (8 floats each), optional skip ids and hit arrays.
template <RangeKind kKind>
struct UserSrc : WarpRange<kKind>, UserRays {
    int idle = kTraceIdle;
    // A warp whose rays all run into one octant is taken for a coherent one (camera rays), whose
    // rays end together: it gets new rays only when all of its own have ended (the rule of
    // the render path's camera rays, which the caller's list does not say).
    static constexpr bool kProbe = true;
    __device__ __forceinline__ void probe(bool live, uint32_t oct) {
        idle = __popc(__reduce_or_sync(0xffffffffu, live ? 1u << oct : 0u)) <= 1 ? 32 : kTraceIdle;
    }
    __device__ __forceinline__ UserSrc(uint32_t n, uint32_t* work, const UserRays& u) : WarpRange<kKind>(n, work, blockIdx.x, gridDim.x), UserRays(u) {}
    __device__ __forceinline__ bool load(uint32_t i, int& key, float4& ro, float4& rd) const {
        const float* r = rays + 8 * (size_t)i;
        if (aligned) {
            ro = *reinterpret_cast<const float4*>(r);
            rd = *reinterpret_cast<const float4*>(r + 4);
        } else {
            ro = make_float4(r[0], r[1], r[2], 0.0f);
            rd = make_float4(r[4], r[5], r[6], r[7]);
        }
        ro.w = __int_as_float(skip ? skip[i] : -1);
        if (!(rd.w >= 0.0f)) {
            prim[i] = -1;
            t[i] = INFINITY;
            return false;
        }
        key = (int)i;
        return true;
    }
    __device__ __forceinline__ uint32_t scene(int) const { return 0u; }
    __device__ __forceinline__ void store(int key, int leaf, float tt, const float4* __restrict__ tris) const {
        prim[key] = leaf >= 0 ? __float_as_int(__ldg(&tris[3 * leaf]).w) : -1;
        t[key] = leaf >= 0 ? tt : INFINITY; // a miss of a bounded ray reports inf, not tmax
    }
};

// Shadow rays of next-event estimation, by position of the last shade's group queue (so a
// reuse group's rays run in adjacent lanes, as they were shaded).  A ray whose
// direction record has w = tmax > 0 is traced for visibility only; if nothing blocks it, its
// contribution is added to the path radiance of its slot.  Rays traced are counted.
template <RangeKind kKind>
struct ShadowSrc : WarpRange<kKind> {
    const uint16_t* slot_scene;
    const float4* sh_o;
    const float4* sh_d;
    const float4* sh_c;
    const int32_t* group_queue;
    float4* __restrict__ radiance;
    uint32_t K, traced = 0;
    static constexpr int idle = kTraceIdle;
    static constexpr bool kProbe = false;
    __device__ __forceinline__ void probe(bool, uint32_t) {}
    __device__ __forceinline__ ShadowSrc(uint32_t n, uint32_t* work, const uint16_t* ss, const float4* o, const float4* d,
                                         const float4* c, const int32_t* gq, float4* rad, uint32_t k, uint32_t block,
                                         uint32_t blocks)
        : WarpRange<kKind>(n, work, block, blocks), slot_scene(ss), sh_o(o), sh_d(d), sh_c(c), group_queue(gq), radiance(rad), K(k) {}
    __device__ __forceinline__ bool load(uint32_t i, int& key, float4& ro, float4& rd) {
        const uint32_t g = group_queue ? (uint32_t)group_queue[i / K] : i / K;
        const int slot = (int)(g * K + i % K);
        rd = sh_d[slot];
        if (!(rd.w > 0.0f)) return false;
        ro = sh_o[slot];
        key = slot;
        ++traced;
        return true;
    }
    __device__ __forceinline__ uint32_t scene(int key) const { return slot_scene[key]; }
    __device__ __forceinline__ void store(int key, int leaf, float, const float4*) const {
        if (leaf >= 0) return;
        const float4 c = sh_c[key];
        const float4 L = radiance[key];
        radiance[key] = make_float4(__fadd_rn(L.x, c.x), __fadd_rn(L.y, c.y), __fadd_rn(L.z, c.z), L.w);
    }
    __device__ __forceinline__ void add_traced(unsigned long long* n_traced) const {
        const uint32_t b = __reduce_add_sync(0xffffffffu, traced);
        if ((threadIdx.x & 31) == 0 && b) atomicAdd(n_traced, (unsigned long long)b);
    }
};

// Node visits and triangle tests of a counting pass, summed over the warp.
__device__ __forceinline__ void add_counts(unsigned long long* counters, unsigned long long n_node,
                                           unsigned long long n_tri) {
    for (int off = 16; off > 0; off >>= 1) {
        n_node += __shfl_down_sync(0xffffffffu, n_node, off);
        n_tri += __shfl_down_sync(0xffffffffu, n_tri, off);
    }
    if ((threadIdx.x & 31) == 0) {
        atomicAdd(&counters[0], n_node);
        atomicAdd(&counters[1], n_tri);
    }
}

// Launches of a kernel with more than 48 KB of shared memory per block need the opt-in first, and so does
// the question how many of them are resident.
template <auto kKernel>
static void allow_smem(size_t smem) {
    if (smem > 48 * 1024) cudaFuncSetAttribute(kKernel, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)smem);
}

// Blocks of a trace kernel that are resident on the current device at once (0: unknown).
template <auto kKernel>
static uint32_t resident_blocks(int block, size_t smem) {
    // per device and block size (block sizes are multiples of 32 up to 512)
    static std::atomic<uint32_t> known[64][17];
    int dev = 0;
    if (cudaGetDevice(&dev) != cudaSuccess || dev < 0 || dev >= 64) return 0;
    std::atomic<uint32_t>& r = known[dev][block / 32];
    uint32_t v = r.load(std::memory_order_relaxed);
    if (!v) {
        int sms = 0, nb = 0;
        allow_smem<kKernel>(smem);
        if (cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, dev) != cudaSuccess ||
            cudaOccupancyMaxActiveBlocksPerMultiprocessor(&nb, kKernel, block, smem) != cudaSuccess || sms <= 0 || nb <= 0)
            return 0;
        v = (uint32_t)sms * (uint32_t)nb;
        r.store(v, std::memory_order_relaxed);
    }
    return v;
}

// Blocks for n positions, one per lane.
static inline uint32_t blocks_for(uint32_t n, int block) { return n / (uint32_t)block + (n % (uint32_t)block ? 1u : 0u); }
// Blocks for n positions spread kTraceShare to a warp, at most `most`.
static inline uint32_t spread_blocks(uint32_t n, int block, uint32_t most) {
    const uint32_t want = blocks_for(n, block / 32 * (int)kTraceShare);
    return want < most ? want : most;
}

} // namespace
} // namespace cr
