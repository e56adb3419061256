// Device functions shared by the megakernel (jr_kernels.cu) and the
// wavefront pipeline (jr_wavefront.cu): Philox, vector helpers, BVH
// traversal, BSDF sampling, the PSS path integrand.
#pragma once
#include <cuda_runtime.h>
#include <math.h>
#include <stdint.h>

#include "../../include/jr.h"
#include "jr_internal.h"

namespace jr {
namespace {

// ------------------------------------------------------------------ Philox
// Philox4x32-10 (Salmon, Moraes, Dror, Shaw, SC'11).
__device__ __forceinline__ uint4 philox4x32_10(uint4 c, uint2 k) {
#pragma unroll
    for (int r = 0; r < 10; ++r) {
        if (r > 0) {
            k.x += 0x9E3779B9u;
            k.y += 0xBB67AE85u;
        }
        const uint32_t hi0 = __umulhi(0xD2511F53u, c.x), lo0 = 0xD2511F53u * c.x;
        const uint32_t hi1 = __umulhi(0xCD9E8D57u, c.z), lo1 = 0xCD9E8D57u * c.z;
        c = make_uint4(hi1 ^ c.y ^ k.x, lo1, hi0 ^ c.w ^ k.y, lo0);
    }
    return c;
}

__device__ __forceinline__ uint4 draw(uint64_t seed, uint32_t tag, uint32_t block, uint32_t chain, uint64_t step) {
    return philox4x32_10(make_uint4(block + 256u * tag, chain, (uint32_t)step, (uint32_t)(step >> 32)),
                         make_uint2((uint32_t)seed, (uint32_t)(seed >> 32)));
}

// (r >> 8) * 2^-24: exact in float, in [0, 1).
__device__ __forceinline__ float u01(uint32_t r) { return (float)(r >> 8) * 5.9604644775390625e-8f; }

// ------------------------------------------------------------------ vectors
__device__ __forceinline__ float3 f3(float x, float y, float z) { return make_float3(x, y, z); }
__device__ __forceinline__ float3 operator+(float3 a, float3 b) { return f3(a.x + b.x, a.y + b.y, a.z + b.z); }
__device__ __forceinline__ float3 operator-(float3 a, float3 b) { return f3(a.x - b.x, a.y - b.y, a.z - b.z); }
__device__ __forceinline__ float3 operator*(float3 a, float s) { return f3(a.x * s, a.y * s, a.z * s); }
__device__ __forceinline__ float3 mul(float3 a, float3 b) { return f3(a.x * b.x, a.y * b.y, a.z * b.z); }
__device__ __forceinline__ float dot(float3 a, float3 b) { return a.x * b.x + a.y * b.y + a.z * b.z; }
__device__ __forceinline__ float3 cross(float3 a, float3 b) {
    return f3(a.y * b.z - a.z * b.y, a.z * b.x - a.x * b.z, a.x * b.y - a.y * b.x);
}
__device__ __forceinline__ float3 normalize(float3 a) { return a * (1.0f / sqrtf(dot(a, a))); }
__device__ __forceinline__ float lum(float3 c) { return 0.2126f * c.x + 0.7152f * c.y + 0.0722f * c.z; }

// Orthonormal basis around unit n (Duff et al., JCGT 2017).
__device__ __forceinline__ void onb(float3 n, float3& t, float3& b) {
    const float sign = copysignf(1.0f, n.z);
    const float a = -1.0f / (sign + n.z);
    const float bb = n.x * n.y * a;
    t = f3(1.0f + sign * n.x * n.x * a, sign * bb, -sign * n.x);
    b = f3(bb, sign + n.y * n.y * a, -n.y);
}

__device__ __forceinline__ float wrap01(float y) {
    const float w = y - floorf(y);
    return w >= 1.0f ? 0.0f : w;
}

// ------------------------------------------------------------------ traversal
constexpr int kSentinel = INT32_MIN;

// Work counters of the instrumented kernel variant (compiled out otherwise).
struct Work {
    uint32_t rays = 0, nodes = 0, tris = 0;
};

// Three-input float min/max (PTX min/max with three sources, sm_100+): one
// instruction where two-input chains take two.
__device__ __forceinline__ float fmin3(float a, float b, float c) {
    float d;
    asm("min.f32 %0, %1, %2, %3;" : "=f"(d) : "f"(a), "f"(b), "f"(c));
    return d;
}
__device__ __forceinline__ float fmax3(float a, float b, float c) {
    float d;
    asm("max.f32 %0, %1, %2, %3;" : "=f"(d) : "f"(a), "f"(b), "f"(c));
    return d;
}

// A ray prepared for slab tests, plus the resumable state of its traversal.
// The stack lives with the caller (per-thread local memory).
struct Trav {
    float3 o, d;
    float ix, iy, iz, ox, oy, oz;
    float tb;          // closest hit so far
    int best, best_id;  // its leaf-order record and original triangle index
    int ref, sp;        // node/leaf ref being visited, stack depth
    uint32_t visits;
    uint32_t oct;       // ray octant: bit 4 + a set when the direction's axis-a component is negative
};

__device__ __forceinline__ void trav_begin_at(Trav& r, float3 o, float3 d, int root) {
    r.o = o;
    r.d = d;
    const float dx = fabsf(d.x) < 1e-20f ? copysignf(1e-20f, d.x) : d.x;
    const float dy = fabsf(d.y) < 1e-20f ? copysignf(1e-20f, d.y) : d.y;
    const float dz = fabsf(d.z) < 1e-20f ? copysignf(1e-20f, d.z) : d.z;
    r.ix = 1.0f / dx;
    r.iy = 1.0f / dy;
    r.iz = 1.0f / dz;
    r.ox = o.x * r.ix;
    r.oy = o.y * r.iy;
    r.oz = o.z * r.iz;
    r.oct = (r.ix < 0.0f ? 16u : 0u) | (r.iy < 0.0f ? 32u : 0u) | (r.iz < 0.0f ? 64u : 0u);
    r.tb = INFINITY;
    r.best = -1;
    r.best_id = INT32_MAX;
    r.ref = root;
    r.sp = 0;
    r.visits = 0;
}
__device__ __forceinline__ void trav_begin(const SceneView& s, Trav& r, float3 o, float3 d) {
    trav_begin_at(r, o, d, s.root);
}

// Order two (distance, ref) pairs so that the nearer comes first.
__device__ __forceinline__ void cswap(float& ta, int& ra, float& tb, int& rb) {
    const bool sw = tb < ta;
    const float t = sw ? tb : ta;
    tb = sw ? ta : tb;
    ta = t;
    const int q = sw ? rb : ra;
    rb = sw ? ra : rb;
    ra = q;
}

// Two FP32 values in one 64-bit register pair, and the packed fused multiply-add
// and multiply (sm_100+): each half is the scalar operation's result.
__device__ __forceinline__ unsigned long long pack_f32x2(float a, float b) {
    unsigned long long r;
    asm("mov.b64 %0, {%1, %2};" : "=l"(r) : "f"(a), "f"(b));
    return r;
}
__device__ __forceinline__ void fma_f32x2(float a0, float a1, unsigned long long b, unsigned long long c, float& d0,
                                          float& d1) {
    unsigned long long r;
    asm("fma.rn.f32x2 %0, %1, %2, %3;" : "=l"(r) : "l"(pack_f32x2(a0, a1)), "l"(b), "l"(c));
    asm("mov.b64 {%0, %1}, %2;" : "=f"(d0), "=f"(d1) : "l"(r));
}

// Plane distances p * i - o of one plane of the four children.
__device__ __forceinline__ void plane4(const float4 p, float i, float o, float (&t)[4]) {
    const unsigned long long ii = pack_f32x2(i, i), oo = pack_f32x2(-o, -o);
    fma_f32x2(p.x, p.y, ii, oo, t[0], t[1]);
    fma_f32x2(p.z, p.w, ii, oo, t[2], t[3]);
}

// Which of the traversal's watchdogs a launch has to check (trav_checks in
// jr_internal.h decides on the host):
//   kCheckNone    neither can fire: a ray visits a node at most once, so a visit
//                 budget of at least the node count is never exceeded, and the
//                 builder knows the deepest stack a traversal can need;
//   kCheckVisits  visits are counted, and the caller compares them with the
//                 budget once per round (a ray over it is a miss either way,
//                 whatever it did in the rest of the round);
//   kCheckAll     both, at every visit.
// The checks cost a node visit 7 % of the path kernel's time (512^2 Cornell +
// spheres: 12.20 with, 11.53 ms without for 16 steps of 2^20 chains).
//
// Visit inner node r.ref of the 4-wide BVH: slab-test its children against
// [0, tb], descend to the nearest hit child and push the other hit children
// (the next nearest last, up to the order of the farthest two), or pop.
// Returns false (and sets a status bit) if a checked limit ran out: the ray
// then counts as a miss.
//
// The visit is bound by issue slots and by the latency of its loads:
//  * The node's 16-byte chunks lie at chunk ^ (node & 7) (swizzle_nodes_kernel):
//    a warp's lanes read the same chunk of different nodes, and every node
//    starts on a 128-byte line, so unswizzled loads all hit the same four L1
//    banks (43 % of the L1 data pipe's cycles at 12 active lanes).  Measured
//    13.10 -> 12.63 ms (Cornell + spheres), 3.40 -> 3.17 ms (2M-triangle
//    terrain, 4 steps of 2^20 chains).
//  * The 24 plane distances are packed FMAs: half the instructions, the same
//    values (13.10 -> 12.77 ms alone).
//  * Three comparators instead of a full sorting network: the nearest child is
//    exact, and so is the order of two hits; with three or more the order of
//    the others is approximate, which costs fewer visits than the two
//    comparators cost instructions (16 steps of 2^20 chains on Cornell + spheres 9.41
//    ms against 9.53, 2^21 samples of path tracing 1.24 ms against 1.27).  That is not so
//    where the rays cross many boxes that overlap: with kSorted, the full network, the
//    batch megakernel takes 3 rooms of 10 % of their pixels in 519 us instead of 702,
//    16 whole rooms in 20.6 ms instead of 22.0.  The closest hit does not depend on the order;
//    which rays a limit stops does, so where one can fire the order is always the
//    full one (the 2M-triangle terrain, 4 steps of 2^20 chains: 3.02 -> 3.00 ms).
enum TravCheck { kCheckNone = 0, kCheckVisits = 1, kCheckAll = 2 };

template <int kCheck, bool kCount, bool kSorted = false>
__device__ __forceinline__ bool trav_node(const SceneView& s, Trav& r, int* stack, unsigned& status, Work& work) {
    if constexpr (kCheck != kCheckNone) ++r.visits;
    if constexpr (kCheck == kCheckAll) {
        if (r.visits > s.visit_budget) {
            status |= JR_STATUS_TRAVERSAL;
            return false;
        }
    }
    if constexpr (kCount) work.nodes++;
    // The planes are stored lo, hi per axis.  For a positive direction
    // component the lo plane is met first, for a negative one the hi plane:
    // (lo * i - o) <= (hi * i - o) for i > 0 and the reverse for i < 0, and
    // both sides round monotonically, so for finite ray data the octant picks
    // exactly the values min and max would pick (with a NaN in the ray the two
    // forms differ, and such a ray carries no contribution either way).
    const char* n = reinterpret_cast<const char*>(s.nodes + r.ref);
    const uint32_t key = ((uint32_t)r.ref & 7u) << 4;
    const uint32_t kx = key ^ (r.oct & 16u), ky = key ^ ((r.oct >> 1) & 16u), kz = key ^ ((r.oct >> 2) & 16u);
    auto chunk = [&](uint32_t at) { return __ldg(reinterpret_cast<const float4*>(n + at)); };
    const float4 nx = chunk(kx), fx = chunk(kx ^ 16u);
    const float4 ny = chunk(ky ^ 32u), fy = chunk(ky ^ 48u);
    const float4 nz = chunk(kz ^ 64u), fz = chunk(kz ^ 80u);
    int4 rf = __ldg(reinterpret_cast<const int4*>(n + (key ^ 96u)));
    float ax[4], ay[4], az[4], bx[4], by[4], bz[4], t[4];
    plane4(nx, r.ix, r.ox, ax);
    plane4(fx, r.ix, r.ox, bx);
    plane4(ny, r.iy, r.oy, ay);
    plane4(fy, r.iy, r.oy, by);
    plane4(nz, r.iz, r.oz, az);
    plane4(fz, r.iz, r.oz, bz);
    // Entry distance of each child box in [0, tb], or +inf for a miss (an empty
    // slot's box always misses).  The far distance is scaled up by 2 ulp so that
    // a ray grazing a face of a box still enters it.
#pragma unroll
    for (int j = 0; j < 4; ++j) {
        const float tn = fmax3(ax[j], ay[j], fmaxf(az[j], 0.0f));
        const float tf = fmin3(bx[j], by[j], fminf(bz[j], r.tb));
        t[j] = tn <= tf * 1.00000024f ? tn : INFINITY;
    }
    cswap(t[0], rf.x, t[1], rf.y);
    cswap(t[2], rf.z, t[3], rf.w);
    cswap(t[0], rf.x, t[2], rf.z);
    if constexpr (kSorted || kCheck != kCheckNone) {
        cswap(t[1], rf.y, t[3], rf.w);
        cswap(t[1], rf.y, t[2], rf.z);
    }
    if constexpr (kCheck == kCheckAll) {
        const int pushes = (t[1] < INFINITY) + (t[2] < INFINITY) + (t[3] < INFINITY);
        if (r.sp + pushes > s.stack_limit) {
            status |= JR_STATUS_STACK;
            return false;
        }
    }
    if (t[3] < INFINITY) stack[r.sp++] = rf.w;
    if (t[2] < INFINITY) stack[r.sp++] = rf.z;
    if (t[1] < INFINITY) stack[r.sp++] = rf.y;
    if (t[0] < INFINITY) r.ref = rf.x;
    else r.ref = r.sp > 0 ? stack[--r.sp] : kSentinel;
    return true;
}

// kCheckVisits: whether ray r has used up its visit budget (called once per
// round; the caller then treats the ray as a miss).
template <int kCheck>
__device__ __forceinline__ bool over_budget(const SceneView& s, const Trav& r, unsigned& status) {
    if constexpr (kCheck == kCheckVisits) {
        if (r.visits > s.visit_budget) {
            status |= JR_STATUS_TRAVERSAL;
            return true;
        }
    }
    return false;
}

// Test the triangles of leaf `leaf` (Moller-Trumbore, JGT 1997; ties on equal
// t to the smaller original index) against the ray, updating the closest hit.
// Branch-free: every quantity is computed and one predicate takes the hit (the
// early-out form diverged per triangle; measured +0.5 % on the path kernel).
template <bool kCount>
__device__ __forceinline__ void trav_test_leaf(const SceneView& s, Trav& r, int leaf, Work& work) {
    const int enc = ~leaf;
    const int first = enc >> 3, cnt = (enc & 7) + 1;
    if constexpr (kCount) work.tris += (uint32_t)cnt;
    for (int k = first; k < first + cnt; ++k) {
        const TriRecord* tr = s.tris + k;
        const float4 q0 = __ldg(&tr->v0_id), q1 = __ldg(&tr->e1_mat), q2 = __ldg(&tr->e2);
        const float3 e1 = f3(q1.x, q1.y, q1.z), e2 = f3(q2.x, q2.y, q2.z);
        const float3 pv = cross(r.d, e2);
        const float det = dot(e1, pv);
        const float inv = 1.0f / det;
        const float3 tv = r.o - f3(q0.x, q0.y, q0.z);
        const float u = dot(tv, pv) * inv;
        const float3 qv = cross(tv, e1);
        const float v = dot(r.d, qv) * inv;
        const float t = dot(e2, qv) * inv;
        const int id = __float_as_int(q0.w);
        const bool hit = det != 0.0f && !(u < 0.0f || u > 1.0f) && !(v < 0.0f || u + v > 1.0f) && t > 0.0f &&
                         (t < r.tb || (t == r.tb && id < r.best_id));
        r.tb = hit ? t : r.tb;
        r.best = hit ? k : r.best;
        r.best_id = hit ? id : r.best_id;
    }
}

// Test the triangles of leaf r.ref, then pop.  Returns false when the ray is done.
template <bool kCount>
__device__ __forceinline__ bool trav_leaf(const SceneView& s, Trav& r, const int* stack, Work& work) {
    trav_test_leaf<kCount>(s, r, r.ref, work);
    r.ref = r.sp > 0 ? stack[--r.sp] : kSentinel;
    return r.ref != kSentinel;
}

// The inner-node loop of a warp-synchronous traversal round ends once at most
// kSearchExit lanes are still on their way to a leaf (after at least one node
// visit), instead of when none is: the few lanes with the longest way no
// longer hold the warp's other lanes, which test their leaves and go on; the
// rest carry on in the next round.  Measured on the 512^2 Cornell + spheres
// workload (look-ahead windows, two visits per vote), relative to an exit at 6:
// 0.96 (4), 1.014 (8), 1.015 (10), 1.008 (14); with one visit per vote and an exit
// at 0, 0.87.  The exit waits while the searching lanes outnumber
// the others (a sparse warp, late in a drain, has nobody to release and would
// only pay an extra round per node visit).
constexpr int kSearchExit = 8;
__device__ __forceinline__ bool search_done(unsigned searching, unsigned tracing) {
    const int ns = __popc(searching);
    return ns <= kSearchExit && 2 * ns <= __popc(tracing);
}

// Closest hit for the lanes in `mask`, which must all call together (lanes
// without a ray pass want = false).  Warp-synchronous while-while traversal
// (Aila & Laine, HPG 2009): each inner-node round and each leaf round ends in
// a __any_sync over `mask`, so the lanes reconverge every iteration instead of
// drifting apart under independent thread scheduling.  Returns the leaf-order
// record index or -1; t_out gets the hit distance.
template <int kCheck, bool kCount, bool kSorted = false>
__device__ __forceinline__ int closest_hit(const SceneView& s, unsigned mask, bool want, float3 o, float3 d,
                                           float& t_out, unsigned& status, Work& work) {
    Trav r;
    trav_begin(s, r, o, d);
    bool active = want && s.root != kSentinel;
    if constexpr (kCount) work.rays += want ? 1u : 0u;
    int stack[kStackSize];
    while (__any_sync(mask, active)) {
        const unsigned tracing = __ballot_sync(mask, active);
        if (__any_sync(mask, active && r.ref >= 0)) {
            do {  // one vote per node visit: it ends the loop when nobody searches, too
                if (active && r.ref >= 0 && !trav_node<kCheck, kCount, kSorted>(s, r, stack, status, work)) {
                    active = false;
                    r.best = -1;
                }
            } while (!search_done(__ballot_sync(mask, active && r.ref >= 0), tracing));
            if (active && over_budget<kCheck>(s, r, status)) {
                active = false;
                r.best = -1;
            }
        }
        if (active && r.ref < 0) active = r.ref != kSentinel && trav_leaf<kCount>(s, r, stack, work);
    }
    t_out = r.best >= 0 ? r.tb : INFINITY;
    return r.best;
}

// ------------------------------------------------------------------ BSDFs
// Exact unpolarised Fresnel reflectance of a smooth dielectric interface.
__device__ __forceinline__ float fresnel(float cos_i, float eta_i, float eta_t, float& cos_t) {
    const float e = eta_i / eta_t;
    const float sin2_t = e * e * (1.0f - cos_i * cos_i);
    if (sin2_t >= 1.0f) {
        cos_t = 0.0f;
        return 1.0f;
    }
    cos_t = sqrtf(1.0f - sin2_t);
    const float rs = (eta_i * cos_i - eta_t * cos_t) / (eta_i * cos_i + eta_t * cos_t);
    const float rp = (eta_t * cos_i - eta_i * cos_t) / (eta_t * cos_i + eta_i * cos_t);
    return 0.5f * (rs * rs + rp * rp);
}

// The modified Phong lobe about the mirror direction, weight rho (n+2)/(n+1) cos_i,
// with every rounding written out: left to the compiler, which product of a sum of
// two becomes the fused one differs between kernels, and a step's state would depend
// on the kernel that ran it (21 of 2^20 chains after 16 steps of Cornell + spheres
// differed in the last bit of F, and a restored checkpoint with them).  The order
// is the one that the compiler most often takes; it costs nothing (9.41 ms for
// those steps before and after; a call that is not inlined fixes it, too, at 9.51).
// kFusedMirror: the mirror direction's product is fused for the chains; path
// tracing, whose FP64 sums keep the bits they have always had, rounds it by itself.
__device__ __forceinline__ float dot_rn(float3 a, float3 b) {
    return __fmaf_rn(a.z, b.z, __fmaf_rn(a.x, b.x, __fmul_rn(a.y, b.y)));
}
__device__ __forceinline__ float mix_rn(float t, float st, float b, float sb, float r, float sr) {
    return __fmaf_rn(r, sr, __fmaf_rn(t, st, __fmul_rn(b, sb)));
}
struct PhongFrame {
    float3 r, t, b;  // mirror direction and the basis around it
    float cos_a, sin_a, sn, cs;
};
template <bool kFusedMirror = true>
__device__ __forceinline__ PhongFrame phong_frame(const Material& m, float3 d, float3 ns, float u1, float u2) {
    PhongFrame q;
    const float k = -__fmul_rn(2.0f, dot_rn(d, ns));
    if constexpr (kFusedMirror)
        q.r = f3(__fmaf_rn(ns.x, k, d.x), __fmaf_rn(ns.y, k, d.y), __fmaf_rn(ns.z, k, d.z));
    else
        q.r = f3(__fadd_rn(d.x, __fmul_rn(ns.x, k)), __fadd_rn(d.y, __fmul_rn(ns.y, k)),
                 __fadd_rn(d.z, __fmul_rn(ns.z, k)));
    q.cos_a = powf(__fsub_rn(1.0f, u1), m.phong_inv_n1);
    q.sin_a = sqrtf(fmaxf(__fmaf_rn(-q.cos_a, q.cos_a, 1.0f), 0.0f));
    sincospif(__fmul_rn(2.0f, u2), &q.sn, &q.cs);
    const float sign = copysignf(1.0f, q.r.z);  // onb
    const float a = __fdiv_rn(-1.0f, __fadd_rn(sign, q.r.z));
    const float bb = __fmul_rn(__fmul_rn(q.r.x, q.r.y), a);
    q.t = f3(__fmaf_rn(__fmul_rn(__fmul_rn(sign, q.r.x), q.r.x), a, 1.0f), __fmul_rn(sign, bb),
             __fmul_rn(-sign, q.r.x));
    q.b = f3(bb, __fmaf_rn(__fmul_rn(q.r.y, q.r.y), a, sign), -q.r.y);
    return q;
}
__device__ __forceinline__ float3 phong_direction(const PhongFrame& q) {
    const float st = __fmul_rn(q.sin_a, q.cs), sb = __fmul_rn(q.sin_a, q.sn);
    return f3(mix_rn(q.t.x, st, q.b.x, sb, q.r.x, q.cos_a), mix_rn(q.t.y, st, q.b.y, sb, q.r.y, q.cos_a),
              mix_rn(q.t.z, st, q.b.z, sb, q.r.z, q.cos_a));
}
__device__ __forceinline__ float3 phong_weight(const Material& m, float cos_i) {
    const float k = __fmul_rn(m.phong_scale, cos_i);
    return f3(__fmul_rn(m.albedo.x, k), __fmul_rn(m.albedo.y, k), __fmul_rn(m.albedo.z, k));
}
template <bool kFusedMirror>
__device__ __forceinline__ bool phong_lobe(const Material& m, float3 d, float3 ns, float u1, float u2, float3& wi,
                                           float3& w) {
    wi = phong_direction(phong_frame<kFusedMirror>(m, d, ns, u1, u2));
    const float cos_i = dot_rn(wi, ns);
    if (cos_i <= 0.0f) return false;
    w = phong_weight(m, cos_i);
    return true;
}

// Sample the continuation direction; returns false when the path ends.
template <bool kFusedMirror = true>
__device__ __forceinline__ bool scatter(const Material& m, float3 d, float3 ng, float u1, float u2, float3& wi,
                                        float3& w) {
    if (m.type == JR_MAT_DIELECTRIC) {
        float cos_i = -dot(d, ng);
        float eta_i = 1.0f, eta_t = m.ior;
        float3 nn = ng;
        if (cos_i < 0.0f) {
            cos_i = -cos_i;
            eta_i = m.ior;
            eta_t = 1.0f;
            nn = ng * -1.0f;
        }
        float cos_t;
        const float R = fresnel(cos_i, eta_i, eta_t, cos_t);
        if (u1 < R) {
            wi = d + nn * (2.0f * cos_i);
        } else {
            const float e = eta_i / eta_t;
            wi = d * e + nn * (e * cos_i - cos_t);
        }
        w = f3(1.0f, 1.0f, 1.0f);
        return true;
    }
    const float3 ns = dot(d, ng) < 0.0f ? ng : ng * -1.0f;
    float3 t, b;
    if (m.type == JR_MAT_LAMBERT) {
        // cosine-weighted hemisphere (Malley's method); weight = albedo
        const float r = sqrtf(u1);
        float sn, cs;
        sincospif(2.0f * u2, &sn, &cs);
        const float lz = sqrtf(fmaxf(1.0f - u1, 0.0f));
        onb(ns, t, b);
        wi = t * (r * cs) + b * (r * sn) + ns * lz;
        w = m.albedo;
        return m.albedo.x > 0.0f || m.albedo.y > 0.0f || m.albedo.z > 0.0f;
    }
    return phong_lobe<kFusedMirror>(m, d, ns, u1, u2, wi, w);
}

// ------------------------------------------------------------------ integrand
// PSS path contribution F(y) (the target of Section 4 is p = lum(F)).  y[d] is
// read at y[d * ys]: film point (y0, y1), bounce b uses (y_{2+2b}, y_{3+2b}).
// Emission (one-sided) is collected at every vertex; a miss ends the path.
// Camera ray through film point (y0, y1).
__device__ __forceinline__ void camera_ray(const SceneView& s, float y0, float y1, float3& o, float3& d) {
    const float3 cf = f3(s.cam[3], s.cam[4], s.cam[5]);
    const float3 cr = f3(s.cam[6], s.cam[7], s.cam[8]);
    const float3 cu = f3(s.cam[9], s.cam[10], s.cam[11]);
    o = f3(s.cam[0], s.cam[1], s.cam[2]);
    d = normalize(cf + cr * (2.0f * y0 - 1.0f) + cu * (1.0f - 2.0f * y1));
}

// One path vertex: the ray (o, d) hit record k at distance t.  Adds the
// one-sided emission T * L_e to F, and unless v == depth samples the
// continuation with (u1, u2) = (y_{2+2v}, y_{3+2v}).  Returns true if the path
// continues, with (o, d, T) updated to the next ray.
template <bool kFusedMirror = true>
__device__ __forceinline__ bool shade_vertex(const SceneView& s, int k, float t, int v, int depth, float u1,
                                             float u2, float3& o, float3& d, float3& T, float3& F) {
    const TriRecord* tr = s.tris + k;
    const float4 q1 = __ldg(&tr->e1_mat), q2 = __ldg(&tr->e2);
    const Material m = s.mats[__float_as_int(q1.w)];
    const float3 ng = normalize(cross(f3(q1.x, q1.y, q1.z), f3(q2.x, q2.y, q2.z)));
    const float3 p = o + d * t;
    if (m.emits && -dot(d, ng) > 0.0f) F = F + mul(T, m.emission);
    if (v == depth) return false;
    float3 wi, w;
    if (!scatter<kFusedMirror>(m, d, ng, u1, u2, wi, w)) return false;
    T = mul(T, w);
    if (T.x == 0.0f && T.y == 0.0f && T.z == 0.0f) return false;
    const float3 off = dot(wi, ng) >= 0.0f ? ng : ng * -1.0f;
    const float mx = fmaxf(fmaxf(fabsf(p.x), fabsf(p.y)), fabsf(p.z));
    o = p + off * (1e-4f * (1.0f + mx));
    d = wi;
    return true;
}

__device__ __forceinline__ float3 finite_or_zero(float3 F, unsigned& status) {
    if (!isfinite(F.x) || !isfinite(F.y) || !isfinite(F.z)) {
        status |= JR_STATUS_NONFINITE;
        return f3(0.f, 0.f, 0.f);
    }
    return F;
}

// The integrand for the lanes in `mask` (all of which must call together;
// lanes with want = false only keep the warp in step).  The bounce loop runs
// until no lane in the warp has a live path.
template <int kCheck, bool kCount, bool kFusedMirror = true, bool kSorted = false>
__device__ __forceinline__ float3 eval_path_w(const SceneView& s, unsigned mask, bool want, int depth, const float* y,
                                              uint32_t ys, int32_t* ids, uint64_t id_stride, unsigned& status,
                                              Work& work) {
    float3 F = f3(0.f, 0.f, 0.f), T = f3(1.f, 1.f, 1.f);
    float3 o = f3(0.f, 0.f, 1.f), d = f3(0.f, 0.f, 1.f);
    if (want) camera_ray(s, y[0], y[ys], o, d);
    if (want && ids)
        for (int v = 0; v <= depth; ++v) ids[v * id_stride] = -1;
    bool alive = want;
    for (int v = 0; v <= depth; ++v) {
        if (!__any_sync(mask, alive)) break;
        float t;
        const int k = closest_hit<kCheck, kCount, kSorted>(s, mask, alive, o, d, t, status, work);
        if (alive) {
            if (k < 0) {
                alive = false;
            } else {
                if (ids) ids[v * id_stride] = __float_as_int(__ldg(&s.tris[k].v0_id.w));
                const float u1 = v < depth ? y[(2 + 2 * v) * ys] : 0.0f;
                const float u2 = v < depth ? y[(3 + 2 * v) * ys] : 0.0f;
                alive = shade_vertex<kFusedMirror>(s, k, t, v, depth, u1, u2, o, d, T, F);
            }
        }
    }
    return want ? finite_or_zero(F, status) : F;
}

template <int kCheck, bool kFusedMirror = true>
__device__ __forceinline__ float3 eval_path(const SceneView& s, unsigned mask, bool want, int depth, const float* y,
                                            uint32_t ys, int32_t* ids, uint64_t id_stride, unsigned& status) {
    Work w;
    return eval_path_w<kCheck, false, kFusedMirror>(s, mask, want, depth, y, ys, ids, id_stride, status, w);
}

// ------------------------------------------------------------------ persistent path tracing
// Whole paths by persistent warps.  A lane keeps its path (ray, throughput T,
// vertex v) in registers and moves between three states: traversing its current
// ray; waiting to shade (its closest hit is known); idle (no path).  Traversal
// rounds are warp-synchronous while-while rounds with speculative traversal
// (Aila & Laine 2009): a lane that meets a leaf postpones it and keeps descending
// inner nodes until all but kSearchExit lanes hold a leaf.  A warp shades its
// waiting lanes together once kShadeBatch of them wait, or once they are at least
// as many as the traversing lanes (measured: 1.22 -> 1.25e9 chain steps/s against
// the batch rule alone); a shaded path either continues with its next ray or
// ends.  Idle lanes take new paths once kRefill of them are idle, so a warp does
// not idle for its longest path; a new path starts at the camera ray through its
// film point with T = 1, F = 0.
//
// Where paths come from and where F goes is the source's:
//   drained          (warp-uniform) no path is left to take
//   take(idle, mine, y0, y1)  all lanes call; the lanes with mine = true are the
//                    idle ones; true: this lane has a new path with film point
//                    (y0, y1)
//   camera(s)        the view whose camera the lane's path starts from
//   root(s), depth() of the lane's scene and path
//   coords(v)        the two coordinates of vertex v
//   emission()       F so far
//   keep(F)          called while the path goes on: what emission() returns next
//   finish(F, status)  the path has ended
//   batch_done()     all lanes call after a shading batch
//   kFusedMirror     see phong_frame
// Sources keep F out of the traversal's registers where they have memory for it:
// it is almost always 0.
constexpr int kRefill = 4;  // refill a warp once this many lanes are idle
constexpr int kShadeBatch = 16;
enum PathState : uint32_t { kIdle = 0, kTraverse = 1, kWaitShade = 2 };

template <int kCheck, class Source>
__device__ __forceinline__ void trace_paths(const SceneView& s, Source& src, unsigned& status) {
    constexpr unsigned kAll = 0xffffffffu;
    Work wk;
    Trav r{};
    int stack[kStackSize];
    uint32_t state = kIdle;
    int v = 0, leaf = kSentinel;
    float3 T = f3(1.f, 1.f, 1.f);
    // One node visit of a lane that has an inner node; a leaf it comes to is
    // postponed if it holds none yet.
    auto visit = [&](bool on) {
        if (on && r.ref >= 0) {
            if (!trav_node<kCheck, false>(s, r, stack, status, wk)) {
                r.best = -1;
                r.ref = leaf = kSentinel;
            } else if (leaf == kSentinel && r.ref < 0 && r.ref != kSentinel) {
                leaf = r.ref;
                r.ref = r.sp > 0 ? stack[--r.sp] : kSentinel;
            }
        }
    };
    while (true) {
        // shade the waiting lanes as a batch
        const unsigned waiting = __ballot_sync(kAll, state == kWaitShade);
        const unsigned tracing = __ballot_sync(kAll, state == kTraverse);
        if (waiting && (__popc(waiting) >= kShadeBatch || __popc(waiting) >= __popc(tracing))) {
            if (state == kWaitShade) {
                bool live = false;
                float3 F = src.emission();
                if (r.best >= 0) {
                    const int depth = src.depth();
                    const float2 uv = v < depth ? src.coords(v) : make_float2(0.f, 0.f);
                    float3 o = r.o, d = r.d;
                    live = shade_vertex<Source::kFusedMirror>(s, r.best, r.tb, v, depth, uv.x, uv.y, o, d, T, F);
                    if (live) {
                        ++v;
                        trav_begin_at(r, o, d, src.root(s));
                        state = kTraverse;
                        src.keep(F);
                    }
                }
                if (!live) {
                    src.finish(F, status);
                    state = kIdle;
                }
            }
            src.batch_done();
        }
        // take new paths for idle lanes
        const unsigned idle = __ballot_sync(kAll, state == kIdle);
        if (!src.drained && idle && (__popc(idle) >= kRefill || idle == kAll)) {
            float y0, y1;
            if (src.take(idle, state == kIdle, y0, y1)) {
                float3 o, d;
                camera_ray(src.camera(s), y0, y1, o, d);
                T = f3(1.f, 1.f, 1.f);
                v = 0;
                const int root = src.root(s);
                trav_begin_at(r, o, d, root);
                state = root != kSentinel ? kTraverse : kWaitShade;  // empty scene: a miss
            }
        }
        if (!__any_sync(kAll, state != kIdle)) {
            if (src.drained) break;
            continue;
        }
        // one speculative while-while traversal round
        const bool trav = state == kTraverse;
        if (trav && leaf == kSentinel && r.ref < 0 && r.ref != kSentinel) {
            leaf = r.ref;
            r.ref = r.sp > 0 ? stack[--r.sp] : kSentinel;
        }
        const unsigned tracing_now = __ballot_sync(kAll, trav);
        if (__any_sync(kAll, trav && leaf == kSentinel && r.ref >= 0)) {
            do {  // two visits per vote: half the votes, and a lane that reaches its leaf goes on speculatively
                visit(trav);
                visit(trav);
            } while (!search_done(__ballot_sync(kAll, trav && leaf == kSentinel && r.ref >= 0), tracing_now));
            if (trav && over_budget<kCheck>(s, r, status)) {
                r.best = -1;
                r.ref = leaf = kSentinel;
            }
        }
        if (trav) {
            if (leaf != kSentinel) {
                trav_test_leaf<false>(s, r, leaf, wk);
                leaf = kSentinel;
            }
            if (r.ref == kSentinel) state = kWaitShade;
        }
    }
}

// ------------------------------------------------------------------ one step of Alg. 2
// Load chain i's coordinates (pair layout) into shared memory y[d * B].
__device__ __forceinline__ void load_coords(const ChainView& c, uint64_t i, float* y, uint32_t B) {
    const float2* x2 = reinterpret_cast<const float2*>(c.x);
    for (int k = 0; 2 * k < (int)c.dim; ++k) {
        const float2 v = x2[(uint64_t)k * c.n + i];
        y[2 * k * B] = v.x;
        y[(2 * k + 1) * B] = v.y;
    }
}

// Alg. 2: holding time t1 ~ Exp(1); killing time t2 ~ Exp(k), k = c~ u / p.  True:
// the local branch; dt gets the time the state is held for.
__device__ __forceinline__ bool restore_clocks_at(const ChainView& c, float E1, float E2, float p, float u,
                                                  float& dt) {
    const float t2 = p > 0.0f ? E2 * p / (c.c_tilde * u) : 0.0f;
    const bool local = E1 < t2;  // a tie goes to the killing branch
    dt = local ? E1 : t2;
    if (c.flags & JR_FLAG_RAO_BLACKWELL) dt = p > 0.0f ? p / (p + c.c_tilde * u) : 0.0f;
    return local;
}
__device__ __forceinline__ bool restore_clocks(const ChainView& c, const uint4& r0, float p, float u, float& dt) {
    return restore_clocks_at(c, -logf(1.0f - u01(r0.x)), -logf(1.0f - u01(r0.y)), p, u, dt);
}

// Candidate y of step `step` (cand[d * B]): a Gaussian small step from cur
// (local) or a fresh draw from mu.
__device__ __forceinline__ void propose(const ChainView& c, uint32_t chain, uint64_t step, bool local,
                                        const float* cur, float* cand, uint32_t B) {
    const int D = (int)c.dim;
    const float sigma = c.sigma;
    for (int b = 0; 4 * b < D; ++b) {
        const uint4 r = draw(c.seed, kTagStep, (uint32_t)(b + 1), chain, step);
        const int d0 = 4 * b;
        if (local) {
            float sn, cs;
            float R = sqrtf(-2.0f * logf(1.0f - u01(r.x)));
            sincospif(2.0f * u01(r.y), &sn, &cs);
            cand[d0 * B] = wrap01(cur[d0 * B] + sigma * R * cs);
            cand[(d0 + 1) * B] = wrap01(cur[(d0 + 1) * B] + sigma * R * sn);
            if (d0 + 2 < D) {
                R = sqrtf(-2.0f * logf(1.0f - u01(r.z)));
                sincospif(2.0f * u01(r.w), &sn, &cs);
                cand[(d0 + 2) * B] = wrap01(cur[(d0 + 2) * B] + sigma * R * cs);
                cand[(d0 + 3) * B] = wrap01(cur[(d0 + 3) * B] + sigma * R * sn);
            }
        } else {
            cand[d0 * B] = u01(r.x);
            cand[(d0 + 1) * B] = u01(r.y);
            if (d0 + 2 < D) {
                cand[(d0 + 2) * B] = u01(r.z);
                cand[(d0 + 3) * B] = u01(r.w);
            }
        }
    }
}

// A chain on its way through a window.  org: where the state's coordinates are:
// 0 in c.x, q > 0: the regeneration of the window's step q - 1.
struct Walk {
    float Fr, Fg, Fb, p, u;
    uint32_t k, org;
    __device__ __forceinline__ void load(const ChainView& c, uint64_t i) {
        Fr = c.fpu[0 * c.n + i];
        Fg = c.fpu[1 * c.n + i];
        Fb = c.fpu[2 * c.n + i];
        p = c.fpu[3 * c.n + i];
        u = c.fpu[4 * c.n + i];
    }
    __device__ __forceinline__ void store(const ChainView& c, uint64_t i) const {
        c.fpu[0 * c.n + i] = Fr;
        c.fpu[1 * c.n + i] = Fg;
        c.fpu[2 * c.n + i] = Fb;
        c.fpu[3 * c.n + i] = p;
        c.fpu[4 * c.n + i] = u;
    }
    // Regenerate at step k: f = the candidate's (F, status).
    __device__ __forceinline__ void regenerate(const float4 f, unsigned& status) {
        status |= __float_as_uint(f.w);
        const float3 F = finite_or_zero(f3(f.x, f.y, f.z), status);
        Fr = F.x;
        Fg = F.y;
        Fb = F.z;
        p = lum(F);
        u = 1.0f;
        org = ++k;
    }
};

__device__ __forceinline__ void splat_state(const ChainView& c, const Walk& w, float x0, float x1, float dt) {
    if (!(dt > 0.0f && w.p > 0.0f)) return;
    const uint32_t px = min((uint32_t)((double)x0 * (double)c.width), c.width - 1);
    const uint32_t py = min((uint32_t)((double)x1 * (double)c.height), c.height - 1);
    const float WH = (float)c.width * (float)c.height;
    const float wgt = c.c_tilde * dt * WH / w.p;
    atomicAdd(c.fb + (py * c.width + px), make_float4(wgt * w.Fr, wgt * w.Fg, wgt * w.Fb, dt));
}

// The coordinates of the regeneration of step `step` into chain i's state.
__device__ __forceinline__ void store_regeneration(const ChainView& c, uint64_t i, uint64_t step) {
    float2* x2 = reinterpret_cast<float2*>(c.x);
    for (int b = 0; 4 * b < (int)c.dim; ++b) {
        const uint4 r = draw(c.seed, kTagStep, (uint32_t)(b + 1), c.chain_offset + (uint32_t)i, step);
        x2[(uint64_t)(2 * b) * c.n + i] = make_float2(u01(r.x), u01(r.y));
        if (4 * b + 2 < (int)c.dim) x2[(uint64_t)(2 * b + 1) * c.n + i] = make_float2(u01(r.z), u01(r.w));
    }
}

// ------------------------------------------------------------------ a whole warp on one path
// Closest hit of the ray (o, d) over all n triangle records, for the whole
// warp (every lane calls with the same ray).  Returns the record index or -1.
__device__ __forceinline__ int closest_hit_warp(const SceneView& s, float3 o, float3 d, float& t_out) {
    const int lane = threadIdx.x & 31;
    float tb = INFINITY;
    int best = -1, bid = INT32_MAX;
    for (uint32_t k = lane; k < s.n_tris; k += 32) {
        const TriRecord* tr = s.tris + k;
        const float4 q0 = __ldg(&tr->v0_id), q1 = __ldg(&tr->e1_mat), q2 = __ldg(&tr->e2);
        const float3 e1 = f3(q1.x, q1.y, q1.z), e2 = f3(q2.x, q2.y, q2.z);
        const float3 pv = cross(d, e2);
        const float det = dot(e1, pv);
        const float inv = 1.0f / det;
        const float3 tv = o - f3(q0.x, q0.y, q0.z);
        const float u = dot(tv, pv) * inv;
        const float3 qv = cross(tv, e1);
        const float v = dot(d, qv) * inv;
        const float t = dot(e2, qv) * inv;
        const int id = __float_as_int(q0.w);
        const bool hit = det != 0.0f && !(u < 0.0f || u > 1.0f) && !(v < 0.0f || u + v > 1.0f) && t > 0.0f &&
                         (t < tb || (t == tb && id < bid));
        tb = hit ? t : tb;
        best = hit ? (int)k : best;
        bid = hit ? id : bid;
    }
    // The warp's closest hit, ties to the smaller original index.  Every tb is
    // a hit distance t > 0 or +inf, and for such floats the bit patterns order
    // as the values do, so two warp-wide integer minima find it: the nearest
    // distance, then the smallest index among the lanes at that distance (the
    // indices are distinct); the lane holding it hands over its record.
    const unsigned tbits = __float_as_uint(tb);
    const unsigned tmin = __reduce_min_sync(0xffffffffu, tbits);
    if (tmin == __float_as_uint(INFINITY)) {  // no lane has a hit
        t_out = INFINITY;
        return -1;
    }
    const unsigned imin = __reduce_min_sync(0xffffffffu, tbits == tmin ? (unsigned)bid : 0xffffffffu);
    const int src = __ffs(__ballot_sync(0xffffffffu, tbits == tmin && (unsigned)bid == imin)) - 1;
    best = __shfl_sync(0xffffffffu, best, src);
    t_out = __uint_as_float(tmin);
    return best;
}

// The integrand F(y) for the warp's chain, y[d] in lane d (eval_path_w's steps).
__device__ __forceinline__ float3 eval_path_warp(const SceneView& s, int depth, float yd, unsigned& status) {
    float3 F = f3(0.f, 0.f, 0.f), T = f3(1.f, 1.f, 1.f);
    float3 o, d;
    camera_ray(s, __shfl_sync(0xffffffffu, yd, 0), __shfl_sync(0xffffffffu, yd, 1), o, d);
    for (int v = 0; v <= depth; ++v) {
        float t;
        const int k = closest_hit_warp(s, o, d, t);
        if (k < 0) break;
        const float u1 = __shfl_sync(0xffffffffu, yd, (2 + 2 * v) & 31);
        const float u2 = __shfl_sync(0xffffffffu, yd, (3 + 2 * v) & 31);
        if (!shade_vertex(s, k, t, v, depth, v < depth ? u1 : 0.0f, v < depth ? u2 : 0.0f, o, d, T, F)) break;
    }
    return finite_or_zero(F, status);
}

// ------------------------------------------------------------------ gradient
// dF/dx for the Langevin local dynamics (MALA), forward mode.  F depends on x
// continuously only through the directions (camera, scattered) and the modified
// Phong weights (Lambertian and dielectric weights are constant; hit points only
// select triangles), so a lane carries the Jacobians of the current direction,
// of the throughput and of F, 3 x D each: column c is d/dx_c.  A Lambertian
// bounce's direction depends only on its own two coordinates, so its Jacobian
// restarts there.  At a change of hit triangle, bounce type or Fresnel choice the
// result is the gradient of the piece the state lies in.
struct Jac3 {
    float c[3][kMaxDim];
};

// J_out = d(normalize(v))/dx from J_v (v unnormalised, n = v / |v|).
__device__ inline void jac_normalize(float3 n, float inv_len, const Jac3& Jv, Jac3& Jn, int D) {
    for (int k = 0; k < D; ++k) {
        const float dvx = Jv.c[0][k], dvy = Jv.c[1][k], dvz = Jv.c[2][k];
        const float proj = n.x * dvx + n.y * dvy + n.z * dvz;
        Jn.c[0][k] = (dvx - n.x * proj) * inv_len;
        Jn.c[1][k] = (dvy - n.y * proj) * inv_len;
        Jn.c[2][k] = (dvz - n.z * proj) * inv_len;
    }
}

// The scatter of `scatter` with the Jacobian of the outgoing direction (Jwi) and
// the weight's log-derivative contribution: dw[ch][k] = d(weight_ch)/dx_k.
// Jd: Jacobian of the incoming direction d; (u1, u2) are coordinates i1, i1+1.
__device__ inline bool scatter_grad(const Material& m, float3 d, float3 ng, float u1, float u2, int i1, const Jac3& Jd,
                                    float3& wi, float3& w, Jac3& Jwi, Jac3& Jw, int D) {
    for (int q = 0; q < 3; ++q)
        for (int k = 0; k < D; ++k) Jw.c[q][k] = 0.f;
    if (m.type == JR_MAT_DIELECTRIC) {
        float cos_i = -dot(d, ng);
        float eta_i = 1.0f, eta_t = m.ior;
        float3 nn = ng;
        if (cos_i < 0.0f) {
            cos_i = -cos_i;
            eta_i = m.ior;
            eta_t = 1.0f;
            nn = ng * -1.0f;
        }
        float cos_t;
        const float R = fresnel(cos_i, eta_i, eta_t, cos_t);
        const float e = eta_i / eta_t;
        const bool refl = u1 < R;
        if (refl) wi = d + nn * (2.0f * cos_i);
        else wi = d * e + nn * (e * cos_i - cos_t);
        for (int k = 0; k < D; ++k) {
            const float dci = -(nn.x * Jd.c[0][k] + nn.y * Jd.c[1][k] + nn.z * Jd.c[2][k]);
            if (refl) {
                Jwi.c[0][k] = Jd.c[0][k] + 2.0f * nn.x * dci;
                Jwi.c[1][k] = Jd.c[1][k] + 2.0f * nn.y * dci;
                Jwi.c[2][k] = Jd.c[2][k] + 2.0f * nn.z * dci;
            } else {
                const float dct = cos_t > 0.0f ? e * e * cos_i * dci / cos_t : 0.0f;
                const float g = e * dci - dct;
                Jwi.c[0][k] = e * Jd.c[0][k] + nn.x * g;
                Jwi.c[1][k] = e * Jd.c[1][k] + nn.y * g;
                Jwi.c[2][k] = e * Jd.c[2][k] + nn.z * g;
            }
        }
        w = f3(1.0f, 1.0f, 1.0f);
        return true;
    }
    const float3 ns = dot(d, ng) < 0.0f ? ng : ng * -1.0f;
    float3 t, b;
    for (int q = 0; q < 3; ++q)
        for (int k = 0; k < D; ++k) Jwi.c[q][k] = 0.f;
    if (m.type == JR_MAT_LAMBERT) {
        const float r = sqrtf(u1);
        float sn, cs;
        sincospif(2.0f * u2, &sn, &cs);
        const float lz = sqrtf(fmaxf(1.0f - u1, 0.0f));
        onb(ns, t, b);
        wi = t * (r * cs) + b * (r * sn) + ns * lz;
        // d/du1 and d/du2 only
        const float dr = r > 0.0f ? 0.5f / r : 0.0f, dlz = lz > 0.0f ? -0.5f / lz : 0.0f;
        const float tw = 2.0f * 3.14159265358979f;
        const float3 d1 = t * (dr * cs) + b * (dr * sn) + ns * dlz;
        const float3 d2 = t * (-r * sn * tw) + b * (r * cs * tw);
        Jwi.c[0][i1] = d1.x; Jwi.c[1][i1] = d1.y; Jwi.c[2][i1] = d1.z;
        Jwi.c[0][i1 + 1] = d2.x; Jwi.c[1][i1 + 1] = d2.y; Jwi.c[2][i1 + 1] = d2.z;
        w = m.albedo;
        return m.albedo.x > 0.0f || m.albedo.y > 0.0f || m.albedo.z > 0.0f;
    }
    // modified Phong: r = d - 2 (d.ns) ns, basis around r, lobe angle from u1, azimuth from u2
    const PhongFrame q = phong_frame(m, d, ns, u1, u2);
    const float3 r = q.r;
    const float cos_a = q.cos_a, sin_a = q.sin_a, sn = q.sn, cs = q.cs;
    t = q.t;
    b = q.b;
    wi = phong_direction(q);
    const float cos_i = dot_rn(wi, ns);
    if (cos_i <= 0.0f) return false;
    const float sign = copysignf(1.0f, r.z);
    const float a = -1.0f / (sign + r.z);  // the basis's a; its bb term is differentiated in the loop
    // d cos_a / d u1 and d sin_a / d u1
    const float dca = 1.0f - u1 > 0.0f ? -m.phong_inv_n1 * cos_a / (1.0f - u1) : 0.0f;
    const float dsa = sin_a > 0.0f ? -cos_a * dca / sin_a : 0.0f;
    const float tw = 2.0f * 3.14159265358979f;
    for (int k = 0; k < D; ++k) {
        const float ddx = Jd.c[0][k], ddy = Jd.c[1][k], ddz = Jd.c[2][k];
        const float dn = ns.x * ddx + ns.y * ddy + ns.z * ddz;
        const float drx = ddx - 2.0f * ns.x * dn, dry = ddy - 2.0f * ns.y * dn, drz = ddz - 2.0f * ns.z * dn;
        const float da = a * a * drz;
        const float dbb = r.y * a * drx + r.x * a * dry + r.x * r.y * da;
        const float dtx = sign * (2.0f * r.x * a * drx + r.x * r.x * da), dty = sign * dbb, dtz = -sign * drx;
        const float dbx = dbb, dby = 2.0f * r.y * a * dry + r.y * r.y * da, dbz = -dry;
        float gx = dtx * (sin_a * cs) + dbx * (sin_a * sn) + drx * cos_a;
        float gy = dty * (sin_a * cs) + dby * (sin_a * sn) + dry * cos_a;
        float gz = dtz * (sin_a * cs) + dbz * (sin_a * sn) + drz * cos_a;
        if (k == i1) {
            gx += t.x * (dsa * cs) + b.x * (dsa * sn) + r.x * dca;
            gy += t.y * (dsa * cs) + b.y * (dsa * sn) + r.y * dca;
            gz += t.z * (dsa * cs) + b.z * (dsa * sn) + r.z * dca;
        } else if (k == i1 + 1) {
            gx += sin_a * tw * (-t.x * sn + b.x * cs);
            gy += sin_a * tw * (-t.y * sn + b.y * cs);
            gz += sin_a * tw * (-t.z * sn + b.z * cs);
        }
        Jwi.c[0][k] = gx;
        Jwi.c[1][k] = gy;
        Jwi.c[2][k] = gz;
        const float dci = ns.x * gx + ns.y * gy + ns.z * gz;
        Jw.c[0][k] = m.albedo.x * m.phong_scale * dci;
        Jw.c[1][k] = m.albedo.y * m.phong_scale * dci;
        Jw.c[2][k] = m.albedo.z * m.phong_scale * dci;
    }
    w = phong_weight(m, cos_i);
    return true;
}

// F(y) and dF/dy (dF->c[ch][k]) for one lane (no warp cooperation: the
// megakernel's lanes call it together, each with its own state).
template <int kCheck, bool kCount>
__device__ inline float3 eval_path_grad(const SceneView& s, unsigned mask, bool want, int depth, const float* y,
                                        uint32_t ys, Jac3& JF, unsigned& status, Work& work) {
    const int D = 2 + 2 * depth;
    Jac3 Jd, JT, Jtmp, Jw;
    for (int q = 0; q < 3; ++q)
        for (int k = 0; k < D; ++k) {
            JF.c[q][k] = 0.f;
            JT.c[q][k] = 0.f;
            Jd.c[q][k] = 0.f;
        }
    float3 F = f3(0.f, 0.f, 0.f), T = f3(1.f, 1.f, 1.f);
    float3 o = f3(0.f, 0.f, 1.f), d = f3(0.f, 0.f, 1.f);
    if (want) {
        const float3 cf = f3(s.cam[3], s.cam[4], s.cam[5]);
        const float3 cr = f3(s.cam[6], s.cam[7], s.cam[8]);
        const float3 cu = f3(s.cam[9], s.cam[10], s.cam[11]);
        o = f3(s.cam[0], s.cam[1], s.cam[2]);
        const float3 c = cf + cr * (2.0f * y[0] - 1.0f) + cu * (1.0f - 2.0f * y[ys]);
        const float il = 1.0f / sqrtf(dot(c, c));
        d = c * il;
        Jtmp.c[0][0] = 2.0f * cr.x; Jtmp.c[1][0] = 2.0f * cr.y; Jtmp.c[2][0] = 2.0f * cr.z;
        Jtmp.c[0][1] = -2.0f * cu.x; Jtmp.c[1][1] = -2.0f * cu.y; Jtmp.c[2][1] = -2.0f * cu.z;
        for (int q = 0; q < 3; ++q)
            for (int k = 2; k < D; ++k) Jtmp.c[q][k] = 0.f;
        jac_normalize(d, il, Jtmp, Jd, D);
    }
    bool alive = want;
    for (int v = 0; v <= depth; ++v) {
        if (!__any_sync(mask, alive)) break;
        float t;
        const int k = closest_hit<kCheck, kCount>(s, mask, alive, o, d, t, status, work);
        if (!alive) continue;
        if (k < 0) {
            alive = false;
            continue;
        }
        const TriRecord* tr = s.tris + k;
        const float4 q1 = __ldg(&tr->e1_mat), q2 = __ldg(&tr->e2);
        const Material m = s.mats[__float_as_int(q1.w)];
        const float3 ng = normalize(cross(f3(q1.x, q1.y, q1.z), f3(q2.x, q2.y, q2.z)));
        const float3 p = o + d * t;
        if (m.emits && -dot(d, ng) > 0.0f) {
            F = F + mul(T, m.emission);
            for (int kk = 0; kk < D; ++kk) {
                JF.c[0][kk] += JT.c[0][kk] * m.emission.x;
                JF.c[1][kk] += JT.c[1][kk] * m.emission.y;
                JF.c[2][kk] += JT.c[2][kk] * m.emission.z;
            }
        }
        if (v == depth) {
            alive = false;
            continue;
        }
        float3 wi, w;
        const float u1 = y[(2 + 2 * v) * ys], u2 = y[(3 + 2 * v) * ys];
        if (!scatter_grad(m, d, ng, u1, u2, 2 + 2 * v, Jd, wi, w, Jtmp, Jw, D)) {
            alive = false;
            continue;
        }
        for (int kk = 0; kk < D; ++kk) {  // d(T w) = dT w + T dw
            JT.c[0][kk] = JT.c[0][kk] * w.x + T.x * Jw.c[0][kk];
            JT.c[1][kk] = JT.c[1][kk] * w.y + T.y * Jw.c[1][kk];
            JT.c[2][kk] = JT.c[2][kk] * w.z + T.z * Jw.c[2][kk];
        }
        T = mul(T, w);
        if (T.x == 0.0f && T.y == 0.0f && T.z == 0.0f) {
            alive = false;
            continue;
        }
        for (int q = 0; q < 3; ++q)
            for (int kk = 0; kk < D; ++kk) Jd.c[q][kk] = Jtmp.c[q][kk];
        const float3 off = dot(wi, ng) >= 0.0f ? ng : ng * -1.0f;
        const float mx = fmaxf(fmaxf(fabsf(p.x), fabsf(p.y)), fabsf(p.z));
        o = p + off * (1e-4f * (1.0f + mx));
        d = wi;
    }
    if (want) {
        if (!isfinite(F.x) || !isfinite(F.y) || !isfinite(F.z)) {
            status |= JR_STATUS_NONFINITE;
            F = f3(0.f, 0.f, 0.f);
        }
    }
    return F;
}

// The MALA drift m = clamp(sigma^2 / 2 grad log p, -2 sigma, 2 sigma) per
// coordinate from F and dF/dx (grad log p = grad lum(F) / lum(F); 0 where p = 0
// or the gradient is not finite).
__device__ inline float mala_drift(float3 F, const Jac3& JF, int k, float sigma) {
    const float p = lum(F);
    if (!(p > 0.0f)) return 0.0f;
    const float g = (0.2126f * JF.c[0][k] + 0.7152f * JF.c[1][k] + 0.0722f * JF.c[2][k]) / p;
    if (!isfinite(g)) return 0.0f;
    return fminf(fmaxf(0.5f * sigma * sigma * g, -2.0f * sigma), 2.0f * sigma);
}

__device__ __forceinline__ float torus_delta(float to, float from) {
    const float d = to - from;
    return d - floorf(d + 0.5f);
}

// log q(b | a) up to the constant, from a's drift ma (all [D] with stride B).
__device__ __forceinline__ float mala_log_q(const float* b, const float* a, const float* ma, int D, uint32_t B,
                                            float sigma) {
    float s = 0.f;
    for (int d = 0; d < D; ++d) {
        const float e = torus_delta(b[d * B], a[d * B]) - ma[d * B];
        s += e * e;
    }
    return -s / (2.0f * sigma * sigma);
}

// The MALA proposal y = x + m(x) + sigma N of step `step` (cand[d * B]).
__device__ __forceinline__ void mala_propose(const ChainView& c, uint32_t chain, uint64_t step, const float* cur,
                                             const float* mc, float* cand, uint32_t B) {
    const int D = (int)c.dim;
    for (int b = 0; 4 * b < D; ++b) {
        const uint4 r = draw(c.seed, kTagStep, (uint32_t)(b + 1), chain, step);
        const int d0 = 4 * b;
        float sn, cs;
        float R = sqrtf(-2.0f * logf(1.0f - u01(r.x)));
        sincospif(2.0f * u01(r.y), &sn, &cs);
        cand[d0 * B] = wrap01(cur[d0 * B] + mc[d0 * B] + c.sigma * R * cs);
        cand[(d0 + 1) * B] = wrap01(cur[(d0 + 1) * B] + mc[(d0 + 1) * B] + c.sigma * R * sn);
        if (d0 + 2 < D) {
            R = sqrtf(-2.0f * logf(1.0f - u01(r.z)));
            sincospif(2.0f * u01(r.w), &sn, &cs);
            cand[(d0 + 2) * B] = wrap01(cur[(d0 + 2) * B] + mc[(d0 + 2) * B] + c.sigma * R * cs);
            cand[(d0 + 3) * B] = wrap01(cur[(d0 + 3) * B] + mc[(d0 + 3) * B] + c.sigma * R * sn);
        }
    }
}

// Its acceptance, U_a < min(1, p(y) q(x|y) / (p(x) q(y|x))), 1 if p(x) = 0.
__device__ __forceinline__ bool mala_accept(const ChainView& c, float Ua, float p, float py, const float* cur,
                                            const float* mc, const float* cand, const float* my, uint32_t B) {
    if (!(p > 0.0f)) return true;
    if (!(py > 0.0f)) return false;
    const int D = (int)c.dim;
    const float la = logf(py) - logf(p) + mala_log_q(cur, cand, my, D, B, c.sigma) -
                     mala_log_q(cand, cur, mc, D, B, c.sigma);
    return Ua > 0.0f ? logf(Ua) < la : true;
}

__device__ __forceinline__ void flush_status(unsigned status, unsigned int* word) {
    if (status) atomicOr(word, status);
}

// Sum of a double over the 32 lanes of a warp (all lanes call; every lane gets the sum).
__device__ __forceinline__ double warp_sum(double v) {
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) v += __shfl_xor_sync(0xffffffffu, v, o);
    return v;
}

}  // namespace
}  // namespace jr
