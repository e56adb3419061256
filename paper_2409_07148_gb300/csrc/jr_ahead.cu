// Look-ahead execution of Jump Restore with uniform regeneration (sm_103a).
//
// A regeneration of Alg. 2 (Section 7.2) draws its state from mu, so the candidate
// of step s of chain i depends on (i, s) only, not on the chain's state: its path
// can be traced before it is known whether step s regenerates at all.  In the
// stationary jump chain a share p_lambda / (p_lambda + c~) of the steps is local
// (Section 6.1), often around one percent, and all the others regenerate.  So an
// advance goes in windows of K steps:
//
//   1. ahead_path_kernel: F of the regeneration candidate of every (chain, step) of
//      the window, n K independent paths in one persistent launch (trace_paths).
//      The coordinates are drawn where they are used; 16 bytes per path go out.
//   2. settle_kernel, one thread per chain: the window's steps in order.  A state
//      with p = 0 is killed at once (k = inf), so a dark step is one 16-byte read;
//      a lit state draws its clocks and is splatted.  A chain whose step turns out
//      local stops and joins a queue.
//   3. The tail: the queued chains, each carried to the window's end by one lane, with
//      the local moves' paths traced on the way.  It runs inside the next window's
//      path launch; the last window's is a launch of its own, or, with few chains queued,
//      jr_runs.cu's.  For few chains in scenes of at most kWarpChainMaxTris triangles
//      jr_runs.cu does 2 and 3.
//
// The wavefront (jr_wavefront.cu) has to end every step's path launch before the
// next step, so it pays a launch's tail per step (12 % of the warp slots at 2^20
// chains), and few chains leave the device idle whatever the step does.  Here a
// launch has K times the paths, and the state is read and written once per window.
// What it costs: a local step's regeneration candidate is traced for nothing.
// Measured (against the other modes): 400 steps of 256 chains in the
// 24-triangle box 1 024 -> 453 us, 32 steps of 10 007 chains on Cornell + spheres
// 1 578 -> 988 us, 16 steps of 2^20 11.23 -> 9.65 ms, 400 steps of 10 007 20.6 -> 4.2 ms;
// with the tail inside the next launch against after its own window, 64 steps of 2^20
// chains 38.4 -> 36.7 ms, on the slit caustic 20.7 -> 19.0 ms, 32 on the terrain 20.1
// -> 18.0 ms.
//
// MALA Restore chains (JR_FLAG_MALA without JR_FLAG_MH) go the same way: their
// regenerations need F only, which the megakernel gets from the gradient's
// evaluation.
//
// The draws, the arithmetic and the order of a chain's steps are the other modes',
// so the chains are the same, bit for bit.
#include <cuda_runtime.h>
#include <stdint.h>

#include <algorithm>

#include "../../include/jr.h"
#include "jr_device.cuh"
#include "jr_internal.h"

namespace jr {
namespace {

constexpr unsigned kFull = 0xffffffffu;

// The paths of one launch: the tail of a window (chains queued with a local step,
// each carried to the window's end by one lane), and the regeneration candidates of
// the next.  The two do not depend on one another, and a tail is a serial chain of
// local steps for its longest run: beside the next window's paths it costs their
// issue slots only.
//
// A lane's path belongs to chain i.  org = kRegen: the regeneration candidate of the
// new window's step k; next.F[k n + i] gets (F, status bits).  Otherwise: the local
// candidate of the tail window's step k, from the state at org (Walk); when it ends
// the lane takes the acceptance, and goes on through the window until the next local
// step (cont: its path is to be taken) or the window's end.
constexpr uint32_t kRegen = 0xffffffffu;
struct Window {
    uint64_t step0;
    uint32_t K;
    float4* F;  // [K][n]
};
// kTail = false: a launch without a tail (1 to 2 % faster without its code).
template <bool kTail>
struct MixedPaths {
    static constexpr bool kFusedMirror = true;
    const ChainView& c;
    Window next, tail;          // next.K = 0: no candidates; tail_count = 0: no tail
    uint32_t tail_count;
    int tail_lanes;             // lanes of a warp that take queued chains (few chains spread over all warps)
    const uint4* queue;
    unsigned int* ctl;
    unsigned int* counts;       // shared memory: J, local steps, accepted
    bool tails_done = false, regens_done = false, drained = false;
    uint32_t i = 0, k = 0, org = kRegen;
    bool cont = false;
    float3 F = f3(0.f, 0.f, 0.f);

    __device__ __forceinline__ bool regen() const { return !kTail || org == kRegen; }
    __device__ __forceinline__ uint64_t step() const { return (regen() ? next.step0 : tail.step0) + k; }
    __device__ __forceinline__ uint4 block(uint32_t b, uint64_t st) const {
        return draw(c.seed, kTagStep, b + 1u, c.chain_offset + i, st);
    }
    __device__ __forceinline__ static float2 half_of(const uint4& r, uint32_t pair) {
        return pair & 1 ? make_float2(u01(r.z), u01(r.w)) : make_float2(u01(r.x), u01(r.y));
    }
    // Coordinate pair `pair` of the state at origin o, and of the lane's candidate.
    __device__ __forceinline__ float2 state_pair(uint32_t o, uint32_t pair) const {
        if (o == 0) return reinterpret_cast<const float2*>(c.x)[(uint64_t)pair * c.n + i];
        return half_of(block(pair >> 1, tail.step0 + o - 1), pair);
    }
    __device__ __forceinline__ float2 cand_pair(uint32_t pair) const {
        const float2 z = half_of(block(pair >> 1, step()), pair);
        if (regen()) return z;
        const float2 x = state_pair(org, pair);
        float sn, cs;
        const float R = sqrtf(-2.0f * logf(1.0f - z.x));
        sincospif(2.0f * z.y, &sn, &cs);
        return make_float2(wrap01(x.x + c.sigma * R * cs), wrap01(x.y + c.sigma * R * sn));
    }
    __device__ __forceinline__ bool take(unsigned idle, bool mine, float& y0, float& y1) {
        const int lane = threadIdx.x & 31;
        const unsigned lt = (1u << lane) - 1u;
        bool got = kTail && mine && cont;
        cont = false;
        if (kTail && !tails_done) {
            const unsigned want = __ballot_sync(kFull, mine && !got && lane < tail_lanes);
            if (want) {
                unsigned base = 0;
                if (lane == 0) base = atomicAdd(ctl + kCtlTail, (unsigned)__popc(want));
                base = __shfl_sync(kFull, base, 0);
                tails_done = base + (unsigned)__popc(want) >= tail_count;
                const unsigned q = base + __popc(want & lt);
                if (((want >> lane) & 1u) && q < tail_count) {
                    const uint4 e = queue[q];
                    i = e.x;
                    k = e.y;
                    org = e.z;
                    got = true;
                }
            }
        }
        if (!regens_done) {
            const unsigned want = __ballot_sync(kFull, mine && !got);
            if (want) {
                const uint32_t n = (uint32_t)c.n, count = n * next.K;
                unsigned base = 0;
                if (lane == 0) base = atomicAdd(ctl + kCtlPaths, (unsigned)__popc(want));
                base = __shfl_sync(kFull, base, 0);
                regens_done = base + (unsigned)__popc(want) >= count;
                const unsigned q = base + __popc(want & lt);
                if (((want >> lane) & 1u) && q < count) {
                    k = q / n;
                    i = q - k * n;
                    org = kRegen;
                    got = true;
                }
            }
        }
        drained = tails_done && regens_done;
        if (!got) return false;
        F = f3(0.f, 0.f, 0.f);
        const float2 y = cand_pair(0);
        y0 = y.x;
        y1 = y.y;
        return true;
    }
    __device__ __forceinline__ const SceneView& camera(const SceneView& s) const { return s; }
    __device__ __forceinline__ int root(const SceneView& s) const { return s.root; }
    __device__ __forceinline__ int depth() const { return (int)c.depth; }
    __device__ __forceinline__ float2 coords(int v) const { return cand_pair(1u + (uint32_t)v); }
    __device__ __forceinline__ float3 emission() const { return F; }
    __device__ __forceinline__ void keep(float3 f) { F = f; }
    __device__ __forceinline__ void finish(float3 f, unsigned& status) {
        if (regen()) {  // the status belongs to the path: it counts only if the chain takes it
            __stcs(next.F + (uint64_t)k * c.n + i, make_float4(f.x, f.y, f.z, __uint_as_float(status)));
        } else {
            local_step_done(f, status);
            flush_status(status, c.status);
        }
        status = 0;
    }
    __device__ __forceinline__ void local_step_done(float3 f, unsigned& status) {
        Walk w;
        w.load(c, i);
        w.k = k;
        w.org = org;
        f = finite_or_zero(f, status);
        const float py = lum(f);
        const bool accept = u01(draw(c.seed, kTagStep, 0, c.chain_offset + i, step()).z) * w.p < py;
        atomicAdd(counts + 1, 1u);
        if (accept) {
            atomicAdd(counts + 2, 1u);
            for (uint32_t q = 0; 2 * q < c.dim; ++q)
                reinterpret_cast<float2*>(c.x)[(uint64_t)q * c.n + i] = cand_pair(q);
            w.Fr = f.x;
            w.Fg = f.y;
            w.Fb = f.z;
            w.p = py;
            w.u = 1.0f;
            w.org = 0;
        }
        ++w.k;
        uint32_t nJ = 0;
        while (w.k < tail.K && !cont) {
            if (w.p > 0.0f) {
                float dt;
                cont = restore_clocks(c, draw(c.seed, kTagStep, 0, c.chain_offset + i, tail.step0 + w.k), w.p, w.u, dt);
                const float2 x = state_pair(w.org, 0);
                splat_state(c, w, x.x, x.y, dt);
            }
            if (!cont) {
                nJ++;
                w.regenerate(__ldcs(tail.F + (uint64_t)w.k * c.n + i), status);
            }
        }
        if (nJ) atomicAdd(counts, nJ);
        w.store(c, i);
        if (!cont && w.org) store_regeneration(c, i, tail.step0 + w.org - 1);
        k = w.k;
        org = w.org;
    }
    __device__ __forceinline__ void batch_done() {
        if (kTail && __any_sync(kFull, cont)) drained = false;
    }
};

template <int kCheck, bool kTail>
__global__ void __launch_bounds__(128, 7) ahead_path_kernel(SceneView s, ChainView c, Window next, Window tail,
                                                            const uint4* queue, unsigned int* ctl) {
    __shared__ unsigned int counts[3];
    if (threadIdx.x < 3) counts[threadIdx.x] = 0;
    __syncthreads();
    const uint32_t tails = kTail ? ctl[kCtlQueue] : 0u;
    const uint32_t warps = gridDim.x * (blockDim.x >> 5);
    MixedPaths<kTail> src{c, next, tail, tails, (int)((tails + warps - 1) / warps), queue, ctl, counts};
    src.tails_done = tails == 0;
    src.regens_done = next.K == 0;
    src.drained = src.tails_done && src.regens_done;
    unsigned status = 0;
    trace_paths<kCheck>(s, src, status);
    if (!kTail) return;
    __syncthreads();
    if (threadIdx.x < 3 && counts[threadIdx.x])
        atomicAdd(c.counters + threadIdx.x, (unsigned long long)counts[threadIdx.x]);
}

// Bound by reading the window's F (16 bytes per step and chain, four steps in
// flight); the lit states' clocks are rare.  kMala: a chain whose window ends lit
// also joins the queue, at step K, for its state's drift.
template <bool kMala>
__global__ void __launch_bounds__(128) settle_kernel(ChainView c, uint64_t step0, uint32_t K, const float4* Fw,
                                                     uint4* queue, unsigned int* ctl) {
    const uint64_t i = blockIdx.x * (uint64_t)blockDim.x + threadIdx.x;
    const bool valid = i < c.n;
    uint32_t nJ = 0;
    unsigned status = 0;
    bool local = false;
    Walk w;
    w.k = w.org = 0;
    w.p = 0.f;
    if (valid) {
        const uint32_t chain = c.chain_offset + (uint32_t)i;
        w.load(c, i);
        const float4* f = Fw + i;
        float4 next[4];
#pragma unroll
        for (int q = 0; q < 4; ++q) next[q] = q < (int)K ? __ldcs(f + (uint64_t)q * c.n) : make_float4(0.f, 0.f, 0.f, 0.f);
        for (uint32_t k0 = 0; k0 < K && !local; k0 += 4) {
#pragma unroll
            for (int q = 0; q < 4; ++q) {
                const uint32_t k = k0 + q;
                if (k >= K || local) break;
                if (w.p > 0.0f) {
                    float dt;
                    local = restore_clocks(c, draw(c.seed, kTagStep, 0, chain, step0 + k), w.p, w.u, dt);
                    float2 x;
                    if (w.org == 0) {
                        x = reinterpret_cast<const float2*>(c.x)[i];
                    } else {
                        const uint4 r = draw(c.seed, kTagStep, 1, chain, step0 + w.org - 1);
                        x = make_float2(u01(r.x), u01(r.y));
                    }
                    splat_state(c, w, x.x, x.y, dt);
                }
                if (!local) {
                    nJ++;
                    w.regenerate(next[q], status);
                    next[q] = k + 4 < K ? __ldcs(f + (uint64_t)(k + 4) * c.n) : make_float4(0.f, 0.f, 0.f, 0.f);
                }
            }
        }
        w.store(c, i);
        if (kMala && !local && w.p > 0.0f) local = true;
        if (!local && w.org) store_regeneration(c, i, step0 + w.org - 1);
        if (kMala && !local)  // the drift is 0 where p = 0
            for (uint32_t d = 0; d < c.dim; ++d) c.drift[d * c.n + i] = 0.0f;
    }
    // one queue atomic per warp
    const unsigned m = __ballot_sync(kFull, local);
    if (m) {
        const int lane = threadIdx.x & 31;
        unsigned base = 0;
        if (lane == 0) base = atomicAdd(ctl + kCtlQueue, (unsigned)__popc(m));
        base = __shfl_sync(kFull, base, 0);
        if (local) queue[base + __popc(m & ((1u << lane) - 1u))] = make_uint4((uint32_t)i, w.k, w.org, 0u);
    }
    nJ = __reduce_add_sync(kFull, nJ);
    status = __reduce_or_sync(kFull, status);
    if ((threadIdx.x & 31) == 0) {
        if (nJ) atomicAdd(c.counters + 0, (unsigned long long)nJ);
        flush_status(status, c.status);
    }
}

// The tail by itself: the queued chains to the window's end, lane = chain, one-warp
// blocks, chains fetched as lanes become free (drain_kernel's scheme: a local step
// waits for no other chain but the few in its warp).  For an advance's last window,
// which has no next one to hide in: there the longest run of local steps counts, and
// this kernel takes a step in less time than trace_paths, whose lanes wait for
// shading batches and refills (10 007 chains, 32 steps of Cornell + spheres: 596
// against 680 us).
template <int kCheck>
__global__ void __launch_bounds__(32, 16) tail_kernel(SceneView s, ChainView c, uint64_t step0, uint32_t K,
                                                      const float4* Fw, const uint4* queue, unsigned int* ctl,
                                                      uint32_t few) {
    extern __shared__ float sh[];
    constexpr uint32_t B = 32;
    const int lane = threadIdx.x;
    const unsigned count = ctl[kCtlQueue];
    if (count <= few) return;
    // Few chains spread over all warps: the first lanes of each take part.
    const unsigned lanes = (count + gridDim.x - 1) / gridDim.x;
    float* cur = sh + lane;
    float* cand = sh + (size_t)c.dim * B + lane;
    uint32_t nJ = 0, nL = 0, nA = 0;
    unsigned status = 0;
    Work work;
    bool live = false, drained = (unsigned)lane >= lanes;
    uint64_t i = 0;
    uint32_t chain = 0;
    Walk w;
    w.k = w.org = 0;
    while (true) {
        if (__any_sync(kFull, !live && !drained)) {
            const unsigned want = __ballot_sync(kFull, !live && !drained);
            unsigned base = 0;
            if (lane == 0) base = atomicAdd(ctl + kCtlTail, (unsigned)__popc(want));
            base = __shfl_sync(kFull, base, 0);
            if (!live && !drained) {
                const unsigned q = base + __popc(want & ((1u << lane) - 1u));
                drained = q >= count;
                if (!drained) {
                    const uint4 e = queue[q];
                    i = e.x;
                    w.k = e.y;
                    w.org = e.z;
                    chain = c.chain_offset + (uint32_t)i;
                    w.load(c, i);
                    if (w.org) propose(c, chain, step0 + w.org - 1, false, cur, cur, B);
                    else load_coords(c, i, cur, B);
                    live = true;
                }
            }
        }
        if (!__any_sync(kFull, live)) break;
        if (live) propose(c, chain, step0 + w.k, true, cur, cand, B);
        const float3 Fy = eval_path_w<kCheck, false>(s, kFull, live, (int)c.depth, cand, B, nullptr, 0, status, work);
        if (live) {
            const float py = lum(Fy);
            const bool accept = u01(draw(c.seed, kTagStep, 0, chain, step0 + w.k).z) * w.p < py;
            nL++;
            nA += accept;
            if (accept) {
                float* t = cur;
                cur = cand;
                cand = t;
                w.Fr = Fy.x;
                w.Fg = Fy.y;
                w.Fb = Fy.z;
                w.p = py;
                w.u = 1.0f;
            }
            w.org = 0;  // the coordinates are in cur
            ++w.k;
            bool local = false;
            while (w.k < K && !local) {
                if (w.p > 0.0f) {
                    float dt;
                    if (w.org) {  // lit after a regeneration: its coordinates are needed now
                        propose(c, chain, step0 + w.org - 1, false, cur, cur, B);
                        w.org = 0;
                    }
                    local = restore_clocks(c, draw(c.seed, kTagStep, 0, chain, step0 + w.k), w.p, w.u, dt);
                    splat_state(c, w, cur[0], cur[B], dt);
                }
                if (!local) {
                    nJ++;
                    w.regenerate(__ldcs(Fw + (uint64_t)w.k * c.n + i), status);
                }
            }
            if (!local) {  // the window's end
                live = false;
                w.store(c, i);
                if (w.org) {
                    store_regeneration(c, i, step0 + w.org - 1);
                } else {
                    float2* x2 = reinterpret_cast<float2*>(c.x);
                    for (int k = 0; 2 * k < (int)c.dim; ++k)
                        x2[(uint64_t)k * c.n + i] = make_float2(cur[2 * k * B], cur[(2 * k + 1) * B]);
                }
            }
        }
    }
    nJ = __reduce_add_sync(kFull, nJ);
    nL = __reduce_add_sync(kFull, nL);
    nA = __reduce_add_sync(kFull, nA);
    status = __reduce_or_sync(kFull, status);
    if (lane == 0) {
        if (nJ) atomicAdd(c.counters + 0, (unsigned long long)nJ);
        if (nL) atomicAdd(c.counters + 1, (unsigned long long)nL);
        if (nA) atomicAdd(c.counters + 2, (unsigned long long)nA);
        flush_status(status, c.status);
    }
}

// The tail with Langevin local moves (MALA Restore; the kernel of chain_steps_mala's
// steps).  Only states that a local move starts from or is accepted to, and those a
// window ends in, need the drift, and so the gradient of their path: a lane's round
// evaluates either the candidate's (its F and drift) or, for a lit state that came
// from a regeneration, the state's own drift.
template <int kCheck>
__global__ void __launch_bounds__(32, 16) mala_tail_kernel(SceneView s, ChainView c, uint64_t step0, uint32_t K,
                                                           const float4* Fw, const uint4* queue, unsigned int* ctl,
                                                           uint32_t few) {
    extern __shared__ float sh[];  // [4][D][32]: x, y, m(x), m(y)
    constexpr uint32_t B = 32;
    const int lane = threadIdx.x, D = (int)c.dim;
    const unsigned count = ctl[kCtlQueue];
    if (count <= few) return;
    const unsigned lanes = (count + gridDim.x - 1) / gridDim.x;  // few chains spread over all warps
    float* cur = sh + lane;
    float* cand = sh + (size_t)D * B + lane;
    float* mc = sh + (size_t)2 * D * B + lane;
    float* my = sh + (size_t)3 * D * B + lane;
    uint32_t nJ = 0, nL = 0, nA = 0;
    unsigned status = 0;
    Work work;
    Jac3 JF;
    bool live = false, known = false, drained = (unsigned)lane >= lanes;  // known: mc is the state's drift
    uint64_t i = 0;
    uint32_t chain = 0;
    Walk w;
    w.k = w.org = 0;
    while (true) {
        if (__any_sync(kFull, !live && !drained)) {
            const unsigned want = __ballot_sync(kFull, !live && !drained);
            unsigned base = 0;
            if (lane == 0) base = atomicAdd(ctl + kCtlTail, (unsigned)__popc(want));
            base = __shfl_sync(kFull, base, 0);
            if (!live && !drained) {
                const unsigned q = base + __popc(want & ((1u << lane) - 1u));
                drained = q >= count;
                if (!drained) {
                    const uint4 e = queue[q];
                    i = e.x;
                    w.k = e.y;
                    w.org = e.z;
                    chain = c.chain_offset + (uint32_t)i;
                    w.load(c, i);
                    known = w.org == 0;
                    if (known) {
                        load_coords(c, i, cur, B);
                        for (int d = 0; d < D; ++d) mc[d * B] = c.drift[d * c.n + i];
                    } else {
                        propose(c, chain, step0 + w.org - 1, false, cur, cur, B);
                        w.org = 0;
                    }
                    live = true;
                }
            }
        }
        if (!__any_sync(kFull, live)) break;
        if (live && known) mala_propose(c, chain, step0 + w.k, cur, mc, cand, B);
        const float3 Fy = eval_path_grad<kCheck, false>(s, kFull, live, (int)c.depth, known ? cand : cur, B, JF, status,
                                                        work);
        if (live) {
            bool local = true;  // a local step is pending
            if (!known) {
                for (int d = 0; d < D; ++d) mc[d * B] = mala_drift(Fy, JF, d, c.sigma);
                known = true;
                local = w.k < K;
            } else {
                for (int d = 0; d < D; ++d) my[d * B] = mala_drift(Fy, JF, d, c.sigma);
                const float py = lum(Fy);
                const float Ua = u01(draw(c.seed, kTagStep, 0, chain, step0 + w.k).z);
                const bool accept = mala_accept(c, Ua, w.p, py, cur, mc, cand, my, B);
                nL++;
                nA += accept;
                if (accept) {
                    float* t = cur;
                    cur = cand;
                    cand = t;
                    t = mc;
                    mc = my;
                    my = t;
                    w.Fr = Fy.x;
                    w.Fg = Fy.y;
                    w.Fb = Fy.z;
                    w.p = py;
                    w.u = 1.0f;
                }
                ++w.k;
                local = false;
                while (w.k < K && !local) {
                    if (w.p > 0.0f) {
                        float dt;
                        if (w.org) {  // lit after a regeneration: its coordinates are needed now
                            propose(c, chain, step0 + w.org - 1, false, cur, cur, B);
                            w.org = 0;
                            known = false;
                        }
                        local = restore_clocks(c, draw(c.seed, kTagStep, 0, chain, step0 + w.k), w.p, w.u, dt);
                        splat_state(c, w, cur[0], cur[B], dt);
                    }
                    if (!local) {
                        nJ++;
                        w.regenerate(__ldcs(Fw + (uint64_t)w.k * c.n + i), status);
                    }
                }
                if (!local && w.org && w.p > 0.0f) {  // the window ends lit: one more round for the drift
                    propose(c, chain, step0 + w.org - 1, false, cur, cur, B);
                    w.org = 0;
                    known = false;
                    local = true;
                }
            }
            if (!local) {  // the window's end
                live = false;
                w.store(c, i);
                if (w.org) {  // dark
                    store_regeneration(c, i, step0 + w.org - 1);
                    for (int d = 0; d < D; ++d) c.drift[d * c.n + i] = 0.0f;
                } else {
                    float2* x2 = reinterpret_cast<float2*>(c.x);
                    for (int k = 0; 2 * k < D; ++k)
                        x2[(uint64_t)k * c.n + i] = make_float2(cur[2 * k * B], cur[(2 * k + 1) * B]);
                    for (int d = 0; d < D; ++d) c.drift[d * c.n + i] = mc[d * B];
                }
            }
        }
    }
    nJ = __reduce_add_sync(kFull, nJ);
    nL = __reduce_add_sync(kFull, nL);
    nA = __reduce_add_sync(kFull, nA);
    status = __reduce_or_sync(kFull, status);
    if (lane == 0) {
        if (nJ) atomicAdd(c.counters + 0, (unsigned long long)nJ);
        if (nL) atomicAdd(c.counters + 1, (unsigned long long)nL);
        if (nA) atomicAdd(c.counters + 2, (unsigned long long)nA);
        flush_status(status, c.status);
    }
}

inline unsigned grid_for(uint64_t n, unsigned b) { return (unsigned)((n + b - 1) / b); }

// Resident one-warp or 128-thread blocks of a kernel on the current device.
template <class K>
cudaError_t resident(K kernel, int threads, size_t shm, long long* blocks) {
    int dev = 0, sms = 0, per_sm = 0;
    cudaError_t e;
    if ((e = cudaGetDevice(&dev)) != cudaSuccess ||
        (e = cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, dev)) != cudaSuccess ||
        (e = cudaOccupancyMaxActiveBlocksPerMultiprocessor(&per_sm, kernel, threads, shm)) != cudaSuccess)
        return e;
    *blocks = (long long)sms * (per_sm > 0 ? per_sm : 1);
    return cudaSuccess;
}

}  // namespace

cudaError_t launch_ahead(const SceneView& s, const ChainView& c, const AheadView& a, uint64_t step_begin,
                         uint32_t n_steps, bool warp_tail, cudaStream_t st, KernelTimer* tm) {
    if (c.n == 0 || n_steps == 0) return cudaSuccess;
    cudaError_t e = cudaSuccess;
    with_checks(trav_checks(s), [&](auto kc) {
        constexpr int kCheck = decltype(kc)::value;
        const bool mala = (c.flags & JR_FLAG_MALA) != 0;
        const auto paths = ahead_path_kernel<kCheck, false>, mixed = ahead_path_kernel<kCheck, true>;
        const auto settle = mala ? settle_kernel<true> : settle_kernel<false>;
        const auto alone = mala ? mala_tail_kernel<kCheck> : tail_kernel<kCheck>;
        const size_t shm = sizeof(float) * (mala ? 4 : 2) * c.dim * 32;  // <= 16 KB
        long long path_blocks = 0, mixed_blocks = 0, tail_blocks = 0;
        if ((e = resident(paths, 128, 0, &path_blocks)) != cudaSuccess ||
            (e = resident(mixed, 128, 0, &mixed_blocks)) != cudaSuccess)
            return;
        if (!warp_tail && (e = resident(alone, 32, shm, &tail_blocks)) != cudaSuccess) return;
        auto mark = [&](int kind) {
            if (tm && e == cudaSuccess) e = tm->mark(kind, st);
        };
        mark(-1);
        Window tail{0, 0, nullptr};  // the window whose tail is still to run
        for (uint32_t done = 0, k = 0; done < n_steps && e == cudaSuccess; ++k) {
            const uint32_t K = std::min(a.window, n_steps - done);
            const Window w{step_begin + done, K, a.F + (a.buffers > 1 ? k & 1 : 0) * (uint64_t)a.window * c.n};
            done += K;
            if ((e = cudaMemsetAsync(a.ctl + kCtlPaths, 0, sizeof(unsigned int), st)) != cudaSuccess) return;
            if (tail.K)
                mixed<<<(unsigned)mixed_blocks, 128, 0, st>>>(s, c, w, tail, a.queue, a.ctl);
            else
                paths<<<(unsigned)std::min<uint64_t>((uint64_t)path_blocks, grid_for(c.n * K, 128)), 128, 0, st>>>(
                    s, c, w, tail, a.queue, a.ctl);
            mark(KernelTimer::kPath);
            tail.K = 0;
            if (warp_tail) {
                if (e == cudaSuccess) e = launch_runs_settle(s, c, w.step0, K, w.F, st);
            } else {
                if (e == cudaSuccess)
                    e = cudaMemsetAsync(a.ctl + kCtlQueue, 0, sizeof(unsigned int) * 2, st);  // and kCtlTail
                settle<<<grid_for(c.n, 128), 128, 0, st>>>(c, w.step0, K, w.F, a.queue, a.ctl);
                if (mala || a.buffers < 2 || done == n_steps) {
                    uint32_t few = 0;  // queues this short are launch_runs_tail's
                    if (!mala && e == cudaSuccess)
                        e = launch_runs_tail(s, c, w.step0, K, w.F, a.queue, a.ctl, &few, st);
                    alone<<<(unsigned)std::min<uint64_t>((uint64_t)tail_blocks, c.n), 32, shm, st>>>(
                        s, c, w.step0, K, w.F, a.queue, a.ctl, few);
                } else {
                    tail = w;
                }
            }
            mark(KernelTimer::kStep);
            if (e == cudaSuccess) e = cudaGetLastError();
        }
    });
    return e;
}

}  // namespace jr
