// Runs of local steps of few chains (sm_103a): the tail of a look-ahead window, the
// tail of a drain, and whole windows in small scenes.
//
// A run of local steps is serial: a step's candidate starts from the state that the
// step before left.  But that state is one of two, known before the step's path is
// traced: the old state, or the candidate; and the draws depend on (chain, step) only.
// So a block takes kLevels steps at once (prefetching, Brockwell, JCGS 2006): its
// warps trace the candidates of all 2^kLevels - 1 outcomes of the steps before, in a
// heap (node j: the candidate of step s + floor(log2 j); node 2j: of the next step
// after j's rejection, 2j + 1: after its acceptance), and warp 0 then follows the
// outcomes that happen.  What it costs is paths that are not taken, on warps that
// would idle; what it needs is that few chains are left.  Same draws and arithmetic
// as the serial step, so the same chains.
//
// Warp 0 controls (the chain's state, clocks, splats, regenerations taken from the
// window); warps 1 .. 2^kLevels - 1 are the nodes.  Lane d holds coordinate d.  kBrute
// (scenes of at most kWarpChainMaxTris triangles): a node's warp traces the path
// together; otherwise its lane 0 traces it with the BVH.
#include <cuda_runtime.h>
#include <stdint.h>

#include <algorithm>

#include "../../include/jr.h"
#include "jr_device.cuh"
#include "jr_internal.h"

namespace jr {
namespace {

constexpr unsigned kFull = 0xffffffffu;

template <int kLevels>
struct RunSmem {
    static constexpr int kNodes = 1 << kLevels;
    float base[32];           // the state's coordinates
    float y[kNodes][32];      // the nodes' candidates
    float3 F[kNodes];
    unsigned status[kNodes];
    uint64_t step, end;       // the first step of the round, the step to stop at
    uint32_t chain;
    int go;                   // 0: the block is done
};

// Coordinate `lane` of a local move of step `step` from x.
__device__ __forceinline__ float move_lane(const ChainView& c, uint32_t chain, uint64_t step, float x) {
    const int lane = threadIdx.x & 31;
    const uint4 r = draw(c.seed, kTagStep, (uint32_t)(lane >> 2) + 1u, chain, step);
    const bool second = (lane & 2) != 0;
    float sn, cs;
    const float R = sqrtf(-2.0f * logf(1.0f - u01(second ? r.z : r.x)));
    sincospif(2.0f * u01(second ? r.w : r.y), &sn, &cs);
    return wrap01(x + c.sigma * R * ((lane & 1) ? sn : cs));
}
// Coordinate `lane` of the regeneration of step `step`.
__device__ __forceinline__ float regen_lane(const ChainView& c, uint32_t chain, uint64_t step) {
    const int lane = threadIdx.x & 31;
    const uint4 r = draw(c.seed, kTagStep, (uint32_t)(lane >> 2) + 1u, chain, step);
    return u01(lane & 2 ? ((lane & 1) ? r.w : r.z) : ((lane & 1) ? r.y : r.x));
}

// A node's warp: its candidate, and the candidate's F.
template <int kCheck, int kLevels, bool kBrute>
__device__ __forceinline__ void trace_node(const SceneView& s, const ChainView& c, RunSmem<kLevels>& sm) {
    const int j = (int)(threadIdx.x >> 5), lane = threadIdx.x & 31;
    const int level = 31 - __clz(j);
    if (sm.step + level >= sm.end) return;  // past the end: nobody asks
    const uint32_t chain = sm.chain;
    float y = sm.base[lane];
    if (lane < (int)c.dim) {
        for (int q = 0; q < level; ++q)  // the accepted moves on the way to the node
            if ((j >> (level - 1 - q)) & 1) y = move_lane(c, chain, sm.step + q, y);
        y = move_lane(c, chain, sm.step + level, y);
    }
    sm.y[j][lane] = y;
    unsigned status = 0;
    float3 F;
    if constexpr (kBrute) {
        F = eval_path_warp(s, (int)c.depth, y, status);
    } else {
        __syncwarp();
        if (lane == 0) {
            Work work;
            F = eval_path_w<kCheck, false>(s, 1u, true, (int)c.depth, sm.y[j], 1, nullptr, 0, status, work);
        }
    }
    if (lane == 0) {
        sm.F[j] = F;
        sm.status[j] = status;
    }
}

struct RunCounts {
    uint32_t nJ = 0, nL = 0, nA = 0;
    unsigned status = 0;
    __device__ __forceinline__ void flush(const ChainView& c) const {  // one lane
        if (nJ) atomicAdd(c.counters + 0, (unsigned long long)nJ);
        if (nL) atomicAdd(c.counters + 1, (unsigned long long)nL);
        if (nA) atomicAdd(c.counters + 2, (unsigned long long)nA);
        flush_status(status, c.status);
    }
};

// Warp 0 after the nodes: the round's steps in order, from step first = sm.step (a
// local one).  E1, E2, Ua: lane l holds those of step first + l.  Updates the state
// (w, xd) and *step to the next step to take; true: that step is local (its clocks
// are drawn and its splat is done).  False: the chain is at sm.end, or the clocks of
// step *step killed it (*killed; splat done).
template <int kLevels>
__device__ __forceinline__ bool follow(const ChainView& c, RunSmem<kLevels>& sm, Walk& w, float& xd, float E1, float E2,
                                       float Ua, uint64_t& step, bool& killed, RunCounts& n) {
    const int lane = threadIdx.x & 31;
    int j = 1;
    killed = false;
#pragma unroll
    for (int l = 0; l < kLevels; ++l) {
        n.status |= sm.status[j];  // eval's finite_or_zero has set its bit there
        const float3 F = sm.F[j];
        const float py = lum(F);
        const bool accept = __shfl_sync(kFull, Ua, l) * w.p < py;
        n.nL++;
        n.nA += accept;
        if (accept) {
            xd = sm.y[j][lane];
            w.Fr = F.x;
            w.Fg = F.y;
            w.Fb = F.z;
            w.p = py;
            w.u = 1.0f;
        }
        ++step;
        if (step == sm.end) return false;
        float dt;
        const bool local =
            restore_clocks_at(c, __shfl_sync(kFull, E1, l + 1), __shfl_sync(kFull, E2, l + 1), w.p, w.u, dt);
        const float x0 = __shfl_sync(kFull, xd, 0), x1 = __shfl_sync(kFull, xd, 1);
        if (lane == 0) splat_state(c, w, x0, x1, dt);
        if (!local) {
            killed = true;
            return false;
        }
        j = 2 * j + (accept ? 1 : 0);
    }
    return true;
}

// Warp 0: through the window's steps from w.k until the next local one (true; its
// splat is done) or the window's end.  org as in Walk; when it returns true, org = 0
// and xd are the state's coordinates.  skip_clocks: step w.k's clocks have killed
// the chain already.
__device__ __forceinline__ bool walk_window(const ChainView& c, uint64_t i, uint64_t step0, uint32_t K,
                                            const float4* Fw, Walk& w, float& xd, bool skip_clocks, RunCounts& n) {
    const int lane = threadIdx.x & 31;
    const uint32_t chain = c.chain_offset + (uint32_t)i;
    while (w.k < K) {
        if (!(w.p > 0.0f)) {  // regenerate up to the first lit candidate
            const uint32_t left = min(32u, K - w.k);
            float4 f = make_float4(0.f, 0.f, 0.f, 0.f);
            if (lane < (int)left) f = __ldcs(Fw + (uint64_t)(w.k + lane) * c.n + i);
            // lit, or not to be skipped: not finite, or with a status to report
            const bool stop = lum(f3(f.x, f.y, f.z)) > 0.0f || !isfinite(f.x) || !isfinite(f.y) || !isfinite(f.z) ||
                              __float_as_uint(f.w) != 0u;
            const unsigned m = __ballot_sync(kFull, stop);
            const uint32_t skip = m ? (uint32_t)__ffs(m) - 1u : left;  // dark ones before it
            n.nJ += skip;
            w.k += skip;
            if (skip) {  // the last skipped candidate is the state (p = 0)
                const int src = (int)skip - 1;
                w.Fr = __shfl_sync(kFull, f.x, src);
                w.Fg = __shfl_sync(kFull, f.y, src);
                w.Fb = __shfl_sync(kFull, f.z, src);
                w.p = lum(f3(w.Fr, w.Fg, w.Fb));
                w.u = 1.0f;
                w.org = w.k;
            }
            if (m) {
                const int src = (int)skip;
                const float4 g = make_float4(__shfl_sync(kFull, f.x, src), __shfl_sync(kFull, f.y, src),
                                             __shfl_sync(kFull, f.z, src), __shfl_sync(kFull, f.w, src));
                n.nJ++;
                w.regenerate(g, n.status);
            }
            skip_clocks = false;
            continue;
        }
        if (w.org) {
            xd = regen_lane(c, chain, step0 + w.org - 1);
            w.org = 0;
        }
        if (!skip_clocks) {
            float dt;
            const bool local = restore_clocks(c, draw(c.seed, kTagStep, 0, chain, step0 + w.k), w.p, w.u, dt);
            const float x0 = __shfl_sync(kFull, xd, 0), x1 = __shfl_sync(kFull, xd, 1);
            if (lane == 0) splat_state(c, w, x0, x1, dt);
            if (local) return true;
        }
        skip_clocks = false;
        n.nJ++;
        w.regenerate(__ldcs(Fw + (uint64_t)w.k * c.n + i), n.status);
    }
    return false;
}

// The round's draws for warp 0: lane l those of step sm.step + l.
template <int kLevels>
__device__ __forceinline__ void round_draws(const ChainView& c, const RunSmem<kLevels>& sm, float& E1, float& E2,
                                            float& Ua) {
    const int lane = threadIdx.x & 31;
    if (lane > kLevels) return;
    const uint4 r0 = draw(c.seed, kTagStep, 0, sm.chain, sm.step + lane);
    E1 = -logf(1.0f - u01(r0.x));
    E2 = -logf(1.0f - u01(r0.y));
    Ua = u01(r0.z);
}

// A window's steps.  queue = null: chain blockIdx.x from the window's start (every
// chain has its block); else the queued chains, if there are at most `most`, fetched
// by the blocks.
template <int kCheck, int kLevels, bool kBrute>
__global__ void __launch_bounds__(32 << kLevels, 16 >> kLevels) runs_window_kernel(
    SceneView s, ChainView c, uint64_t step0, uint32_t K, const float4* Fw, const uint4* queue, unsigned int* ctl,
    uint32_t most) {
    __shared__ RunSmem<kLevels> sm;
    const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
    const uint32_t count = queue ? ctl[kCtlQueue] : 0u;
    if (queue && (count > most || blockIdx.x >= count)) return;
    const bool mine = lane < (int)c.dim;
    RunCounts n;
    Walk w;
    w.k = w.org = 0;
    w.p = 0.f;
    float xd = 0.f, E1 = 0.f, E2 = 0.f, Ua = 0.f;
    uint64_t i = 0;
    bool have = false, local = false;
    while (true) {
        if (warp == 0) {
            bool done = false;
            while (!local && !done) {  // until a chain has a local step
                if (have) {  // the window's end
                    if (w.org && mine) xd = regen_lane(c, c.chain_offset + (uint32_t)i, step0 + w.org - 1);
                    if (mine) c.x[xidx((uint32_t)lane, i, c.n)] = xd;
                    if (lane == 0) w.store(c, i);
                    have = false;
                    if (!queue) done = true;
                    continue;
                }
                if (queue) {
                    unsigned q = 0;
                    if (lane == 0) q = atomicAdd(ctl + kCtlTail, 1u);
                    q = __shfl_sync(kFull, q, 0);
                    if (q >= count) {
                        done = true;
                        continue;
                    }
                    const uint4 e = queue[q];
                    i = e.x;
                    w.k = e.y;
                    w.org = e.z;
                } else {
                    i = blockIdx.x;
                }
                have = true;
                w.load(c, i);
                xd = mine ? c.x[xidx((uint32_t)lane, i, c.n)] : 0.0f;
                if (queue) {  // the queued step is local
                    if (w.org && mine) xd = regen_lane(c, c.chain_offset + (uint32_t)i, step0 + w.org - 1);
                    w.org = 0;
                    local = true;
                } else {
                    local = walk_window(c, i, step0, K, Fw, w, xd, false, n);
                }
            }
            sm.base[lane] = xd;
            if (lane == 0) {
                sm.step = step0 + w.k;
                sm.end = step0 + K;
                sm.chain = c.chain_offset + (uint32_t)i;
                sm.go = !done;
            }
        }
        __syncthreads();
        if (!sm.go) break;
        if (warp > 0) trace_node<kCheck, kLevels, kBrute>(s, c, sm);
        else round_draws(c, sm, E1, E2, Ua);
        __syncthreads();
        if (warp == 0) {
            uint64_t step = step0 + w.k;
            bool killed;
            local = follow(c, sm, w, xd, E1, E2, Ua, step, killed, n);
            w.k = (uint32_t)(step - step0);
            if (killed) local = walk_window(c, i, step0, K, Fw, w, xd, true, n);
        }
    }
    if (warp == 0 && lane == 0) n.flush(c);
}

// The same for more chains than that: one warp per chain, a step at a time.
__global__ void __launch_bounds__(128) settle_warp_kernel(SceneView s, ChainView c, uint64_t step0, uint32_t K,
                                                          const float4* Fw) {
    const uint64_t i = (blockIdx.x * (uint64_t)blockDim.x + threadIdx.x) >> 5;
    if (i >= c.n) return;  // a whole warp
    const int lane = threadIdx.x & 31;
    const bool mine = lane < (int)c.dim;
    const uint32_t chain = c.chain_offset + (uint32_t)i;
    RunCounts n;
    Walk w;
    w.k = w.org = 0;
    w.load(c, i);
    float xd = mine ? c.x[xidx((uint32_t)lane, i, c.n)] : 0.0f;
    while (walk_window(c, i, step0, K, Fw, w, xd, false, n)) {
        const float yd = mine ? move_lane(c, chain, step0 + w.k, xd) : 0.0f;
        const float3 F = eval_path_warp(s, (int)c.depth, yd, n.status);
        const float py = lum(F);
        const bool accept = u01(draw(c.seed, kTagStep, 0, chain, step0 + w.k).z) * w.p < py;
        n.nL++;
        n.nA += accept;
        if (accept) {
            xd = yd;
            w.Fr = F.x;
            w.Fg = F.y;
            w.Fb = F.z;
            w.p = py;
            w.u = 1.0f;
        }
        ++w.k;
    }
    if (w.org && mine) xd = regen_lane(c, chain, step0 + w.org - 1);
    if (mine) c.x[xidx((uint32_t)lane, i, c.n)] = xd;
    if (lane == 0) {
        w.store(c, i);
        n.flush(c);
    }
}

// A drain's open tours (drain_kernel's steps): chains with c.wf.done = 0, fetched 32
// at a time.
template <int kCheck, int kLevels>
__global__ void __launch_bounds__(32 << kLevels, 16 >> kLevels) runs_drain_kernel(SceneView s, ChainView c,
                                                                                  uint64_t step_begin,
                                                                                  uint32_t n_steps,
                                                                                  unsigned long long* ctl) {
    __shared__ RunSmem<kLevels> sm;
    const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
    const bool mine = lane < (int)c.dim;
    RunCounts n;
    Walk w;
    w.k = w.org = 0;
    w.p = 0.f;
    float xd = 0.f, E1 = 0.f, E2 = 0.f, Ua = 0.f;
    uint64_t i = 0, step = step_begin, mark = 0, base = 0;
    const uint64_t end = step_begin + n_steps;
    unsigned todo = 0;  // the fetched chains base .. base + 31 still to do
    uint32_t open = 0;
    bool have = false, local = false;
    while (true) {
        if (warp == 0) {
            bool done = false;
            while (!local && !done) {
                if (have) {  // the tour's end, or the last step
                    if (mine) c.x[xidx((uint32_t)lane, i, c.n)] = xd;
                    if (lane == 0) w.store(c, i);
                    have = false;
                    continue;
                }
                if (!todo) {
                    unsigned long long b = 0;
                    if (lane == 0) b = atomicAdd(ctl, 32ull);
                    base = __shfl_sync(kFull, b, 0);
                    if (base >= c.n) {
                        done = true;
                        continue;
                    }
                    todo = __ballot_sync(kFull, base + lane < c.n && !c.wf.done[base + lane]);
                    continue;
                }
                i = base + (uint64_t)__ffs(todo) - 1;
                todo &= todo - 1;
                have = true;
                step = step_begin;
                w.load(c, i);
                xd = mine ? c.x[xidx((uint32_t)lane, i, c.n)] : 0.0f;
                float dt;
                local = restore_clocks(c, draw(c.seed, kTagStep, 0, c.chain_offset + (uint32_t)i, step), w.p, w.u, dt);
                const float x0 = __shfl_sync(kFull, xd, 0), x1 = __shfl_sync(kFull, xd, 1);
                if (lane == 0) splat_state(c, w, x0, x1, dt);
                if (!local) {
                    n.nJ++;
                    if (lane == 0) c.wf.done[i] = 1;
                }
            }
            if (local) mark = max(mark, step + 1);
            sm.base[lane] = xd;
            if (lane == 0) {
                sm.step = step;
                sm.end = end;
                sm.chain = c.chain_offset + (uint32_t)i;
                sm.go = !done;
            }
        }
        __syncthreads();
        if (!sm.go) break;
        if (warp > 0) trace_node<kCheck, kLevels, false>(s, c, sm);
        else round_draws(c, sm, E1, E2, Ua);
        __syncthreads();
        if (warp == 0) {
            bool killed;
            local = follow(c, sm, w, xd, E1, E2, Ua, step, killed, n);
            // the last local step: the one before `step` (killed, or the end), or `step` itself
            mark = max(mark, local ? step + 1 : step);
            if (killed) {
                n.nJ++;
                if (lane == 0) c.wf.done[i] = 1;
            } else if (!local) {
                open++;
            }
        }
    }
    if (warp == 0 && lane == 0) {
        n.flush(c);
        if (mark) atomicMax(c.counters + 3, (unsigned long long)mark);
        if (open) atomicAdd(ctl + 1, (unsigned long long)open);
    }
}

// Blocks of kernel the device holds at once.
template <class K>
cudaError_t resident(K kernel, int threads, long long* blocks) {
    int dev = 0, sms = 0, per_sm = 0;
    cudaError_t e;
    if ((e = cudaGetDevice(&dev)) != cudaSuccess ||
        (e = cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, dev)) != cudaSuccess ||
        (e = cudaOccupancyMaxActiveBlocksPerMultiprocessor(&per_sm, kernel, threads, 0)) != cudaSuccess)
        return e;
    *blocks = (long long)sms * (per_sm > 0 ? per_sm : 1);
    return cudaSuccess;
}

constexpr int kDeep = 3;  // steps per round: 7 node warps and the control warp
// Queues of up to this many chains per resident block go to the blocks: 32 steps of
// 10 007 chains on Cornell + spheres 984 us without them, 809 at one, 696 at two and
// above; 16 steps of 2^16 chains 1 039 at two, 928 at five, 927 at ten.
constexpr uint32_t kRunsTailWaves = 8;

}  // namespace

cudaError_t launch_runs_settle(const SceneView& s, const ChainView& c, uint64_t step0, uint32_t K, const float4* F,
                               cudaStream_t st) {
    // The deepest round whose blocks the device still holds all at once; beyond two
    // steps' worth the spare warps are gone (24-triangle box, 400 steps: 256 chains
    // 334 us at three steps a round, 453 us a step at a time; 600 chains 421 at two, 507;
    // 3 000 chains 991 with a second warp per chain, 769 without).
    long long deep = 0, mid = 0;
    cudaError_t e;
    if ((e = resident(runs_window_kernel<0, 3, true>, 256, &deep)) != cudaSuccess ||
        (e = resident(runs_window_kernel<0, 2, true>, 128, &mid)) != cudaSuccess)
        return e;
    const unsigned n = (unsigned)c.n;
    if (c.n <= (uint64_t)deep)
        runs_window_kernel<0, 3, true><<<n, 256, 0, st>>>(s, c, step0, K, F, nullptr, nullptr, 0);
    else if (c.n <= (uint64_t)mid)
        runs_window_kernel<0, 2, true><<<n, 128, 0, st>>>(s, c, step0, K, F, nullptr, nullptr, 0);
    else
        settle_warp_kernel<<<(unsigned)((32 * c.n + 127) / 128), 128, 0, st>>>(s, c, step0, K, F);
    return cudaGetLastError();
}

cudaError_t launch_runs_tail(const SceneView& s, const ChainView& c, uint64_t step0, uint32_t K, const float4* F,
                             const uint4* queue, unsigned int* ctl, uint32_t* most, cudaStream_t st) {
    cudaError_t e = cudaSuccess;
    with_checks(trav_checks(s), [&](auto kc) {
        const auto kernel = runs_window_kernel<decltype(kc)::value, kDeep, false>;
        long long blocks = 0;
        if ((e = resident(kernel, 32 << kDeep, &blocks)) != cudaSuccess) return;
        *most = (uint32_t)(kRunsTailWaves * blocks);
        kernel<<<(unsigned)std::min<uint64_t>((uint64_t)blocks, c.n), 32 << kDeep, 0, st>>>(s, c, step0, K, F, queue,
                                                                                           ctl, *most);
        e = cudaGetLastError();
    });
    return e;
}

cudaError_t launch_runs_drain(const SceneView& s, const ChainView& c, uint64_t step_begin, uint32_t n_steps,
                              unsigned long long* ctl, cudaStream_t st) {
    cudaError_t e = cudaMemsetAsync(ctl, 0, 2 * sizeof(unsigned long long), st);
    if (e != cudaSuccess) return e;
    with_checks(trav_checks(s), [&](auto kc) {
        const auto kernel = runs_drain_kernel<decltype(kc)::value, kDeep>;
        long long blocks = 0;
        if ((e = resident(kernel, 32 << kDeep, &blocks)) != cudaSuccess) return;
        kernel<<<(unsigned)blocks, 32 << kDeep, 0, st>>>(s, c, step_begin, n_steps, ctl);
        e = cudaGetLastError();
    });
    return e;
}

}  // namespace jr
