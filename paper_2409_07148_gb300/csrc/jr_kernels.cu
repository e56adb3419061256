// Device code of the Jump Restore light-transport library (sm_103a).
//
// One thread owns one chain for a whole launch (persistent over n_steps).  The
// current state x and the candidate y live in dynamic shared memory, [buf][d]
// [thread] (bank-conflict free), so the accepted move is a buffer flip; F, p
// and u of the current state stay in registers.  Each step runs Alg. 2
// (Section 7.2) of Holl, Singh, Seidel, "Jump Restore Light Transport":
//   t1 ~ Exp(1), t2 ~ Exp(k(x)) with k = c~ u / p (Section 6.2),
//   splat (dt, x) into the framebuffer (Section 6.3 / 7.4 estimator),
//   t1 < t2: local MH move with the Gaussian small-step kernel (Alg. 1),
//   else   : regenerate x ~ mu (uniform) and count a tour.
// Both branches end in exactly one evaluation of the integrand, so the only
// divergence between them is the few instructions that build y.
#include <cuda_runtime.h>
#include <math.h>
#include <stdint.h>

#include <algorithm>

#include "../../include/jr.h"
#include "jr_device.cuh"
#include "jr_internal.h"

namespace jr {
namespace {

// ------------------------------------------------------------------ kernels
// x0 ~ mu (tag 1); y built in shared memory, then written to the SoA state.  The sum
// of p goes to counters[kCounterMuP], one atomic per block (a launch of its own
// took 6 to 30 us of a set's creation).
template <int kCheck>
__global__ void init_kernel(SceneView s, ChainView c) {
    extern __shared__ float sh[];
    __shared__ double sum_p;
    const uint32_t B = blockDim.x, tid = threadIdx.x;
    const uint64_t i = blockIdx.x * (uint64_t)B + tid;
    const bool valid = i < c.n;
    if (tid == 0) sum_p = 0.0;
    __syncthreads();
    const int D = (int)c.dim;
    float* y = sh + tid;
    if (valid) {
        const uint32_t chain = c.chain_offset + (uint32_t)i;
        for (int b = 0; 4 * b < D; ++b) {
            const uint4 r = draw(c.seed, kTagInit, (uint32_t)(b + 1), chain, 0);
            const uint32_t rr[4] = {r.x, r.y, r.z, r.w};
#pragma unroll
            for (int q = 0; q < 4; ++q)
                if (4 * b + q < D) y[(4 * b + q) * B] = u01(rr[q]);
        }
    }
    unsigned status = 0;
    const float3 F = eval_path<kCheck>(s, 0xffffffffu, valid, (int)c.depth, y, B, nullptr, 0, status);
    const float p = valid ? lum(F) : 0.0f;
    if (valid) {
        float2* x2 = reinterpret_cast<float2*>(c.x);
        for (int k = 0; 2 * k < D; ++k) x2[(uint64_t)k * c.n + i] = make_float2(y[2 * k * B], y[(2 * k + 1) * B]);
        c.fpu[0 * c.n + i] = F.x;
        c.fpu[1 * c.n + i] = F.y;
        c.fpu[2 * c.n + i] = F.z;
        c.fpu[3 * c.n + i] = p;
        c.fpu[4 * c.n + i] = 1.0f;  // u of uniform mu
        flush_status(status, c.status);
    }
    const double v = warp_sum((double)p);
    if ((tid & 31) == 0 && v != 0.0) atomicAdd(&sum_p, v);
    __syncthreads();
    if (tid == 0 && sum_p != 0.0) atomicAdd(reinterpret_cast<double*>(c.counters + kCounterMuP), sum_p);
}

// Re-evaluate F, p, u of the stored states (after jr_set_state).
__global__ void reeval_kernel(SceneView s, ChainView c) {
    extern __shared__ float sh[];
    const uint64_t i = blockIdx.x * (uint64_t)blockDim.x + threadIdx.x;
    const unsigned mask = __ballot_sync(0xffffffffu, i < c.n);
    if (i >= c.n) return;
    unsigned status = 0;
    load_coords(c, i, sh + threadIdx.x, blockDim.x);
    const float3 F = eval_path<kCheckAll>(s, mask, true, (int)c.depth, sh + threadIdx.x, blockDim.x, nullptr, 0, status);
    c.fpu[0 * c.n + i] = F.x;
    c.fpu[1 * c.n + i] = F.y;
    c.fpu[2 * c.n + i] = F.z;
    c.fpu[3 * c.n + i] = lum(F);
    c.fpu[4 * c.n + i] = 1.0f;
    flush_status(status, c.status);
}

// n_steps of Alg. 2 for chain i of set c (thread tid of the block; `active`
// false for threads without a chain).  Every thread of the block calls it;
// sh holds [2][D][blockDim] floats.
template <int kCheck, bool kTrace, bool kCount, bool kSorted = false>
__device__ __forceinline__ void chain_steps(const SceneView& s, const ChainView& c, uint64_t i, bool active, float* sh,
                                            uint64_t step_begin, uint32_t n_steps, uint8_t* tr_flags, float* tr_dt,
                                            int32_t* tr_pix, unsigned long long* work_out) {
    const uint32_t B = blockDim.x, tid = threadIdx.x;
    const unsigned mask = __ballot_sync(0xffffffffu, active);  // lanes that trace together
    const int D = (int)c.dim;
    float* buf0 = sh + tid;
    float* buf1 = sh + (size_t)D * B + tid;
    uint32_t nJ = 0, nL = 0, nA = 0;
    unsigned status = 0;
    Work work;
    const bool mh = (c.flags & JR_FLAG_MH) != 0;
    double psum = 0.0;  // MH: sum of p over this chain's large-step proposals
    if (active) {
        load_coords(c, i, buf0, B);
        float Fr = c.fpu[0 * c.n + i], Fg = c.fpu[1 * c.n + i], Fb = c.fpu[2 * c.n + i];
        float p = c.fpu[3 * c.n + i], u = c.fpu[4 * c.n + i];
        float* cur = buf0;
        float* cand = buf1;
        const uint32_t chain = c.chain_offset + (uint32_t)i;
        const float WH = (float)c.width * (float)c.height;
        for (uint32_t st = 0; st < n_steps; ++st) {
            const uint64_t step = step_begin + st;
            const uint4 r0 = draw(c.seed, kTagStep, 0, chain, step);
            const float Ua = u01(r0.z);
            bool local;
            float dt;
            if (mh) {
                // the MH baseline: a large step (from mu) with probability l, else
                // a small step; the state before the iteration enters the
                // estimator once the burn-in is over (dt = 1 counts it)
                local = !(u01(r0.x) < c.large_step);
                dt = step >= c.burn_in ? 1.0f : 0.0f;
            } else {
                local = restore_clocks(c, r0, p, u, dt);
            }
            int32_t pix = -1;
            if (dt > 0.0f && p > 0.0f) {
                // left-rectangle estimator: x_{i-1} weighted by dt_i (Section 7.4);
                // MH: the ergodic average's term W H F / p of the held state
                uint32_t px = (uint32_t)((double)cur[0] * (double)c.width);
                uint32_t py = (uint32_t)((double)cur[B] * (double)c.height);
                px = min(px, c.width - 1);
                py = min(py, c.height - 1);
                pix = (int32_t)(py * c.width + px);
                const float wgt = mh ? WH / p : c.c_tilde * dt * WH / p;
                atomicAdd(c.fb + pix, make_float4(wgt * Fr, wgt * Fg, wgt * Fb, dt));
            }
            propose(c, chain, step, local, cur, cand, B);
            const float3 Fy = eval_path_w<kCheck, kCount, true, kSorted>(s, mask, true, (int)c.depth, cand, B, nullptr, 0,
                                                                         status, work);
            const float py_ = lum(Fy);
            bool accept;
            if (mh) {  // Alg. 1: U < min(1, p(y)/p(x)), 1 if p(x) = 0
                accept = !(p > 0.0f) || Ua * p < py_;
                if (local) {
                    nL++;
                } else {
                    nJ++;
                    psum += (double)py_;
                }
                nA += accept;
            } else if (local) {
                accept = Ua * p < py_;  // U < min(1, p(y)/p(x)), p(x) > 0 on this branch
                nL++;
                nA += accept;
            } else {
                accept = true;
                nJ++;
            }
            if (accept) {
                float* tmp = cur;
                cur = cand;
                cand = tmp;
                Fr = Fy.x;
                Fg = Fy.y;
                Fb = Fy.z;
                p = py_;
                u = 1.0f;
            }
            if (kTrace) {
                const uint64_t o = i * n_steps + st;
                if (tr_flags) tr_flags[o] = (uint8_t)((local ? 0 : 1) | ((mh || local) && accept ? 2 : 0));
                if (tr_dt) tr_dt[o] = pix >= 0 ? dt : 0.0f;
                if (tr_pix) tr_pix[o] = pix;
            }
        }
        float2* x2 = reinterpret_cast<float2*>(c.x);
        for (int k = 0; 2 * k < D; ++k) x2[(uint64_t)k * c.n + i] = make_float2(cur[2 * k * B], cur[(2 * k + 1) * B]);
        c.fpu[0 * c.n + i] = Fr;
        c.fpu[1 * c.n + i] = Fg;
        c.fpu[2 * c.n + i] = Fb;
        c.fpu[3 * c.n + i] = p;
        c.fpu[4 * c.n + i] = u;
    }
    // warp-aggregated counters: one 64-bit atomic per warp and counter
    nJ = __reduce_add_sync(0xffffffffu, nJ);
    nL = __reduce_add_sync(0xffffffffu, nL);
    nA = __reduce_add_sync(0xffffffffu, nA);
    status = __reduce_or_sync(0xffffffffu, status);
    if (mh) psum = warp_sum(psum);
    if constexpr (kCount) {
        const uint32_t r = __reduce_add_sync(0xffffffffu, work.rays);
        const uint32_t nd = __reduce_add_sync(0xffffffffu, work.nodes);
        const uint32_t tr = __reduce_add_sync(0xffffffffu, work.tris);
        if ((tid & 31) == 0) {
            atomicAdd(work_out + 0, (unsigned long long)r);
            atomicAdd(work_out + 1, (unsigned long long)nd);
            atomicAdd(work_out + 2, (unsigned long long)tr);
        }
    }
    if ((tid & 31) == 0) {
        if (nJ) atomicAdd(c.counters + 0, (unsigned long long)nJ);
        if (nL) atomicAdd(c.counters + 1, (unsigned long long)nL);
        if (nA) atomicAdd(c.counters + 2, (unsigned long long)nA);
        if (psum != 0.0) atomicAdd(reinterpret_cast<double*>(c.counters + kCounterPSum), psum);
        flush_status(status, c.status);
    }
}

// Both persistent kernels are capped at 64 registers (4 blocks of 256 threads
// per SM): the 4-wide traversal would take 110, and the occupancy the cap buys
// outweighs its small spill (measured: 5.0 -> 5.9e8 chain steps/s for the
// megakernel, 5.9 -> 6.1e8 for the 64-scene batch).
// The traced and the counted variant hold more and run with few chains, so they may
// take 80 registers, and sort fully (5 000 chains, 8 steps, traced: Cornell + spheres 1 032 ->
// 906 us, glass furnace 1 358 -> 930, 180 000-triangle terrain 726 -> 548).
template <int kCheck, bool kTrace, bool kCount>
__global__ void __launch_bounds__(256, kTrace || kCount ? 3 : 4) step_kernel(SceneView s, ChainView c, uint64_t step_begin, uint32_t n_steps,
                                                   uint8_t* tr_flags, float* tr_dt, int32_t* tr_pix,
                                                   unsigned long long* work_out) {
    extern __shared__ float sh[];
    const uint64_t i = blockIdx.x * (uint64_t)blockDim.x + threadIdx.x;
    chain_steps<kCheck, kTrace, kCount, kTrace || kCount>(s, c, i, i < c.n, sh, step_begin, n_steps, tr_flags, tr_dt,
                                                          tr_pix, work_out);
}

// The megakernel where all chains fit on the device at once: a warp holds only
// `per_warp` chains, in its first lanes, so that the chains spread over all the
// warps that can be resident.  Such a launch is bound by latency: a warp's step
// lasts as long as the divergent paths of all its lanes together, so fewer lanes
// per warp shorten it (1 000 chains, 16 steps of Cornell + spheres: 1 377 us
// with 32 chains per warp, 1 024 with 16, 770 with 8, 570 with 4, 426 with 2, 340 with
// one) while issue slots are left over.  Blocks of one warp, so that warps spread
// evenly over the SMs, and no register cap below what 16 warps per SM leave: a
// spill would lengthen the step (1 587 -> 1 377 us) and more warps would not be
// resident anyway.
template <int kCheck>
__global__ void __launch_bounds__(32, 16) step_kernel_spread(SceneView s, ChainView c, uint64_t step_begin,
                                                             uint32_t n_steps, uint32_t per_warp) {
    extern __shared__ float sh[];
    const uint64_t i = blockIdx.x * (uint64_t)per_warp + threadIdx.x;
    const bool active = threadIdx.x < per_warp && i < c.n;
    chain_steps<kCheck, false, false>(s, c, i, active, sh, step_begin, n_steps, nullptr, nullptr, nullptr, nullptr);
}

// ------------------------------------------------------------------ drain tail
// The open tours of a drain, each run to its end in one launch: lane = chain,
// one-warp blocks, chains fetched from [0, n) (those with done[i] skipped) as
// lanes become free.  A chain takes steps step_begin, step_begin + 1, ... of Alg. 2
// until a kill ends its tour (J += 1, done = 1) or n_steps are taken; a chain
// still open then is stored and counted in ctl[1] (ctl[0]: the fetch cursor).
//
// The tail of a drain is a few hundred chains with tours of up to several
// hundred steps.  In the wavefront every step waits for the longest of their
// paths and for three launches over all chains; here a chain waits for no other
// but the few in its warp, so the drain lasts as long as its longest tour.
template <int kCheck>
__global__ void __launch_bounds__(32, 16) drain_kernel(SceneView s, ChainView c, uint64_t step_begin,
                                                       uint32_t n_steps, unsigned long long* ctl) {
    extern __shared__ float sh[];
    constexpr uint32_t B = 32;
    const int lane = threadIdx.x;
    const float WH = (float)c.width * (float)c.height;
    const uint64_t end = step_begin + n_steps;
    float* cur = sh + lane;
    float* cand = sh + (size_t)c.dim * B + lane;
    uint32_t nJ = 0, nL = 0, nA = 0, open = 0;
    unsigned status = 0;
    Work work;
    bool live = false, drained = false;
    uint64_t i = 0, step = step_begin, mark = 0;
    float Fr = 0.f, Fg = 0.f, Fb = 0.f, p = 0.f, u = 1.f;
    // The start of step `step`: clocks and splat.  False: the tour ends here.
    auto begin_step = [&](float x0, float x1) {
        float dt;
        const bool local = restore_clocks(c, draw(c.seed, kTagStep, 0, c.chain_offset + (uint32_t)i, step), p, u, dt);
        if (dt > 0.0f && p > 0.0f) {
            const uint32_t px = min((uint32_t)((double)x0 * (double)c.width), c.width - 1);
            const uint32_t py = min((uint32_t)((double)x1 * (double)c.height), c.height - 1);
            const float wgt = c.c_tilde * dt * WH / p;
            atomicAdd(c.fb + (py * c.width + px), make_float4(wgt * Fr, wgt * Fg, wgt * Fb, dt));
        }
        if (local) {
            mark = max(mark, step + 1);
        } else {
            nJ++;
            c.wf.done[i] = 1;
        }
        return local;
    };
    while (true) {
        while (__any_sync(0xffffffffu, !live && !drained)) {  // free lanes take chains until one is in a tour
            const unsigned want = __ballot_sync(0xffffffffu, !live && !drained);
            unsigned long long base = 0;
            if (lane == 0) base = atomicAdd(ctl, (unsigned long long)__popc(want));
            base = __shfl_sync(0xffffffffu, base, 0);
            if (!live && !drained) {
                i = base + __popc(want & ((1u << lane) - 1u));
                drained = i >= c.n;
                if (!drained && !c.wf.done[i]) {
                    p = c.fpu[3 * c.n + i];
                    step = step_begin;
                    if (!(p > 0.0f)) {  // k = inf: killed at once, nothing to splat
                        nJ++;
                        c.wf.done[i] = 1;
                    } else {
                        Fr = c.fpu[0 * c.n + i];
                        Fg = c.fpu[1 * c.n + i];
                        Fb = c.fpu[2 * c.n + i];
                        u = c.fpu[4 * c.n + i];
                        load_coords(c, i, cur, B);
                        live = begin_step(cur[0], cur[B]);
                    }
                }
            }
        }
        if (!__any_sync(0xffffffffu, live)) break;
        if (live) propose(c, c.chain_offset + (uint32_t)i, step, true, cur, cand, B);
        const float3 Fy = eval_path_w<kCheck, false>(s, 0xffffffffu, live, (int)c.depth, cand, B, nullptr, 0, status, work);
        if (live) {
            const float py = lum(Fy);
            const bool accept = u01(draw(c.seed, kTagStep, 0, c.chain_offset + (uint32_t)i, step).z) * p < py;
            nL++;
            nA += accept;
            if (accept) {
                float* t = cur;
                cur = cand;
                cand = t;
                Fr = Fy.x;
                Fg = Fy.y;
                Fb = Fy.z;
                p = py;
                u = 1.0f;
            }
            ++step;
            const bool last = step == end;
            if (last) open++;
            else live = begin_step(cur[0], cur[B]);
            if (last || !live) {
                live = false;
                float2* x2 = reinterpret_cast<float2*>(c.x);
                for (int k = 0; 2 * k < (int)c.dim; ++k)
                    x2[(uint64_t)k * c.n + i] = make_float2(cur[2 * k * B], cur[(2 * k + 1) * B]);
                c.fpu[0 * c.n + i] = Fr;
                c.fpu[1 * c.n + i] = Fg;
                c.fpu[2 * c.n + i] = Fb;
                c.fpu[3 * c.n + i] = p;
                c.fpu[4 * c.n + i] = u;
            }
        }
    }
    nJ = __reduce_add_sync(0xffffffffu, nJ);
    nL = __reduce_add_sync(0xffffffffu, nL);
    nA = __reduce_add_sync(0xffffffffu, nA);
    open = __reduce_add_sync(0xffffffffu, open);
    status = __reduce_or_sync(0xffffffffu, status);
    if (mark) atomicMax(c.counters + 3, (unsigned long long)mark);
    if (lane == 0) {
        if (nJ) atomicAdd(c.counters + 0, (unsigned long long)nJ);
        if (nL) atomicAdd(c.counters + 1, (unsigned long long)nL);
        if (nA) atomicAdd(c.counters + 2, (unsigned long long)nA);
        if (open) atomicAdd(ctl + 1, (unsigned long long)open);
        flush_status(status, c.status);
    }
}

// ------------------------------------------------------------------ one chain per warp
// For scenes of at most kWarpChainMaxTris triangles with few chains (the
// megakernel's case), one warp carries one chain: lane d holds coordinate d,
// draws its own Philox block and Box-Muller pair, and a ray tests every
// triangle, triangle k in lane k mod 32, before a butterfly reduction picks the
// closest hit.  A step's latency then shrinks to a few triangle tests and one
// shading per vertex, and a few hundred chains spread over as many SMs as
// their warps fill.  The per-chain arithmetic is chain_steps': the same draws,
// the same Box-Muller expressions and acceptance, the same camera_ray and
// shade_vertex; the closest hit is the least (t, original index) over all
// triangles with t > 0, which is what the BVH traversal returns too.

constexpr int kWarpChainThreads = 128;  // four chains per block

__global__ void __launch_bounds__(kWarpChainThreads) step_kernel_warp(SceneView s, ChainView c, uint64_t step_begin,
                                                                      uint32_t n_steps) {
    const uint64_t i = (blockIdx.x * (uint64_t)blockDim.x + threadIdx.x) >> 5;
    if (i >= c.n) return;  // a whole warp
    const int lane = threadIdx.x & 31;
    const int D = (int)c.dim;
    const bool mine = lane < D;  // this lane holds coordinate `lane`
    const uint32_t chain = c.chain_offset + (uint32_t)i;
    const bool mh = (c.flags & JR_FLAG_MH) != 0, rb = (c.flags & JR_FLAG_RAO_BLACKWELL) != 0;
    const float c_tilde = c.c_tilde, sigma = c.sigma;
    const float WH = (float)c.width * (float)c.height;
    uint32_t nJ = 0, nL = 0, nA = 0;
    unsigned status = 0;
    double psum = 0.0;
    float xd = mine ? c.x[xidx((uint32_t)lane, i, c.n)] : 0.0f;
    float Fr = c.fpu[0 * c.n + i], Fg = c.fpu[1 * c.n + i], Fb = c.fpu[2 * c.n + i];
    float p = c.fpu[3 * c.n + i], u = c.fpu[4 * c.n + i];
    for (uint32_t st = 0; st < n_steps; ++st) {
        const uint64_t step = step_begin + st;
        const uint4 r0 = draw(c.seed, kTagStep, 0, chain, step);
        const float Ua = u01(r0.z);
        bool local;
        float dt;
        if (mh) {
            local = !(u01(r0.x) < c.large_step);
            dt = step >= c.burn_in ? 1.0f : 0.0f;
        } else {
            const float E1 = -logf(1.0f - u01(r0.x));
            const float E2 = -logf(1.0f - u01(r0.y));
            const float t2 = p > 0.0f ? E2 * p / (c_tilde * u) : 0.0f;
            local = E1 < t2;  // a tie goes to the killing branch
            dt = local ? E1 : t2;
            if (rb) dt = p > 0.0f ? p / (p + c_tilde * u) : 0.0f;
        }
        const float x0 = __shfl_sync(0xffffffffu, xd, 0), x1 = __shfl_sync(0xffffffffu, xd, 1);
        if (lane == 0 && dt > 0.0f && p > 0.0f) {
            uint32_t px = (uint32_t)((double)x0 * (double)c.width);
            uint32_t py = (uint32_t)((double)x1 * (double)c.height);
            px = min(px, c.width - 1);
            py = min(py, c.height - 1);
            const float wgt = mh ? WH / p : c_tilde * dt * WH / p;
            atomicAdd(c.fb + (py * c.width + px), make_float4(wgt * Fr, wgt * Fg, wgt * Fb, dt));
        }
        // candidate coordinate `lane`: Philox block lane / 4 + 1; a local move's
        // Box-Muller pair is (r.x, r.y) for the block's first two coordinates
        // and (r.z, r.w) for the last two
        float yd = 0.0f;
        if (mine) {
            const uint4 r = draw(c.seed, kTagStep, (uint32_t)(lane >> 2) + 1u, chain, step);
            const bool second = (lane & 2) != 0;
            if (local) {
                float sn, cs;
                const float R = sqrtf(-2.0f * logf(1.0f - u01(second ? r.z : r.x)));
                sincospif(2.0f * u01(second ? r.w : r.y), &sn, &cs);
                yd = wrap01(xd + sigma * R * ((lane & 1) ? sn : cs));
            } else {
                yd = u01(second ? ((lane & 1) ? r.w : r.z) : ((lane & 1) ? r.y : r.x));
            }
        }
        const float3 Fy = eval_path_warp(s, (int)c.depth, yd, status);
        const float py_ = lum(Fy);
        bool accept;
        if (mh) {
            accept = !(p > 0.0f) || Ua * p < py_;
            if (local) {
                nL++;
            } else {
                nJ++;
                psum += (double)py_;
            }
            nA += accept;
        } else if (local) {
            accept = Ua * p < py_;
            nL++;
            nA += accept;
        } else {
            accept = true;
            nJ++;
        }
        if (accept) {
            xd = yd;
            Fr = Fy.x;
            Fg = Fy.y;
            Fb = Fy.z;
            p = py_;
            u = 1.0f;
        }
    }
    if (mine) c.x[xidx((uint32_t)lane, i, c.n)] = xd;
    if (lane == 0) {
        c.fpu[0 * c.n + i] = Fr;
        c.fpu[1 * c.n + i] = Fg;
        c.fpu[2 * c.n + i] = Fb;
        c.fpu[3 * c.n + i] = p;
        c.fpu[4 * c.n + i] = u;
        if (nJ) atomicAdd(c.counters + 0, (unsigned long long)nJ);
        if (nL) atomicAdd(c.counters + 1, (unsigned long long)nL);
        if (nA) atomicAdd(c.counters + 2, (unsigned long long)nA);
        if (psum != 0.0) atomicAdd(reinterpret_cast<double*>(c.counters + kCounterPSum), psum);
        flush_status(status, c.status);
    }
}

// ------------------------------------------------------------------ MALA
// Langevin local dynamics (JR_FLAG_MALA), one chain per thread for the whole
// launch.  The state's drift m(x) = clamp(sigma^2/2 grad log p(x), -2 sigma,
// 2 sigma) lives beside it (shared memory during the launch, c.drift between
// launches).  A MALA move proposes y = (x + m(x) + sigma N) mod 1 and accepts
// with min(1, p(y) q(x|y) / (p(x) q(y|x))), q(b|a) = prod_d phi_sigma(b_d - a_d
// - m_d(a)) on the signed torus difference.  With JR_FLAG_MH the chain is the
// MALA baseline (large steps from mu with probability l, MALA small steps);
// otherwise MALA Restore (Alg. 2, local move = the MALA step, k = c~ u / p).
template <int kCheck, bool kTrace>
__device__ __forceinline__ void chain_steps_mala(const SceneView& s, const ChainView& c, uint64_t i, bool active,
                                                 float* sh, uint64_t step_begin, uint32_t n_steps, uint8_t* tr_flags,
                                                 float* tr_dt, int32_t* tr_pix) {
    const uint32_t B = blockDim.x, tid = threadIdx.x;
    const unsigned mask = __ballot_sync(0xffffffffu, active);
    const int D = (int)c.dim;
    float* x0 = sh + tid;                            // [4][D][B]: x, y, m(x), m(y)
    float* x1 = sh + (size_t)D * B + tid;
    float* m0 = sh + (size_t)2 * D * B + tid;
    float* m1 = sh + (size_t)3 * D * B + tid;
    const bool mh = (c.flags & JR_FLAG_MH) != 0;
    uint32_t nJ = 0, nL = 0, nA = 0;
    unsigned status = 0;
    double psum = 0.0;
    Work work;
    Jac3 JF;
    if (active) {
        load_coords(c, i, x0, B);
        for (int d = 0; d < D; ++d) m0[d * B] = c.drift[d * c.n + i];
    }
    float Fr = 0.f, Fg = 0.f, Fb = 0.f, p = 0.f, u = 1.f;
    if (active) {
        Fr = c.fpu[0 * c.n + i];
        Fg = c.fpu[1 * c.n + i];
        Fb = c.fpu[2 * c.n + i];
        p = c.fpu[3 * c.n + i];
        u = c.fpu[4 * c.n + i];
    }
    float *cur = x0, *cand = x1, *mc = m0, *my = m1;
    const uint32_t chain = c.chain_offset + (uint32_t)i;
    const float WH = (float)c.width * (float)c.height;
    for (uint32_t st = 0; st < n_steps; ++st) {
        const uint64_t step = step_begin + st;
        const uint4 r0 = active ? draw(c.seed, kTagStep, 0, chain, step) : make_uint4(0, 0, 0, 0);
        const float Ua = u01(r0.z);
        bool local = false;
        float dt = 0.f;
        if (mh) {
            local = !(u01(r0.x) < c.large_step);
            dt = step >= c.burn_in ? 1.0f : 0.0f;
        } else {
            const float E1 = -logf(1.0f - u01(r0.x));
            const float E2 = -logf(1.0f - u01(r0.y));
            const float t2 = p > 0.0f ? E2 * p / (c.c_tilde * u) : 0.0f;
            local = E1 < t2;
            dt = local ? E1 : t2;
        }
        int32_t pix = -1;
        if (active && dt > 0.0f && p > 0.0f) {
            uint32_t px = min((uint32_t)((double)cur[0] * (double)c.width), c.width - 1);
            uint32_t py = min((uint32_t)((double)cur[B] * (double)c.height), c.height - 1);
            pix = (int32_t)(py * c.width + px);
            const float wgt = mh ? WH / p : c.c_tilde * dt * WH / p;
            atomicAdd(c.fb + pix, make_float4(wgt * Fr, wgt * Fg, wgt * Fb, dt));
        }
        if (active) {
            if (local) mala_propose(c, chain, step, cur, mc, cand, B);
            else propose(c, chain, step, false, cur, cand, B);
        }
        const float3 Fy = eval_path_grad<kCheck, false>(s, mask, active, (int)c.depth, cand, B, JF, status, work);
        bool accept = false;
        if (active) {
            for (int d = 0; d < D; ++d) my[d * B] = mala_drift(Fy, JF, d, c.sigma);
            const float py_ = lum(Fy);
            if (local) {
                accept = mala_accept(c, Ua, p, py_, cur, mc, cand, my, B);
                nL++;
                nA += accept;
            } else if (mh) {  // a large step: uniform and symmetric
                accept = !(p > 0.0f) || Ua * p < py_;
                nJ++;
                psum += (double)py_;
                nA += accept;
            } else {          // regeneration from mu
                accept = true;
                nJ++;
            }
            if (accept) {
                float* t0 = cur;
                cur = cand;
                cand = t0;
                float* t1 = mc;
                mc = my;
                my = t1;
                Fr = Fy.x;
                Fg = Fy.y;
                Fb = Fy.z;
                p = py_;
                u = 1.0f;
            }
            if (kTrace) {
                const uint64_t o = i * n_steps + st;
                if (tr_flags) tr_flags[o] = (uint8_t)((local ? 0 : 1) | ((mh || local) && accept ? 2 : 0));
                if (tr_dt) tr_dt[o] = pix >= 0 ? dt : 0.0f;
                if (tr_pix) tr_pix[o] = pix;
            }
        }
    }
    if (active) {
        float2* x2 = reinterpret_cast<float2*>(c.x);
        for (int k = 0; 2 * k < D; ++k) x2[(uint64_t)k * c.n + i] = make_float2(cur[2 * k * B], cur[(2 * k + 1) * B]);
        for (int d = 0; d < D; ++d) c.drift[d * c.n + i] = mc[d * B];
        c.fpu[0 * c.n + i] = Fr;
        c.fpu[1 * c.n + i] = Fg;
        c.fpu[2 * c.n + i] = Fb;
        c.fpu[3 * c.n + i] = p;
        c.fpu[4 * c.n + i] = u;
    }
    nJ = __reduce_add_sync(0xffffffffu, nJ);
    nL = __reduce_add_sync(0xffffffffu, nL);
    nA = __reduce_add_sync(0xffffffffu, nA);
    status = __reduce_or_sync(0xffffffffu, status);
    if (mh) psum = warp_sum(psum);
    if ((tid & 31) == 0) {
        if (nJ) atomicAdd(c.counters + 0, (unsigned long long)nJ);
        if (nL) atomicAdd(c.counters + 1, (unsigned long long)nL);
        if (nA) atomicAdd(c.counters + 2, (unsigned long long)nA);
        if (psum != 0.0) atomicAdd(reinterpret_cast<double*>(c.counters + kCounterPSum), psum);
        flush_status(status, c.status);
    }
}

// One-warp blocks of per_warp chains, as in step_kernel_spread (chains_per_warp).
template <int kCheck, bool kTrace>
__global__ void __launch_bounds__(32, 16) step_kernel_mala(SceneView s, ChainView c, uint64_t step_begin,
                                                           uint32_t n_steps, uint32_t per_warp, uint8_t* tr_flags,
                                                           float* tr_dt, int32_t* tr_pix) {
    extern __shared__ float sh[];
    const uint64_t i = blockIdx.x * (uint64_t)per_warp + threadIdx.x;
    const bool active = threadIdx.x < per_warp && i < c.n;
    chain_steps_mala<kCheck, kTrace>(s, c, i, active, sh, step_begin, n_steps, tr_flags, tr_dt, tr_pix);
}

// F, p and the drift of the stored states (chain creation and jr_set_state).
__global__ void __launch_bounds__(128) mala_reeval_kernel(SceneView s, ChainView c) {
    extern __shared__ float sh[];
    const uint64_t i = blockIdx.x * (uint64_t)blockDim.x + threadIdx.x;
    const unsigned mask = __ballot_sync(0xffffffffu, i < c.n);
    if (i >= c.n) return;
    unsigned status = 0;
    Work w;
    Jac3 JF;
    load_coords(c, i, sh + threadIdx.x, blockDim.x);
    const float3 F =
        eval_path_grad<kCheckAll, false>(s, mask, true, (int)c.depth, sh + threadIdx.x, blockDim.x, JF, status, w);
    c.fpu[0 * c.n + i] = F.x;
    c.fpu[1 * c.n + i] = F.y;
    c.fpu[2 * c.n + i] = F.z;
    c.fpu[3 * c.n + i] = lum(F);
    c.fpu[4 * c.n + i] = 1.0f;
    for (int d = 0; d < (int)c.dim; ++d) c.drift[d * c.n + i] = mala_drift(F, JF, d, c.sigma);
    flush_status(status, c.status);
}

// F and dF/dx for given states: x [D][n], F [3][n], dF [3][D][n].
__global__ void __launch_bounds__(128) eval_grad_kernel(SceneView s, uint32_t depth, const float* x, uint64_t n,
                                                        float* F, float* dF) {
    const uint64_t i = blockIdx.x * (uint64_t)blockDim.x + threadIdx.x;
    const unsigned mask = __ballot_sync(0xffffffffu, i < n);
    if (i >= n) return;
    unsigned status = 0;
    Work w;
    Jac3 JF;
    const float3 f = eval_path_grad<kCheckVisits, false>(s, mask, true, (int)depth, x + i, (uint32_t)n, JF, status, w);
    const int D = 2 + 2 * (int)depth;
    if (F) {
        F[i] = f.x;
        F[n + i] = f.y;
        F[2 * n + i] = f.z;
    }
    if (dF)
        for (int q = 0; q < 3; ++q)
            for (int d = 0; d < D; ++d) dF[((uint64_t)q * D + d) * n + i] = JF.c[q][d];
}

// One persistent launch over a batch of chain sets (scenes with different
// triangle counts, images and depths).  Blocks take work items -- a block of
// chains of one set -- from a global cursor; the host orders the items by
// estimated cost, so the longest items start first.  Every item runs all
// n_steps of Alg. 2 for its chains with the same code as step_kernel.
template <int kCheck>
__global__ void __launch_bounds__(256, 4) batch_step_kernel(const BatchEntry* entries, const BatchItem* items,
                                                         uint32_t n_items, unsigned int* cursor, uint32_t n_steps) {
    extern __shared__ float sh[];
    __shared__ unsigned int item_s;
    while (true) {
        if (threadIdx.x == 0) item_s = atomicAdd(cursor, 1u);
        __syncthreads();
        const unsigned it = item_s;
        __syncthreads();  // every thread has read item_s before it is overwritten
        if (it >= n_items) break;
        const BatchItem wi = items[it];
        const BatchEntry& e = entries[wi.set];  // descriptor fields are read where used
        const uint64_t i = wi.begin + threadIdx.x;
        chain_steps<kCheck, false, false, true>(e.s, e.c, i, i < wi.end, sh, e.step, n_steps, nullptr, nullptr, nullptr,
                                                nullptr);
        __syncthreads();  // the shared state buffers are reused by the next item
    }
}

// Fold every set's framebuffer into its accumulator; advance every set's step
// index by n_steps; reset the work cursor for the next launch.
__global__ void batch_fold_kernel(BatchEntry* entries, const uint64_t* px_off, uint32_t n_sets, uint64_t total_px,
                                  unsigned int* cursor, uint32_t n_steps) {
    const uint64_t j = blockIdx.x * (uint64_t)blockDim.x + threadIdx.x;
    if (j == 0) *cursor = 0u;
    if (j < n_sets) entries[j].step += n_steps;
    if (j >= total_px) return;
    uint32_t lo = 0, hi = n_sets;  // the set whose pixel range holds j
    while (hi - lo > 1) {
        const uint32_t mid = (lo + hi) / 2;
        if (px_off[mid] <= j) lo = mid;
        else hi = mid;
    }
    const uint64_t p = j - px_off[lo];
    float4* fb = entries[lo].c.fb;
    const float4 v = fb[p];
    if (v.x != 0.f || v.y != 0.f || v.z != 0.f || v.w != 0.f) {
        double4_32a* acc = entries[lo].c.acc64;
        double4_32a a = acc[p];
        a.x += v.x;
        a.y += v.y;
        a.z += v.z;
        a.w += v.w;
        acc[p] = a;
        fb[p] = make_float4(0.f, 0.f, 0.f, 0.f);
    }
}

// FP32 framebuffer -> FP64 accumulator, then clear (keeps long runs exact to
// FP64 while the hot loop does single 16-byte vector atomics).
__global__ void fold_kernel(float4* fb, double4_32a* acc, uint32_t n) {
    const uint32_t j = blockIdx.x * blockDim.x + threadIdx.x;
    if (j >= n) return;
    const float4 v = fb[j];
    if (v.x != 0.f || v.y != 0.f || v.z != 0.f || v.w != 0.f) {
        double4_32a a = acc[j];
        a.x += v.x;
        a.y += v.y;
        a.z += v.z;
        a.w += v.w;
        acc[j] = a;
        fb[j] = make_float4(0.f, 0.f, 0.f, 0.f);
    }
}

// image = accumulator / J (Section 6.3, normalisation-free estimator); MH
// (mh_samples > 0): image = b_hat accumulator / N, the ergodic average over the
// N post-burn-in iterations scaled by b_hat = mean p of the large-step proposals.
__global__ void resolve_kernel(const double4_32a* acc, const unsigned long long* counters, float* rgb, uint32_t n,
                               int mh, uint64_t mh_samples) {
    const uint32_t j = blockIdx.x * blockDim.x + threadIdx.x;
    if (j >= n) return;
    const unsigned long long J = counters[0];
    const double4_32a a = acc[j];
    double inv = J > 0 ? 1.0 / (double)J : 0.0;
    if (mh) {
        const double psum = __longlong_as_double((long long)counters[kCounterPSum]);
        inv = J > 0 && mh_samples > 0 ? psum / (double)J / (double)mh_samples : 0.0;
    }
    rgb[3 * j] = (float)(a.x * inv);
    rgb[3 * j + 1] = (float)(a.y * inv);
    rgb[3 * j + 2] = (float)(a.z * inv);
}

template <int kCheck>
__global__ void eval_states_kernel(SceneView s, uint32_t depth, float c_tilde, const float* x, uint64_t n, float* F,
                                   float* p, float* u, float* k, int32_t* ids, unsigned int* status_word) {
    const uint64_t i = blockIdx.x * (uint64_t)blockDim.x + threadIdx.x;
    const unsigned mask = __ballot_sync(0xffffffffu, i < n);
    if (i >= n) return;
    unsigned status = 0;
    const float3 f = eval_path<kCheck>(s, mask, true, (int)depth, x + i, (uint32_t)n, ids ? ids + i : nullptr, n, status);
    const float pp = lum(f);
    const float uu = 1.0f;
    if (F) {
        F[i] = f.x;
        F[n + i] = f.y;
        F[2 * n + i] = f.z;
    }
    if (p) p[i] = pp;
    if (u) u[i] = uu;
    if (k) k[i] = pp > 0.0f ? c_tilde * uu / pp : INFINITY;  // Section 6.2
    if (status && status_word) atomicOr(status_word, status);
}

// Plain path tracing by persistent warps (trace_paths).  Warp w of the grid traces
// samples [w n / warps, (w + 1) n / warps): no cursor in memory, so calls on
// several streams share nothing.  The coordinates are drawn where they are used (one Philox
// block per two vertices), so a path reads and writes nothing but its pixel.  Bound by
// the divergent traversal's L1/L2 latency and issue, as the chains' path kernel.
// Against one thread per path, whose warp waits for the longest ray of every vertex
// and for its longest path: 2 649 -> 1 182 us for 2 10^6 samples of Cornell + spheres,
// 10.26 -> 4.36 ms for 8 10^6.
struct PtPaths {
    static constexpr bool kFusedMirror = false;
    uint32_t W, H;
    int dep;
    uint64_t seed, next, end;  // next sample of the warp, end of its range
    double* accum;
    bool drained = false;
    uint64_t smp = 0;
    uint2 spare{};  // the second half of the path's latest block
    float3 F = f3(0.f, 0.f, 0.f);

    __device__ __forceinline__ uint4 block(uint32_t b) const {
        return draw(seed, kTagPt, b + 1u, (uint32_t)smp, smp >> 32);
    }
    __device__ __forceinline__ bool take(unsigned idle, bool mine, float& y0, float& y1) {
        const uint64_t j = next + __popc(idle & ((1u << (threadIdx.x & 31)) - 1u));
        next += __popc(idle);
        drained = next >= end;
        if (!mine || j >= end) return false;
        smp = j;
        F = f3(0.f, 0.f, 0.f);
        const uint4 r = block(0);
        spare = make_uint2(r.z, r.w);
        y0 = u01(r.x);
        y1 = u01(r.y);
        return true;
    }
    __device__ __forceinline__ const SceneView& camera(const SceneView& s) const { return s; }
    __device__ __forceinline__ int root(const SceneView& s) const { return s.root; }
    __device__ __forceinline__ int depth() const { return dep; }
    __device__ __forceinline__ float2 coords(int v) {  // coordinates 2 + 2v, 3 + 2v, in order of v
        if (!(v & 1)) return make_float2(u01(spare.x), u01(spare.y));
        const uint4 r = block((uint32_t)(1 + v) >> 1);
        spare = make_uint2(r.z, r.w);
        return make_float2(u01(r.x), u01(r.y));
    }
    __device__ __forceinline__ float3 emission() const { return F; }
    __device__ __forceinline__ void keep(float3 f) { F = f; }
    __device__ __forceinline__ void finish(float3 f, unsigned& status) {
        if (f.x == 0.f && f.y == 0.f && f.z == 0.f) return;
        f = finite_or_zero(f, status);
        const uint4 r = block(0);
        const uint32_t px = min((uint32_t)((double)u01(r.x) * (double)W), W - 1);
        const uint32_t py = min((uint32_t)((double)u01(r.y) * (double)H), H - 1);
        const double WH = (double)W * (double)H;
        double* a = accum + 4 * ((size_t)py * W + px);
        if (f.x != 0.f) atomicAdd(a, WH * f.x);
        if (f.y != 0.f) atomicAdd(a + 1, WH * f.y);
        if (f.z != 0.f) atomicAdd(a + 2, WH * f.z);
        // channel 3 is left to the caller: the sample count is n, known on the host
    }
    __device__ __forceinline__ void batch_done() const {}
};

template <int kCheck>
__global__ void __launch_bounds__(128, 7) render_pt_kernel(SceneView s, uint32_t W, uint32_t H, uint32_t depth,
                                                           uint64_t seed, uint64_t sample_begin, uint64_t n,
                                                           double* accum) {
    const uint64_t warps = (uint64_t)gridDim.x * (blockDim.x >> 5);
    const uint64_t w = (blockIdx.x * (uint64_t)blockDim.x + threadIdx.x) >> 5;
    const uint64_t per = n / warps, more = n % warps;  // the first `more` warps take one sample more
    const uint64_t first = sample_begin + w * per + min(w, more);
    PtPaths src{W, H, (int)depth, seed, first, first + per + (w < more ? 1 : 0), accum};
    unsigned status = 0;
    src.drained = src.next >= src.end;
    trace_paths<kCheck>(s, src, status);
}

// One thread per path.
template <int kCheck>
__global__ void render_pt_each_kernel(SceneView s, uint32_t W, uint32_t H, uint32_t depth, uint64_t seed,
                                      uint64_t sample_begin, uint64_t n, double* accum) {
    extern __shared__ float sh[];
    const uint32_t B = blockDim.x, tid = threadIdx.x;
    const uint64_t i = blockIdx.x * (uint64_t)B + tid;
    const unsigned mask = __ballot_sync(0xffffffffu, i < n);
    if (i >= n) return;
    const int D = 2 + 2 * (int)depth;
    float* y = sh + tid;
    const uint64_t smp = sample_begin + i;
    for (int b = 0; 4 * b < D; ++b) {
        const uint4 r = draw(seed, kTagPt, (uint32_t)(b + 1), (uint32_t)smp, smp >> 32);
        const uint32_t rr[4] = {r.x, r.y, r.z, r.w};
#pragma unroll
        for (int q = 0; q < 4; ++q)
            if (4 * b + q < D) y[(4 * b + q) * B] = u01(rr[q]);
    }
    unsigned status = 0;
    const float3 F = eval_path<kCheck, false>(s, mask, true, (int)depth, y, B, nullptr, 0, status);
    uint32_t px = min((uint32_t)((double)y[0] * (double)W), W - 1);
    uint32_t py = min((uint32_t)((double)y[B] * (double)H), H - 1);
    const double WH = (double)W * (double)H;
    double* a = accum + 4 * ((size_t)py * W + px);
    if (F.x != 0.f) atomicAdd(a, WH * F.x);
    if (F.y != 0.f) atomicAdd(a + 1, WH * F.y);
    if (F.z != 0.f) atomicAdd(a + 2, WH * F.z);
}

__global__ void philox_kernel(uint64_t seed, uint32_t tag, uint32_t block, uint64_t chain_begin, uint64_t step,
                              uint64_t n, uint32_t* out) {
    const uint64_t i = blockIdx.x * (uint64_t)blockDim.x + threadIdx.x;
    if (i >= n) return;
    const uint4 r = draw(seed, tag, block, (uint32_t)(chain_begin + i), step);
    reinterpret_cast<uint4*>(out)[i] = r;
}

// FP32 peak: every thread runs kChainsFma independent FMA chains for `iters`
// rounds (2 FLOP per FMA), so the FMA pipes never wait on a dependency; the
// values stay finite (a contraction towards 1) and are written out only if a
// condition that never holds is met, so nothing is optimised away.
constexpr int kChainsFma = 8;
__global__ void __launch_bounds__(256) fma_peak_kernel(uint32_t iters, float* sink) {
    float a[kChainsFma];
    const float m = 0.999f, c = 1e-3f * (float)(threadIdx.x & 7);
#pragma unroll
    for (int k = 0; k < kChainsFma; ++k) a[k] = 1.0f + 1e-3f * (float)k;
    for (uint32_t it = 0; it < iters; ++it) {
#pragma unroll
        for (int r = 0; r < 16; ++r) {
#pragma unroll
            for (int k = 0; k < kChainsFma; ++k) a[k] = fmaf(a[k], m, c);
        }
    }
    float s = 0.f;
#pragma unroll
    for (int k = 0; k < kChainsFma; ++k) s += a[k];
    if (s == -1.0f && sink) sink[blockIdx.x * blockDim.x + threadIdx.x] = s;
}

inline unsigned grid_for(uint64_t n, unsigned b) { return (unsigned)((n + b - 1) / b); }

// Chains per warp for a kernel that gives each one-warp block that many chains:
// the fewest with which `most` warps per SM hold them all, or 0 where the
// device cannot hold them all at once even in full warps: there the launch is
// bound by throughput, which full warps have the most of.  kSpreadWarps: three
// warps per scheduler; more of them, with fewer chains each, wait for one another
// (10 007 chains, 32 steps of Cornell + spheres: 1 702 us at 8, 1 578 at 12,
// 1 600 at 16; 30 000 chains, 16 steps: 1 431, 1 357, 1 375 us; 6 000 chains in the
// 24-triangle box, 64 steps: 785, 842, 892 us).
// kSpreadWarpsSmall: scenes of at most kWarpChainMaxTris triangles, whose rays are short
// and alike, so that the lanes of a warp hardly wait for one another: two warps per
// scheduler (10 steps of 5 000 and 12 000 chains, 8 / 12 warps: 24-triangle box, depth 6,
// 218, 219 and 250, 261 us; 100 boxes in a room 361, 361 and 444, 455; the furnace, depth
// 8, where the lanes never part, 194, 220 and 203, 221, and in blocks of 128 198 and 199).
//
// MALA: a step's gradient keeps four 3 x D Jacobians per lane in local memory, whose
// lines a warp with few lanes fills with as few of its chains (1536 D bytes a warp, beside
// 512 D of shared memory).  So the warps per SM are as many as their lines fit L1 with:
// 4, or 3 beyond D = 24; and the launch asks for no more shared memory than they take
// (left alone, the split is made for 16 of them, and L1 has 28 to 90 of its 256 KB).  Gain
// over one thread per chain in blocks of 128 (in brackets 12 warps per SM, in scenes of at
// most 128 triangles 4, without the request), 2 500 and 10 000 chains: Cornell + spheres,
// depth 8, 2.3, 1.7 (1.8, 1.2), depth 15 3.0, 2.0 (1.5, 1.2); 180 000-triangle terrain 2.2, 1.7
// (1.4, 1.2); glass furnace, depth 12, 2.4, 1.9 (1.2, 0.98); 24-triangle box, depth 15, 3.2, 2.4
// (1.1, 1.0); furnace, depth 8, 1.5, 1.4 (0.76, 0.75).  Up to kCarveWarps one-warp blocks
// per SM the request still pays (30 000 chains 1.2, 1.05); beyond it costs.
constexpr int kSpreadWarps = 12, kSpreadWarpsSmall = 8, kSpreadWarpsMala = 4, kSpreadWarpsMalaDeep = 3, kCarveWarps = 12;
template <class K>
cudaError_t chains_per_warp(K kernel, size_t shm, uint64_t n, int most, unsigned* per_warp, long long* sm_count = nullptr) {
    static DeviceOnce once;  // per device: its SM count
    long long sms = 0;
    cudaError_t e = once.get(
        [](int dev, long long* v) {
            int n = 0;
            const cudaError_t r = cudaDeviceGetAttribute(&n, cudaDevAttrMultiProcessorCount, dev);
            *v = n;
            return r;
        },
        &sms);
    int per_sm = 0;
    if (e == cudaSuccess) e = cudaOccupancyMaxActiveBlocksPerMultiprocessor(&per_sm, kernel, 32, shm);
    if (e != cudaSuccess) return e;
    const uint64_t warps = (uint64_t)sms * (uint64_t)std::min(per_sm, most);
    const bool fits = per_sm > 0 && n <= 32 * (uint64_t)sms * (uint64_t)per_sm;
    *per_warp = fits ? (unsigned)std::min<uint64_t>(32, (n + warps - 1) / warps) : 0u;
    if (sm_count) *sm_count = sms;
    return cudaSuccess;
}

// A kernel as a type, so that a generic launcher has one set of statics per kernel.
template <auto K>
struct Kernel {
    static constexpr auto value = K;
};

}  // namespace

cudaError_t measure_fma_peak(double* tflops, double* ms_out, cudaStream_t st) {
    int dev = 0, sms = 0, per_sm = 0;
    cudaError_t e;
    if ((e = cudaGetDevice(&dev)) != cudaSuccess ||
        (e = cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, dev)) != cudaSuccess ||
        (e = cudaOccupancyMaxActiveBlocksPerMultiprocessor(&per_sm, fma_peak_kernel, 256, 0)) != cudaSuccess)
        return e;
    const unsigned grid = (unsigned)(sms * (per_sm > 0 ? per_sm : 1));
    const uint32_t iters = 1u << 14;
    cudaEvent_t e0 = nullptr, e1 = nullptr;
    if ((e = cudaEventCreate(&e0)) != cudaSuccess) return e;
    if ((e = cudaEventCreate(&e1)) != cudaSuccess) {
        cudaEventDestroy(e0);
        return e;
    }
    float best = 0.f;
    for (int rep = 0; rep < 4 && e == cudaSuccess; ++rep) {  // the first launch warms up
        fma_peak_kernel<<<grid, 256, 0, st>>>(iters, nullptr);
        if ((e = cudaEventRecord(e0, st)) != cudaSuccess) break;
        fma_peak_kernel<<<grid, 256, 0, st>>>(iters, nullptr);
        if ((e = cudaEventRecord(e1, st)) != cudaSuccess || (e = cudaEventSynchronize(e1)) != cudaSuccess) break;
        float t = 0.f;
        if ((e = cudaEventElapsedTime(&t, e0, e1)) != cudaSuccess) break;
        if (rep == 0 || t < best) best = t;
    }
    if (e == cudaSuccess) e = cudaGetLastError();
    cudaEventDestroy(e0);
    cudaEventDestroy(e1);
    if (e != cudaSuccess) return e;
    const double flop = 2.0 * (double)grid * 256.0 * (double)iters * 16.0 * kChainsFma;
    *tflops = flop / (best * 1e-3) / 1e12;
    if (ms_out) *ms_out = best;
    return cudaSuccess;
}

cudaError_t launch_init(const SceneView& s, const ChainView& c, cudaStream_t st) {
    const unsigned B = 128;
    with_checks(trav_checks(s), [&](auto k) {
        init_kernel<k()><<<grid_for(c.n, B), B, sizeof(float) * c.dim * B, st>>>(s, c);
    });
    return cudaGetLastError();
}

cudaError_t launch_reeval(const SceneView& s, const ChainView& c, cudaStream_t st) {
    const unsigned B = 128;
    reeval_kernel<<<grid_for(c.n, B), B, sizeof(float) * c.dim * B, st>>>(s, c);
    return cudaGetLastError();
}

cudaError_t launch_step_warp(const SceneView& s, const ChainView& c, uint64_t step_begin, uint32_t n_steps,
                             cudaStream_t st) {
    if (c.n == 0 || n_steps == 0) return cudaSuccess;
    const uint64_t threads = 32 * c.n;
    step_kernel_warp<<<grid_for(threads, kWarpChainThreads), kWarpChainThreads, 0, st>>>(s, c, step_begin, n_steps);
    return cudaGetLastError();
}

cudaError_t launch_step(const SceneView& s, const ChainView& c, uint64_t step_begin, uint32_t n_steps,
                        uint8_t* tr_flags, float* tr_dt, int32_t* tr_pix, unsigned long long* work_out, int block,
                        cudaStream_t st) {
    const unsigned B = (unsigned)block;
    const size_t shm = sizeof(float) * 2 * c.dim * B;  // <= 2 * 32 * 256 * 4 = 64 KB
    const unsigned G = grid_for(c.n, B);
    const auto run = [&](auto kernel, uint8_t* f, float* dt, int32_t* pix, unsigned long long* work) {
        static DeviceOnce once;  // per device and variant: opt in to > 48 KB of dynamic shared memory
        const cudaError_t e = once.get(
            [&](int, long long*) {
                return cudaFuncSetAttribute(kernel.value, cudaFuncAttributeMaxDynamicSharedMemorySize,
                                            (int)(sizeof(float) * 2 * kMaxDim * 256));
            },
            nullptr);
        if (e != cudaSuccess) return e;
        kernel.value<<<G, B, shm, st>>>(s, c, step_begin, n_steps, f, dt, pix, work);
        return cudaGetLastError();
    };
    cudaError_t e = cudaSuccess;
    if (work_out || tr_flags || tr_dt || tr_pix) {  // both watchdogs checked, or neither
        with_checks(trav_checks(s) == kCheckNone ? kCheckNone : kCheckAll, [&](auto k) {
            if constexpr (k() != kCheckVisits)
                e = work_out ? run(Kernel<step_kernel<k(), false, true>>{}, nullptr, nullptr, nullptr, work_out)
                             : run(Kernel<step_kernel<k(), true, false>>{}, tr_flags, tr_dt, tr_pix, nullptr);
        });
        return e;
    }
    with_checks(trav_checks(s), [&](auto k) {
        const auto spread = step_kernel_spread<decltype(k)::value>;
        const size_t wshm = sizeof(float) * 2 * c.dim * 32;  // <= 8 KB
        unsigned per_warp = 0;
        if ((e = chains_per_warp(spread, wshm, c.n,
                                 s.n_tris <= kWarpChainMaxTris ? kSpreadWarpsSmall : kSpreadWarps, &per_warp)) != cudaSuccess) return;
        if (per_warp) {
            spread<<<grid_for(c.n, per_warp), 32, wshm, st>>>(s, c, step_begin, n_steps, per_warp);
            e = cudaGetLastError();
        } else {
            e = run(Kernel<step_kernel<k(), false, false>>{}, nullptr, nullptr, nullptr, nullptr);
        }
    });
    return e;
}

cudaError_t launch_drain(const SceneView& s, const ChainView& c, uint64_t step_begin, uint32_t n_steps,
                         unsigned long long* ctl, cudaStream_t st) {
    const size_t shm = sizeof(float) * 2 * c.dim * 32;  // <= 8 KB
    cudaError_t e = cudaMemsetAsync(ctl, 0, 2 * sizeof(unsigned long long), st);
    if (e != cudaSuccess) return e;
    with_checks(trav_checks(s), [&](auto k) {
        static DeviceOnce once;  // per device and variant: its SM count
        const auto kernel = drain_kernel<decltype(k)::value>;
        long long sms = 0;
        e = once.get(
            [](int dev, long long* v) {
                int n = 0;
                const cudaError_t r = cudaDeviceGetAttribute(&n, cudaDevAttrMultiProcessorCount, dev);
                *v = n;
                return r;
            },
            &sms);
        int per_sm = 0;
        if (e == cudaSuccess) e = cudaOccupancyMaxActiveBlocksPerMultiprocessor(&per_sm, kernel, 32, shm);
        if (e != cudaSuccess) return;
        const uint64_t blocks = std::min<uint64_t>((uint64_t)sms * (per_sm > 0 ? per_sm : 1), (c.n + 31) / 32);
        kernel<<<(unsigned)blocks, 32, shm, st>>>(s, c, step_begin, n_steps, ctl);
        e = cudaGetLastError();
    });
    return e;
}

cudaError_t launch_step_mala(const SceneView& s, const ChainView& c, uint64_t step_begin, uint32_t n_steps,
                             uint8_t* tr_flags, float* tr_dt, int32_t* tr_pix, cudaStream_t st) {
    const size_t shm = sizeof(float) * 4 * c.dim * 32;  // <= 16 KB
    const auto run = [&](auto kernel) {
        unsigned per_warp = 0;
        long long sms = 0;
        const cudaError_t e = chains_per_warp(kernel, shm, c.n, c.dim <= 24 ? kSpreadWarpsMala : kSpreadWarpsMalaDeep,
                                              &per_warp, &sms);
        if (e != cudaSuccess) return e;
        if (per_warp == 0) per_warp = 32;
        cudaLaunchConfig_t cfg{};
        cfg.gridDim = dim3(grid_for(c.n, per_warp));
        cfg.blockDim = dim3(32);
        cfg.dynamicSmemBytes = shm;
        cfg.stream = st;
        cudaLaunchAttribute carve;
        const long long warps = (cfg.gridDim.x + sms - 1) / sms;
        if (warps <= kCarveWarps) {  // percent of the SM's 228 KB; a block takes 1 KB beside its own
            carve.id = cudaLaunchAttributePreferredSharedMemoryCarveout;
            carve.val.sharedMemCarveout = (unsigned)std::min<size_t>(100, 100 * warps * (shm + 1024) / (228 * 1024) + 1);
            cfg.attrs = &carve;
            cfg.numAttrs = 1;
        }
        return cudaLaunchKernelEx(&cfg, kernel, s, c, step_begin, n_steps, (uint32_t)per_warp, tr_flags, tr_dt, tr_pix);
    };
    if (tr_flags || tr_dt || tr_pix) return run(step_kernel_mala<kCheckAll, true>);
    cudaError_t e = cudaSuccess;
    with_checks(trav_checks(s), [&](auto k) { e = run(step_kernel_mala<decltype(k)::value, false>); });
    return e;
}

cudaError_t launch_mala_reeval(const SceneView& s, const ChainView& c, cudaStream_t st) {
    mala_reeval_kernel<<<grid_for(c.n, 128), 128, sizeof(float) * c.dim * 128, st>>>(s, c);
    return cudaGetLastError();
}

cudaError_t launch_eval_grad(const SceneView& s, uint32_t depth, const float* x, uint64_t n, float* F, float* dF,
                             cudaStream_t st) {
    if (n == 0) return cudaSuccess;
    eval_grad_kernel<<<grid_for(n, 128), 128, 0, st>>>(s, depth, x, n, F, dF);
    return cudaGetLastError();
}

cudaError_t launch_fold(const ChainView& c, cudaStream_t st) {
    const uint32_t n = c.width * c.height;
    fold_kernel<<<grid_for(n, 256), 256, 0, st>>>(c.fb, c.acc64, n);
    return cudaGetLastError();
}

cudaError_t launch_batch(BatchEntry* entries, const BatchItem* items, uint32_t n_items, const uint64_t* px_off,
                         uint32_t n_sets, uint64_t total_px, unsigned int* cursor, uint32_t max_dim, int block,
                         int checks, uint32_t n_steps, cudaStream_t st) {
    const size_t shm = sizeof(float) * 2 * max_dim * (size_t)block;
    const auto run = [&](auto kernel) {
        static DeviceOnce once;  // per device and variant: the SM count, after the shared-memory opt-in
        long long sms = 0;
        cudaError_t e = once.get(
            [&](int dev, long long* v) {
                int n = 0;
                cudaError_t r;
                if ((r = cudaDeviceGetAttribute(&n, cudaDevAttrMultiProcessorCount, dev)) != cudaSuccess ||
                    (r = cudaFuncSetAttribute(kernel.value, cudaFuncAttributeMaxDynamicSharedMemorySize,
                                              (int)(sizeof(float) * 2 * kMaxDim * 256))) != cudaSuccess)
                    return r;
                *v = n;
                return cudaSuccess;
            },
            &sms);
        if (e != cudaSuccess) return e;
        int per_sm = 0;
        if ((e = cudaOccupancyMaxActiveBlocksPerMultiprocessor(&per_sm, kernel.value, block, shm)) != cudaSuccess)
            return e;
        const unsigned grid = (unsigned)std::min<uint64_t>((uint64_t)sms * (per_sm > 0 ? per_sm : 1), n_items);
        if (n_steps > 0 && n_items > 0)
            kernel.value<<<grid, block, shm, st>>>(entries, items, n_items, cursor, n_steps);
        return cudaSuccess;
    };
    cudaError_t e = cudaSuccess;
    with_checks(checks, [&](auto k) { e = run(Kernel<batch_step_kernel<k()>>{}); });
    if (e != cudaSuccess) return e;
    const uint64_t total = total_px > n_sets ? total_px : n_sets;
    batch_fold_kernel<<<grid_for(total, 256), 256, 0, st>>>(entries, px_off, n_sets, total_px, cursor, n_steps);
    return cudaGetLastError();
}

cudaError_t launch_resolve(const ChainView& c, float* rgb, uint64_t mh_samples, cudaStream_t st) {
    const uint32_t n = c.width * c.height;
    resolve_kernel<<<grid_for(n, 256), 256, 0, st>>>(c.acc64, c.counters, rgb, n, (c.flags & JR_FLAG_MH) != 0,
                                                     mh_samples);
    return cudaGetLastError();
}

cudaError_t launch_eval_states(const SceneView& s, uint32_t depth, float c_tilde, const float* x, uint64_t n,
                               float* F, float* p, float* u, float* k, int32_t* ids, cudaStream_t st) {
    if (n == 0) return cudaSuccess;
    with_checks(trav_checks(s), [&](auto kc) {
        eval_states_kernel<kc()><<<grid_for(n, 128), 128, 0, st>>>(s, depth, c_tilde, x, n, F, p, u, k, ids, nullptr);
    });
    return cudaGetLastError();
}

// Small calls keep one thread per path: the persistent warps' tail is then most of the
// launch.  One thread per path / persistent, us, at 100 000, 160 000, 262 144 and 2 10^6 samples:
//   Cornell + spheres, depth 8   219, 204   313, 220   429, 305   2 649, 1 182
//   slit caustic, depth 10       186, 195   200, 200   272, 231   1 383,   602
//   2M-triangle terrain          180, 194   209, 206   282, 241   1 564,   892
//   5 000 boxes, depth 8         191, 226   272, 279   374, 358   2 386, 2 063
// In scenes of a few triangles rays are short and alike, so that a warp waits for
// nobody unless some of its paths leave the scene early and the others go on for long
// (24-triangle box, depth 2: 54, 63 at 200 000, 318, 327 at 2 10^6; depth 4: 78, 83; 508, 433;
// depth 8: 118, 109; 835, 541).  Where no path can leave (100 boxes in a room, depth 6: 211,
// 243 at 262 144, 1 318, 1 398 at 2 10^6; the 12-triangle furnace, depth 8: 79, 94; 435, 526) the
// persistent warps only cost.
constexpr uint64_t kRenderPersistentMin = 5u << 15, kRenderPersistentMinSmall = 1u << 18;
constexpr uint32_t kRenderSmallDepth = 4;

cudaError_t launch_render_pt(const SceneView& s, uint32_t width, uint32_t height, uint32_t depth, uint64_t seed,
                             uint64_t sample_begin, uint64_t n, double* accum, cudaStream_t st) {
    if (n == 0) return cudaSuccess;
    cudaError_t e = cudaSuccess;
    const bool small = s.n_tris <= kWarpChainMaxTris;
    const bool each = small ? s.closed || n < kRenderPersistentMinSmall || depth < kRenderSmallDepth
                            : n < kRenderPersistentMin;
    with_checks(trav_checks(s), [&](auto k) {
        if (each) {
            const size_t shm = sizeof(float) * (2 + 2 * depth) * 128;
            render_pt_each_kernel<k()><<<grid_for(n, 128), 128, shm, st>>>(s, width, height, depth, seed, sample_begin,
                                                                           n, accum);
            e = cudaGetLastError();
            return;
        }
        static DeviceOnce once;  // per device and variant: the persistent grid
        const auto kernel = render_pt_kernel<decltype(k)::value>;
        long long blocks = 0;
        e = once.get(
            [&](int dev, long long* v) {
                int sms = 0, per_sm = 0;
                cudaError_t r;
                if ((r = cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, dev)) != cudaSuccess ||
                    (r = cudaOccupancyMaxActiveBlocksPerMultiprocessor(&per_sm, kernel, 128, 0)) != cudaSuccess)
                    return r;
                *v = (long long)sms * (per_sm > 0 ? per_sm : 1);
                return cudaSuccess;
            },
            &blocks);
        if (e != cudaSuccess) return;
        const uint64_t want = (n + 255) / 256;  // two samples per lane: a warp that refills hides its longest path
        kernel<<<(unsigned)std::min<uint64_t>((uint64_t)blocks, want), 128, 0, st>>>(s, width, height, depth, seed,
                                                                                    sample_begin, n, accum);
        e = cudaGetLastError();
    });
    return e;
}

cudaError_t launch_philox(uint64_t seed, uint32_t tag, uint32_t block, uint64_t chain_begin, uint64_t step,
                          uint64_t n, uint32_t* out, cudaStream_t st) {
    if (n == 0) return cudaSuccess;
    philox_kernel<<<grid_for(n, 256), 256, 0, st>>>(seed, tag, block, chain_begin, step, n, out);
    return cudaGetLastError();
}

}  // namespace jr
