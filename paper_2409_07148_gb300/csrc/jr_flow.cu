// The learned regeneration flow on the tensor cores (sm_103a).
//
// Not in the paper: the library's own regeneration distribution
//   mu = beta mu_flow + (1 - beta) uniform,   u = beta q + (1 - beta),
// so the killing rate k = c~ u / p (Section 6.2) keeps an exact density.  The
// flow has L coupling layers on [0,1)^D; layer l conditions on x[perm[l][:A]]
// (A = D/2) and moves each x[perm[l][A + j]] through a piecewise-linear CDF of
// K bins whose masses come from an MLP (2 hidden layers of 64, ReLU):
//   Q_j = (1 - E) softmax(o_j) + E / K,  density factor K Q_j[bin],
// the piecewise-linear coupling of Mueller et al. ("Neural Importance
// Sampling", 2019).  The MLP GEMMs run as mma.sync m16n8k16 with bf16
// operands and FP32 accumulation; everything else is FP32.
//
// This file holds the training side (forward with stored layer inputs,
// backward, Adam, parameter packing, training rows from the chains); the
// inference kernels are in jr_flow_infer.cu.
#include <cuda_bf16.h>
#include <cuda_runtime.h>
#include <stdint.h>

#include "../../include/jr.h"
#include "jr_device.cuh"
#include "jr_internal.h"

namespace jr {
namespace {

// ---------------------------------------------------------------------------
// Training: the time-weighted maximum-likelihood loss  -sum_r w_r log q(x_r) /
// sum_r w_r  over a minibatch and its gradient w.r.t. the FP32 master
// parameters.  Per tile of 64 rows: a forward pass (density direction) stores
// the state entering every layer; the backward pass goes through the layers in
// reverse, recomputes the layer's MLP from the stored state, and back-propagates
// through the couplings (FP32) and the MLP (tensor cores: activation gradients
// dO W3, dh2 W2, dh1 W1 and weight gradients dO^T h2, dh2^T h1, dh1^T xa, all
// bf16 operands with FP32 accumulation; bf16 roundings of the forward pass
// pass gradients straight through).  Weight gradients go to an FP32 buffer
// with atomics.
//
// A minibatch of 8 192 rows is 128 tiles, less than one per SM, and a tile is a
// serial chain of 12 layer passes of small GEMMs: the kernel is bound by the
// latency of that chain, not by the tensor cores (25 steps of 8 192 rows at D =
// 22 cost 64 us of them).  So a tile takes 16 warps, 4 row groups x 4 column
// groups: warp (wr, wc) owns rows 16 wr .. 16 wr + 15 and every fourth 16-column
// block, and the (row, coordinate) pairs of the softmax spread over 512 lanes.
// Fragments come by ldmatrix (.trans for the transposed operands), gradients
// leave as 8-byte vector atomics, and the next layer's weights arrive by
// cp.async in the buffers that the present layer is done with.  Measured against
// 4 warps per tile with scalar fragment loads, and a weight-sum, a memset and a
// packing launch per step besides Adam's: 204 -> 98 us per Adam step of 8 192 rows
// at D = 22, 124 -> 65 us at D = 8, 117 -> 58 us for 512 rows at D = 6.

constexpr int kRows = 64;          // rows per tile
constexpr int kTrainThreads = 512;
constexpr int kXs = 33;            // row stride of the state tile (floats)
constexpr int kLs = 36;            // row stride of a warp's logits tile (floats): two coordinates
constexpr int kSO = kFMaxAK + 8;   // row stride of the logits-gradient tile (bf16)

struct TrainSmem {
    float x[kRows * kXs];
    float g[kRows * kXs];           // dL/d(state)
    float stash[kFL][kRows * kXs];  // state entering each layer
    union {  // the logits are done with before dh2 and dh1 are written, and the other way round
        float lg[kTrainThreads / 32][16 * kLs];
        struct {
            __nv_bfloat16 dh2[kRows * kFS2], dh1[kRows * kFS2];
        };
    };
    uint8_t perm[kFL * kMaxDim];
    float lq[4][kRows];             // log q per row, one part per column group
    float s[kRows];                 // dL/d(log q) per row
    float b1[2][kFH], b2[kFH], b3[kFMaxAK];
    __nv_bfloat16 xa[kRows * kFS1];
    __nv_bfloat16 h1[kRows * kFS2];
    __nv_bfloat16 h2[kRows * kFS2];
    __nv_bfloat16 dO[kRows * kSO];  // dL/d(logits)
    __nv_bfloat16 w1[2][kFH * kFS1];
    __nv_bfloat16 w2[kFH * kFS2];
    __nv_bfloat16 w3[kFMaxAK * kFS2];
};
static_assert(sizeof(TrainSmem) <= 227 * 1024, "one training tile per SM");
static_assert(kFS1 % 8 == 0 && kFS2 % 8 == 0 && kSO % 8 == 0, "ldmatrix rows start on 16 bytes");

// D[16x8] += A[16x16] (row-major) * B[16x8] (col-major), bf16 in, FP32 accumulate.
__device__ __forceinline__ void mma_bf16(float (&d)[4], const uint32_t (&a)[4], uint32_t b0, uint32_t b1) {
    asm volatile(
        "mma.sync.aligned.m16n8k16.row.col.f32.bf16.bf16.f32 {%0,%1,%2,%3}, {%4,%5,%6,%7}, {%8,%9}, "
        "{%0,%1,%2,%3};\n"
        : "+f"(d[0]), "+f"(d[1]), "+f"(d[2]), "+f"(d[3])
        : "r"(a[0]), "r"(a[1]), "r"(a[2]), "r"(a[3]), "r"(b0), "r"(b1));
}
__device__ __forceinline__ uint32_t smem_at(const void* p) { return (uint32_t)__cvta_generic_to_shared(p); }
__device__ __forceinline__ void ldsm(const __nv_bfloat16* p, uint32_t (&r)[4]) {
    asm volatile("ldmatrix.sync.aligned.m8n8.x4.shared.b16 {%0,%1,%2,%3}, [%4];"
                 : "=r"(r[0]), "=r"(r[1]), "=r"(r[2]), "=r"(r[3])
                 : "r"(smem_at(p)));
}
__device__ __forceinline__ void ldsm_t(const __nv_bfloat16* p, uint32_t (&r)[4]) {
    asm volatile("ldmatrix.sync.aligned.m8n8.x4.trans.shared.b16 {%0,%1,%2,%3}, [%4];"
                 : "=r"(r[0]), "=r"(r[1]), "=r"(r[2]), "=r"(r[3])
                 : "r"(smem_at(p)));
}

// acc[16 x 16] = A B over K (a multiple of 16), for the warp's 16 x 16 block at
// (m0, n0).  A is A[m * sa + k], or with kTA A[k * sa + m]; B is B[n * sb + k]
// (a weight matrix [out][in] applied forwards), or with kTB B[k * sb + n].
template <bool kTA, bool kTB>
__device__ __forceinline__ void gemm16(float (&acc)[2][4], const __nv_bfloat16* A, int sa, int m0,
                                       const __nv_bfloat16* B, int sb, int n0, int K) {
    const int lane = threadIdx.x & 31, r = lane & 7, q = lane >> 3;
    const __nv_bfloat16* pa = kTA ? A + (size_t)(r + (q >> 1) * 8) * sa + m0 + (q & 1) * 8
                                  : A + (size_t)(m0 + r + (q & 1) * 8) * sa + (q >> 1) * 8;
    const __nv_bfloat16* pb = kTB ? B + (size_t)(r + (q & 1) * 8) * sb + n0 + (q >> 1) * 8
                                  : B + (size_t)(n0 + r + (q >> 1) * 8) * sb + (q & 1) * 8;
#pragma unroll
    for (int h = 0; h < 2; ++h) acc[h][0] = acc[h][1] = acc[h][2] = acc[h][3] = 0.f;
#pragma unroll 4
    for (int k0 = 0; k0 < K; k0 += 16) {
        uint32_t a[4], b[4];
        if constexpr (kTA) ldsm_t(pa + (size_t)k0 * sa, a);
        else ldsm(pa + k0, a);
        if constexpr (kTB) ldsm_t(pb + (size_t)k0 * sb, b);
        else ldsm(pb + k0, b);
        mma_bf16(acc[0], a, b[0], b[1]);
        mma_bf16(acc[1], a, b[2], b[3]);
    }
}

// The block's 2 x 2 pieces (row g or g + 8, column pair 2t of n-tile h) as bf16
// pairs: f(h, column, lower half?, value 0, value 1) -> stored pair.
template <class F>
__device__ __forceinline__ void store_bf16(__nv_bfloat16* out, int ld, int m0, int n0, const float (&acc)[2][4], F&& f) {
    const int lane = threadIdx.x & 31, g = lane >> 2, t = lane & 3;
#pragma unroll
    for (int h = 0; h < 2; ++h)
#pragma unroll
        for (int lo = 0; lo < 2; ++lo) {
            const int row = m0 + g + 8 * lo, col = n0 + 8 * h + 2 * t;
            *reinterpret_cast<__nv_bfloat162*>(out + row * ld + col) =
                f(row, col, acc[h][2 * lo], acc[h][2 * lo + 1]);
        }
}

// Add a 16 x 16 block of a weight gradient to grad (row stride ld).
__device__ __forceinline__ void add_grad(float* grad, int ld, int m0, int n0, const float (&acc)[2][4]) {
    const int lane = threadIdx.x & 31, g = lane >> 2, t = lane & 3;
#pragma unroll
    for (int h = 0; h < 2; ++h) {
        float* p = grad + (size_t)(m0 + g) * ld + n0 + 8 * h + 2 * t;
        atomicAdd(reinterpret_cast<float2*>(p), make_float2(acc[h][0], acc[h][1]));
        atomicAdd(reinterpret_cast<float2*>(p + 8 * ld), make_float2(acc[h][2], acc[h][3]));
    }
}

// Column sums over rows [r0, r0 + n) of the column pair `cp` of m, added to out.
__device__ __forceinline__ void add_column_sums(float* out, const __nv_bfloat16* m, int ld, int cp, int r0, int n) {
    float s0 = 0.f, s1 = 0.f;
    for (int r = r0; r < r0 + n; ++r) {
        const float2 v = __bfloat1622float2(*reinterpret_cast<const __nv_bfloat162*>(m + r * ld + 2 * cp));
        s0 += v.x;
        s1 += v.y;
    }
    atomicAdd(reinterpret_cast<float2*>(out + 2 * cp), make_float2(s0, s1));
}

// Start copying n bytes (a multiple of 16) to shared memory, all threads of the tile.
__device__ __forceinline__ void copy_async(void* dst, const void* src, int n) {
    for (int e = threadIdx.x * 16; e < n; e += kTrainThreads * 16)
        asm volatile("cp.async.cg.shared.global [%0], [%1], 16;" ::"r"(smem_at(dst) + e),
                     "l"(static_cast<const char*>(src) + e)
                     : "memory");
}
__device__ __forceinline__ void copy_commit() { asm volatile("cp.async.commit_group;" ::: "memory"); }
template <int kPending>
__device__ __forceinline__ void copy_wait() {
    asm volatile("cp.async.wait_group %0;" ::"n"(kPending) : "memory");
}

__device__ __forceinline__ const __nv_bfloat16* layer_w(const FlowView& f, int l) {
    return f.wb + (size_t)l * (kFH * kFS1 + kFH * kFS2 + (size_t)f.AK * kFS2);
}
__device__ __forceinline__ const float* layer_b(const FlowView& f, int l) {
    return f.bias + (size_t)l * (2 * kFH + f.AK);
}
// Layer l's matrix 1, 2 or 3 with its bias, as one copy group.  Matrix 1 has two
// buffers (layer l in l & 1), the others one.
__device__ __forceinline__ void fetch_w1(const FlowView& f, int l, TrainSmem& sm) {
    copy_async(sm.w1[l & 1], layer_w(f, l), 2 * kFH * kFS1);
    copy_async(sm.b1[l & 1], layer_b(f, l), 4 * kFH);
    copy_commit();
}
__device__ __forceinline__ void fetch_w2(const FlowView& f, int l, TrainSmem& sm) {
    copy_async(sm.w2, layer_w(f, l) + kFH * kFS1, 2 * kFH * kFS2);
    copy_async(sm.b2, layer_b(f, l) + kFH, 4 * kFH);
    copy_commit();
}
__device__ __forceinline__ void fetch_w3(const FlowView& f, int l, TrainSmem& sm) {
    copy_async(sm.w3, layer_w(f, l) + kFH * kFS1 + kFH * kFS2, 2 * (int)f.AK * kFS2);
    copy_async(sm.b3, layer_b(f, l) + 2 * kFH, 4 * (int)f.AK);
    copy_commit();
}

// Offsets of the parameters of one layer in the master layout.
__device__ __forceinline__ size_t off_b1() { return (size_t)kFH * kFAP; }
__device__ __forceinline__ size_t off_w2() { return off_b1() + kFH; }
__device__ __forceinline__ size_t off_b2() { return off_w2() + kFH * kFH; }
__device__ __forceinline__ size_t off_w3() { return off_b2() + kFH; }
__device__ __forceinline__ size_t off_b3(uint32_t AK) { return off_w3() + (size_t)AK * kFH; }

// The conditioning coordinates of the tile as bf16 (zero-padded to kFAP).
__device__ __forceinline__ void load_xa(const uint8_t* pm, int A, TrainSmem& sm) {
    for (int e = threadIdx.x; e < kRows * kFAP; e += kTrainThreads) {
        const int r = e / kFAP, c = e % kFAP;
        sm.xa[r * kFS1 + c] = __float2bfloat16_rn(c < A ? sm.x[r * kXs + pm[c]] : 0.0f);
    }
}
// One hidden layer of the warp's block: out = relu(W in + b).
__device__ __forceinline__ void hidden(__nv_bfloat16* out, const __nv_bfloat16* in, int sin, const __nv_bfloat16* W,
                                       int sw, const float* bias, int K, int m0, int n0) {
    float acc[2][4];
    gemm16<false, false>(acc, in, sin, m0, W, sw, n0, K);
    store_bf16(out, kFS2, m0, n0, acc, [&](int, int c, float a, float b) {
        return __floats2bfloat162_rn(fmaxf(a + bias[c], 0.f), fmaxf(b + bias[c + 1], 0.f));
    });
}
// The biased logits of coordinates j and j + 1 (if below A) for the warp's rows
// into its tile lg [16][kLs].
__device__ __forceinline__ void logits_pair(float* lg, int j, int A, int m0, const TrainSmem& sm) {
    const int lane = threadIdx.x & 31, g = lane >> 2, t = lane & 3;
#pragma unroll
    for (int jj = 0; jj < 2; ++jj) {
        if (j + jj >= A) break;
        float acc[2][4];
        gemm16<false, false>(acc, sm.h2, kFS2, m0, sm.w3, kFS2, 16 * (j + jj), kFH);
#pragma unroll
        for (int h = 0; h < 2; ++h) {
            const int c = 16 * jj + 8 * h + 2 * t;
            const float c0 = sm.b3[16 * j + c], c1 = sm.b3[16 * j + c + 1];
            *reinterpret_cast<float2*>(lg + g * kLs + c) = make_float2(acc[h][0] + c0, acc[h][1] + c1);
            *reinterpret_cast<float2*>(lg + (g + 8) * kLs + c) = make_float2(acc[h][2] + c0, acc[h][3] + c1);
        }
    }
    __syncwarp();
}

__device__ __forceinline__ void load_logits(const float* p, float (&L)[kFK]) {
#pragma unroll
    for (int k = 0; k < kFK; k += 4) {
        const float4 v = *reinterpret_cast<const float4*>(p + k);
        L[k] = v.x;
        L[k + 1] = v.y;
        L[k + 2] = v.z;
        L[k + 3] = v.w;
    }
}

// One minibatch: rows x[d][off + j], weights w[off + j], j < batch.
// wsum_dev = sum of the minibatch weights; loss_dev += -sum w log q / wsum.
__global__ void __launch_bounds__(kTrainThreads) flow_train_kernel(FlowView f, const float* x, const float* w,
                                                                   uint64_t n, uint64_t off, uint32_t batch,
                                                                   const float* wsum_dev, float* grad,
                                                                   float* loss_dev) {
    extern __shared__ __align__(16) unsigned char smem_raw[];
    TrainSmem& sm = *reinterpret_cast<TrainSmem*>(smem_raw);
    const int D = (int)f.D, A = (int)f.A, AK = (int)f.AK;
    const size_t S = flow_layer_floats(f.D);
    const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
    const int wr = warp & 3, wc = warp >> 2;  // row group, column group
    const int m0 = 16 * wr, n0 = 16 * wc;
    float* lg = sm.lg[warp];
    const int lr = lane & 15, lj = lane >> 4;  // softmax: row and coordinate of the pair
    const int row = m0 + lr;
    fetch_w1(f, 0, sm);
    fetch_w2(f, 0, sm);
    fetch_w3(f, 0, sm);
    for (int e = threadIdx.x; e < kFL * D; e += kTrainThreads) sm.perm[e] = f.perm[e];
    const uint32_t j0 = blockIdx.x * kRows;
    const float inv_w = 1.0f / fmaxf(*wsum_dev, 1e-30f);
    for (int r = threadIdx.x; r < kRows; r += kTrainThreads) {
        const uint32_t j = j0 + r;
        sm.s[r] = -(j < batch ? w[off + j] : 0.f) * inv_w;
    }
    for (int e = threadIdx.x; e < kRows * D; e += kTrainThreads) {
        const int r = e & (kRows - 1), d = e / kRows;
        const uint32_t j = j0 + r;
        sm.x[r * kXs + d] = j < batch ? x[(uint64_t)d * n + off + j] : 0.5f;
        sm.g[r * kXs + d] = 0.f;
    }
    // ---- forward (density direction), storing the state entering each layer.
    // Copy groups: the next layer's matrix 1 starts with the layer (its other
    // buffer), matrix 2 once h2 is done, matrix 3 once the logits are; each wait
    // leaves the groups started later pending.
    float dlq = 0.f;  // this lane's part of log q of its row
    for (int l = 0; l < kFL; ++l) {
        const uint8_t* pm = sm.perm + l * D;
        const bool next = l + 1 < kFL;
        __syncthreads();  // x is complete
        for (int e = threadIdx.x; e < kRows * kXs; e += kTrainThreads) sm.stash[l][e] = sm.x[e];
        load_xa(pm, A, sm);
        copy_wait<1>();   // matrices 1 and 2
        __syncthreads();
        if (next) fetch_w1(f, l + 1, sm);
        hidden(sm.h1, sm.xa, kFS1, sm.w1[l & 1], kFS1, sm.b1[l & 1], kFAP, m0, n0);
        __syncthreads();
        hidden(sm.h2, sm.h1, kFS2, sm.w2, kFS2, sm.b2, kFH, m0, n0);
        if (next) copy_wait<1>();
        else copy_wait<0>();  // matrix 3
        __syncthreads();
        if (next) fetch_w2(f, l + 1, sm);
        for (int j = 2 * wc; j < A; j += 8) {
            logits_pair(lg, j, A, m0, sm);
            if (j + lj < A) {
                float L[kFK];
                load_logits(lg + lr * kLs + 16 * lj, L);
                float m = L[0];
#pragma unroll
                for (int k = 1; k < kFK; ++k) m = fmaxf(m, L[k]);
                float Q[kFK], sum = 0.f;
#pragma unroll
                for (int k = 0; k < kFK; ++k) {
                    Q[k] = __expf(L[k] - m);
                    sum += Q[k];
                }
                const float sc = (1.0f - kFE) / sum;
                float* xv = sm.x + row * kXs + pm[A + j + lj];
                const float tt = *xv;
                const int b = min((int)(tt * (float)kFK), kFK - 1);
                const int at = max(b, 0);  // a coordinate below 0 (b < 0) continues bin 0
                float lo = 0.f, qb = 0.f;
#pragma unroll
                for (int k = 0; k < kFK; ++k) {
                    const float q = Q[k] * sc + kFE / kFK;
                    if (k < b) lo += q;
                    if (k == at) qb = q;
                }
                *xv = lo + (tt * (float)kFK - (float)b) * qb;
                dlq += __logf((float)kFK * qb);
            }
            __syncwarp();
        }
        if (next) {
            __syncthreads();
            fetch_w3(f, l + 1, sm);
        }
    }
    dlq += __shfl_down_sync(0xffffffffu, dlq, 16);
    if (lane < 16) sm.lq[wc][row] = dlq;
    __syncthreads();
    if (threadIdx.x < 32) {
        float part = 0.f;
        for (int r = threadIdx.x; r < kRows; r += 32)
            part += sm.s[r] * ((sm.lq[0][r] + sm.lq[1][r]) + (sm.lq[2][r] + sm.lq[3][r]));
        for (int o = 16; o > 0; o >>= 1) part += __shfl_down_sync(0xffffffffu, part, o);
        if (threadIdx.x == 0) atomicAdd(loss_dev, part);
    }
    // ---- backward through the layers.  The last layer's weights, xa, h1 and h2
    // are still there; for the others the hidden layers are recomputed.
    for (int l = kFL - 1; l >= 0; --l) {
        const uint8_t* pm = sm.perm + l * D;
        float* gl = grad + (size_t)l * S;
        for (int e = threadIdx.x; e < kRows * kXs; e += kTrainThreads) sm.x[e] = sm.stash[l][e];
        if (l > 0) fetch_w1(f, l - 1, sm);
        __syncthreads();
        if (l < kFL - 1) {
            load_xa(pm, A, sm);
            if (l > 0) copy_wait<1>();  // this layer's three matrices
            else copy_wait<0>();
            __syncthreads();
            hidden(sm.h1, sm.xa, kFS1, sm.w1[l & 1], kFS1, sm.b1[l & 1], kFAP, m0, n0);
            __syncthreads();
            hidden(sm.h2, sm.h1, kFS2, sm.w2, kFS2, sm.b2, kFH, m0, n0);
            __syncthreads();
        }
        // logits, two coordinates at a time -> dL/dO (bf16) and dL/dt of the transformed coordinates
        for (int j = 2 * wc; j < A; j += 8) {
            logits_pair(lg, j, A, m0, sm);
            if (j + lj < A) {
                float L[kFK];
                load_logits(lg + lr * kLs + 16 * lj, L);
                float m = L[0];
#pragma unroll
                for (int k = 1; k < kFK; ++k) m = fmaxf(m, L[k]);
                float P[kFK], sum = 0.f;
#pragma unroll
                for (int k = 0; k < kFK; ++k) {
                    P[k] = __expf(L[k] - m);
                    sum += P[k];
                }
#pragma unroll
                for (int k = 0; k < kFK; ++k) P[k] /= sum;
                const int cb = pm[A + j + lj];
                const float tt = sm.x[row * kXs + cb];
                const int b = min((int)(tt * (float)kFK), kFK - 1);
                const int at = max(b, 0);  // as in the forward pass
                float pb = 0.f;
#pragma unroll
                for (int k = 0; k < kFK; ++k) pb = k == at ? P[k] : pb;
                const float qb = (1.0f - kFE) * pb + kFE / kFK;
                const float up = sm.g[row * kXs + cb];  // dL/d(output coordinate)
                const float at_b = up * (tt * (float)kFK - (float)b) + sm.s[row] / qb;
                // dL/dQ_k = up ([k < b] + [k == at](tK - b)) + s [k == at] / Q_at
                float dot = 0.f;
#pragma unroll
                for (int k = 0; k < kFK; ++k) dot += P[k] * (k < b ? up : k == at ? at_b : 0.f);
                uint32_t o[kFK / 2];
#pragma unroll
                for (int k = 0; k < kFK; k += 2) {
                    const float d0 = k < b ? up : k == at ? at_b : 0.f;
                    const float d1 = k + 1 < b ? up : k + 1 == at ? at_b : 0.f;
                    const __nv_bfloat162 v = __floats2bfloat162_rn((1.0f - kFE) * P[k] * (d0 - dot),
                                                                   (1.0f - kFE) * P[k + 1] * (d1 - dot));
                    o[k / 2] = *reinterpret_cast<const uint32_t*>(&v);
                }
                uint4* dst = reinterpret_cast<uint4*>(sm.dO + row * kSO + 16 * (j + lj));
                dst[0] = make_uint4(o[0], o[1], o[2], o[3]);
                dst[1] = make_uint4(o[4], o[5], o[6], o[7]);
                sm.g[row * kXs + cb] = up * (float)kFK * qb;  // dL/dt through the CDF
            }
            __syncwarp();
        }
        __syncthreads();
        {   // dh2 = (dO W3) * [h2 > 0]
            float acc[2][4];
            gemm16<false, true>(acc, sm.dO, kSO, m0, sm.w3, kFS2, n0, AK);
            store_bf16(sm.dh2, kFS2, m0, n0, acc, [&](int r, int c, float a, float b) {
                const float2 h = __bfloat1622float2(*reinterpret_cast<const __nv_bfloat162*>(sm.h2 + r * kFS2 + c));
                return __floats2bfloat162_rn(h.x > 0.f ? a : 0.f, h.y > 0.f ? b : 0.f);
            });
        }
        // dW3 = dO^T h2, 16 x 16 blocks over the warps; db3 = column sums of dO
        for (int u = warp; u < AK / 4; u += kTrainThreads / 32) {
            float acc[2][4];
            gemm16<true, true>(acc, sm.dO, kSO, 16 * (u >> 2), sm.h2, kFS2, 16 * (u & 3), kRows);
            add_grad(gl + off_w3(), kFH, 16 * (u >> 2), 16 * (u & 3), acc);
        }
        for (int e = threadIdx.x; e < 2 * AK; e += kTrainThreads)  // 4 quarters of the rows
            add_column_sums(gl + off_b3(f.AK), sm.dO, kSO, e % (AK / 2), 16 * (e / (AK / 2)), 16);
        __syncthreads();
        if (l > 0) fetch_w3(f, l - 1, sm);
        {   // dh1 = (dh2 W2) * [h1 > 0]
            float acc[2][4];
            gemm16<false, true>(acc, sm.dh2, kFS2, m0, sm.w2, kFS2, n0, kFH);
            store_bf16(sm.dh1, kFS2, m0, n0, acc, [&](int r, int c, float a, float b) {
                const float2 h = __bfloat1622float2(*reinterpret_cast<const __nv_bfloat162*>(sm.h1 + r * kFS2 + c));
                return __floats2bfloat162_rn(h.x > 0.f ? a : 0.f, h.y > 0.f ? b : 0.f);
            });
            gemm16<true, true>(acc, sm.dh2, kFS2, m0, sm.h1, kFS2, n0, kRows);  // dW2 = dh2^T h1
            add_grad(gl + off_w2(), kFH, m0, n0, acc);
            if (wr == 0) add_column_sums(gl + off_b2(), sm.dh2, kFS2, lane, 16 * wc, 16);
        }
        __syncthreads();
        if (l > 0) fetch_w2(f, l - 1, sm);
        if (wc == 0) {  // d x_A = dh1 W1 -> into the conditioner coordinates' gradient
            float acc[2][4];
            gemm16<false, true>(acc, sm.dh1, kFS2, m0, sm.w1[l & 1], kFS1, 0, kFH);
            const int g = lane >> 2, t = lane & 3;
#pragma unroll
            for (int h = 0; h < 2; ++h)
#pragma unroll
                for (int q = 0; q < 4; ++q) {
                    const int r = m0 + g + (q >= 2 ? 8 : 0), c = 8 * h + 2 * t + (q & 1);
                    if (c < A) sm.g[r * kXs + pm[c]] += acc[h][q];
                }
        } else if (wc == 1) {  // dW1 = dh1^T xa
            float acc[2][4];
            gemm16<true, true>(acc, sm.dh1, kFS2, m0, sm.xa, kFS1, 0, kRows);
            add_grad(gl, kFAP, m0, 0, acc);
        } else if (wc == 2) {
            add_column_sums(gl + off_b1(), sm.dh1, kFS2, lane, 16 * wr, 16);
        }
        if (l > 0) __syncthreads();  // the next layer overwrites x, and w1's other buffer
    }
}

// Weight sums of minibatch windows: block k sums w[off_k .. off_k + batch) into
// out[k * stride], off_k = offs[k] (off when offs is null).
__global__ void __launch_bounds__(512) wsum_kernel(const float* w, const uint64_t* offs, uint64_t off, uint32_t batch,
                                                   float* out, uint32_t stride) {
    const float* p = w + (offs ? offs[blockIdx.x] : off);
    float s = 0.f;
    for (uint32_t j = threadIdx.x; j < batch; j += blockDim.x) s += p[j];
    for (int o = 16; o > 0; o >>= 1) s += __shfl_down_sync(0xffffffffu, s, o);
    __shared__ float part[16];
    if ((threadIdx.x & 31) == 0) part[threadIdx.x >> 5] = s;
    __syncthreads();
    if (threadIdx.x < 32) {
        s = threadIdx.x < (blockDim.x >> 5) ? part[threadIdx.x] : 0.f;
        for (int o = 8; o > 0; o >>= 1) s += __shfl_down_sync(0xffffffffu, s, o);
        if (threadIdx.x == 0) out[(size_t)blockIdx.x * stride] = s;
    }
}

// Where parameter o of a layer (master layout) lies in the training copy: a
// padded bf16 weight (wb) or an FP32 bias.
__device__ __forceinline__ void pack_param(uint32_t l, uint32_t o, float v, __nv_bfloat16* wb, float* bias,
                                           uint32_t AK) {
    __nv_bfloat16* w = wb + (size_t)l * (kFH * kFS1 + kFH * kFS2 + (size_t)AK * kFS2);
    float* b = bias + (size_t)l * (2 * kFH + AK);
    const uint32_t ob1 = kFH * kFAP, ow2 = ob1 + kFH, ob2 = ow2 + kFH * kFH, ow3 = ob2 + kFH, ob3 = ow3 + AK * kFH;
    if (o < ob1) w[o / kFAP * kFS1 + o % kFAP] = __float2bfloat16_rn(v);
    else if (o < ow2) b[o - ob1] = v;
    else if (o < ob2) w[kFH * kFS1 + (o - ow2) / kFH * kFS2 + (o - ow2) % kFH] = __float2bfloat16_rn(v);
    else if (o < ow3) b[kFH + o - ob2] = v;
    else if (o < ob3) w[kFH * kFS1 + kFH * kFS2 + (o - ow3) / kFH * kFS2 + (o - ow3) % kFH] = __float2bfloat16_rn(v);
    else b[2 * kFH + o - ob3] = v;
}

// Adam (Kingma & Ba, 2015) on the FP32 master parameters; leaves the gradient
// zeroed for the next step and the training copy (wb, bias) up to date, which
// otherwise cost a memset and a packing launch per step.
__global__ void adam_kernel(float* p, float* gr, float* m, float* v, uint32_t count, uint32_t layer, float lr, float b1,
                            float b2, float eps, float bc1, float bc2, __nv_bfloat16* wb, float* bias, uint32_t AK) {
    for (uint32_t e = blockIdx.x * blockDim.x + threadIdx.x; e < count; e += gridDim.x * blockDim.x) {
        const float gg = gr[e];
        const float mm = b1 * m[e] + (1.f - b1) * gg;
        const float vv = b2 * v[e] + (1.f - b2) * gg * gg;
        gr[e] = 0.f;
        m[e] = mm;
        v[e] = vv;
        const float q = p[e] - lr * (mm / bc1) / (sqrtf(vv / bc2) + eps);
        p[e] = q;
        pack_param(e / layer, e % layer, q, wb, bias, AK);
    }
}

// FP32 master parameters (the documented layout: per layer W1 [64][16], b1,
// W2 [64][64], b2, W3 [AK][64], b3) -> padded bf16 weights + FP32 biases.
__global__ void pack_kernel(const float* master, __nv_bfloat16* wb, float* bias, uint32_t AK) {
    const int l = blockIdx.y;
    const size_t S = (size_t)kFH * kFAP + kFH + kFH * kFH + kFH + (size_t)AK * kFH + AK;
    const float* m = master + l * S;
    __nv_bfloat16* w = wb + (size_t)l * (kFH * kFS1 + kFH * kFS2 + (size_t)AK * kFS2);
    float* b = bias + (size_t)l * (2 * kFH + AK);
    const uint32_t tot = kFH * kFS1 + kFH * kFS2 + AK * kFS2;
    for (uint32_t e = blockIdx.x * blockDim.x + threadIdx.x; e < tot; e += gridDim.x * blockDim.x) {
        float v = 0.f;
        if (e < (uint32_t)(kFH * kFS1)) {
            const uint32_t r = e / kFS1, c = e % kFS1;
            if (c < (uint32_t)kFAP) v = m[r * kFAP + c];
        } else if (e < (uint32_t)(kFH * kFS1 + kFH * kFS2)) {
            const uint32_t q = e - kFH * kFS1, r = q / kFS2, c = q % kFS2;
            if (c < (uint32_t)kFH) v = m[kFH * kFAP + kFH + r * kFH + c];
        } else {
            const uint32_t q = e - kFH * kFS1 - kFH * kFS2, r = q / kFS2, c = q % kFS2;
            if (c < (uint32_t)kFH) v = m[kFH * kFAP + kFH + kFH * kFH + kFH + r * kFH + c];
        }
        w[e] = __float2bfloat16_rn(v);
    }
    for (uint32_t e = blockIdx.x * blockDim.x + threadIdx.x; e < 2 * kFH + AK; e += gridDim.x * blockDim.x) {
        if (e < (uint32_t)kFH) b[e] = m[kFH * kFAP + e];
        else if (e < (uint32_t)(2 * kFH)) b[e] = m[kFH * kFAP + kFH + kFH * kFH + (e - kFH)];
        else b[e] = m[kFH * kFAP + kFH + kFH * kFH + kFH + (size_t)AK * kFH + (e - 2 * kFH)];
    }
}

// Chain states as training rows for the flow: x_out [D][n] = the current
// states, w_out[i] = p / (p + c~ u) = E[dt | x] = 1 / (1 + k(x)), which turns
// the states' jump-chain law (proportional to p + c~ u) into pi.
__global__ void snapshot_kernel(ChainView c, float* x_out, float* w_out) {
    const uint64_t i = blockIdx.x * (uint64_t)blockDim.x + threadIdx.x;
    if (i >= c.n) return;
    for (uint32_t d = 0; d < c.dim; ++d) x_out[d * c.n + i] = c.x[xidx(d, i, c.n)];
    const float p = c.fpu[3 * c.n + i], u = c.fpu[4 * c.n + i];
    w_out[i] = p > 0.f ? p / (p + c.c_tilde * u) : 0.f;
}

// The rows of weight > 0 appended to a ring: one counter update per warp.
__global__ void snapshot_append_kernel(ChainView c, float* x_ring, float* w_ring, uint64_t cap,
                                       unsigned long long* total) {
    const uint64_t i = blockIdx.x * (uint64_t)blockDim.x + threadIdx.x;
    const int lane = threadIdx.x & 31;
    float w = 0.f;
    if (i < c.n) {
        const float p = c.fpu[3 * c.n + i], u = c.fpu[4 * c.n + i];
        w = p > 0.f ? p / (p + c.c_tilde * u) : 0.f;
    }
    const unsigned keep = __ballot_sync(0xffffffffu, w > 0.f);
    if (!keep) return;
    unsigned long long base = 0;
    if (lane == 0) base = atomicAdd(total, (unsigned long long)__popc(keep));
    base = __shfl_sync(0xffffffffu, base, 0);
    if (!(w > 0.f)) return;
    const uint64_t slot = (base + __popc(keep & ((1u << lane) - 1u))) % cap;
    for (uint32_t d = 0; d < c.dim; ++d) x_ring[d * cap + slot] = c.x[xidx(d, i, c.n)];
    w_ring[slot] = w;
}

}  // namespace

cudaError_t launch_snapshot(const ChainView& c, float* x_out, float* w_out, cudaStream_t st) {
    snapshot_kernel<<<(unsigned)((c.n + 255) / 256), 256, 0, st>>>(c, x_out, w_out);
    return cudaGetLastError();
}

cudaError_t launch_snapshot_append(const ChainView& c, float* x_ring, float* w_ring, uint64_t cap,
                                   unsigned long long* total, cudaStream_t st) {
    snapshot_append_kernel<<<(unsigned)((c.n + 255) / 256), 256, 0, st>>>(c, x_ring, w_ring, cap, total);
    return cudaGetLastError();
}

cudaError_t launch_flow_wsum(const float* w, const uint64_t* offs, uint64_t off, uint32_t batch, float* out,
                             uint32_t stride, uint32_t count, cudaStream_t st) {
    wsum_kernel<<<count, 512, 0, st>>>(w, offs, off, batch, out, stride);
    return cudaGetLastError();
}

cudaError_t launch_flow_train_step(const FlowView& f, const float* x, const float* w, uint64_t n, uint64_t off,
                                   uint32_t batch, float* grad, const float* wsum, float* loss, cudaStream_t st) {
    static DeviceOnce once;  // per device: the opt-in to the training kernel's shared memory
    const size_t shm = sizeof(TrainSmem);
    cudaError_t e0 = once.get(
        [&](int, long long*) {
            return cudaFuncSetAttribute(flow_train_kernel, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)shm);
        },
        nullptr);
    if (e0 != cudaSuccess) return e0;
    flow_train_kernel<<<(batch + kRows - 1) / kRows, kTrainThreads, shm, st>>>(f, x, w, n, off, batch, wsum, grad,
                                                                              loss);
    return cudaGetLastError();
}

cudaError_t launch_adam(float* p, float* g, float* m, float* v, uint32_t D, float lr, uint64_t t, __nv_bfloat16* wb,
                        float* bias, cudaStream_t st) {
    const float b1 = 0.9f, b2 = 0.999f;
    const float bc1 = 1.0f - powf(b1, (float)t), bc2 = 1.0f - powf(b2, (float)t);
    const uint32_t layer = (uint32_t)flow_layer_floats(D), count = kFL * layer;
    adam_kernel<<<(count + 255) / 256, 256, 0, st>>>(p, g, m, v, count, layer, lr, b1, b2, 1e-8f, bc1, bc2, wb, bias,
                                                     D / 2 * kFK);
    return cudaGetLastError();
}

cudaError_t launch_flow_pack(const float* master, __nv_bfloat16* wb, float* bias, uint32_t AK, cudaStream_t st) {
    pack_kernel<<<dim3(16, kFL), 256, 0, st>>>(master, wb, bias, AK);
    return cudaGetLastError();
}

}  // namespace jr
