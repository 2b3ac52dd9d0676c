// Learned coarse-derivative surrogate: a multilayer perceptron c -> dc/dt trained on the
// least-squares slopes that resolved bursts measure (Section 3.3, Eq. (leastsquares)),
// with BF16 tensor-core GEMMs accumulating in FP32, GELU hidden layers, MSE loss and
// Adam. Every product runs on the tcgen05 tile of pe_tc.cuh (TMEM accumulator, TMA-staged operands)
// with the bias, activation, loss or GELU' factor fused into its epilogue: one launch per layer
// forward and per data gradient, one launch for all weight gradients. The weight gradients
// contract over the batch and read the row-major activations and gradients as they are
// (operands with M and N contiguous); the data gradients read the BF16 weights' transposes
// (rewritten with the mirror by Adam).
//
// What bounds a training step: the chain of its launches. Each product of the usual widths (512,
// batch 2048) is under 1 us of tensor-core time, so the work around it sets the time: a step
// of 512-512-512-512-512 at batch 2048 took 259 us in 20 launches (epilogues writing every row
// in 4-byte pieces and a second time transposed, an Adam kernel finding each weight's place with
// 64-bit divisions) and takes 91 us in 10, each started under its predecessor's tail
// (programmatic dependent launch); both as the mean of 200 steps of one call.
//
// Storage (caller-owned arena, see pe_mlp_layout_for): FP32 master parameters (the flat
// vector W_1 [d1][d0], b_1, W_2, ...), their BF16 mirror and its per-layer transposes used by
// the GEMMs, FP32 gradients, Adam moments, per-component z-score statistics, and a batch
// workspace.
#include <cuda_bf16.h>
#include <cuda_runtime.h>
#include <math.h>
#include <stdint.h>
#include <stdlib.h>
#include <string.h>

#include <algorithm>
#include <vector>

#include "pe_common.cuh"
#include "pe_ctx.h"
#include "pe_internal.h"
#include "pe_tc.cuh"
#include "pepic.h"

namespace pe {
namespace {

constexpr int kNormBlocks = 64;    // row blocks of the z-score statistics
constexpr int kLossSlots = 4096;

enum Epi { kEpiHidden = 0, kEpiHiddenInfer = 1, kEpiOutInfer = 2, kEpiOutTrain = 3, kEpiDgrad = 4, kEpiWgrad = 5 };

__device__ __forceinline__ float warp_sum_f(float v)
{
    for (int o = 16; o > 0; o >>= 1) v += __shfl_xor_sync(0xffffffffu, v, o);
    return v;
}

__device__ __forceinline__ float gelu_f(float z) { return 0.5f * z * (1.0f + erff(z * 0.70710678118654752f)); }
__device__ __forceinline__ float gelu_grad_f(float z)
{
    return 0.5f * (1.0f + erff(z * 0.70710678118654752f)) + z * 0.39894228040143268f * expf(-0.5f * z * z);
}

struct GemmArgs {
    const __nv_bfloat16* A;
    const __nv_bfloat16* B;
    int M, N, K, lda, ldb;
    const float* bias;     // [N] (hidden / output epilogues)
    float* Z;              // hidden: pre-activation out [M][N]; dgrad: pre-activation in
    __nv_bfloat16* Aout;   // hidden: GELU(z) out; train / dgrad: gradient out [M][N] (BF16)
    const float* T;        // train: normalised target [M][N]
    float* Y;              // output: FP32 out [M][N] (infer: de-normalised unless Y64 set)
    double* Y64;           // infer: de-normalised FP64 out
    const float* mu;       // infer: output mean [N]
    const float* sd;       // infer: output deviation [N]
    float* loss_part;      // train: one partial per block
    float gscale;          // train: 2 / (B D)
};

__device__ __forceinline__ uint32_t bf16_pair(float a, float b)
{
    const __nv_bfloat162 p = __floats2bfloat162_rn(a, b);
    return *reinterpret_cast<const uint32_t*>(&p);
}

// Epilogue of the tensor-core GEMM for row m, columns n0 .. n0 + 31 of C (FP32 from TMEM): the
// bias + GELU of a hidden layer (Aout, and Z in training), the de-normalised output (inference),
// the loss and output gradient (training), the data gradient times GELU'(Z), or the FP32 weight
// gradient. Rows beyond M are not stored. A lane holds a whole row piece, so rows go to memory in
// 32-byte vectors (every arena row is 128-byte aligned). finish() folds the training loss of
// the block into loss_part[block] (every thread calls it).
template <int EPI>
struct TcEpi {
    GemmArgs g;
    float lsum;

    __device__ __forceinline__ void operator()(int m, int n0, const float* v)
    {
        if (m >= g.M) return;
        const size_t o = (size_t)m * g.N + n0;
        uint32_t r[8], a[8];
#pragma unroll
        for (int j0 = 0; j0 < 32; j0 += 16) {
#pragma unroll
            for (int q = 0; q < 16; q += 8) {
                const int j = j0 + q;
                if (EPI == kEpiWgrad) {
#pragma unroll
                    for (int k = 0; k < 8; ++k) r[k] = __float_as_uint(v[j + k]);
                    tc::st_global32(g.Y + o + j, r);
                } else if (EPI == kEpiOutInfer) {
#pragma unroll
                    for (int k = 0; k < 8; k += 2) {
                        const int n = n0 + j + k;
                        const float v0 = v[j + k] + g.bias[n], v1 = v[j + k + 1] + g.bias[n + 1];
                        const float y0 = fmaf(v0, g.sd[n], g.mu[n]), y1 = fmaf(v1, g.sd[n + 1], g.mu[n + 1]);
                        if (g.Y64) {
                            g.Y64[o + j + k] = (double)y0;
                            g.Y64[o + j + k + 1] = (double)y1;
                        } else {
                            *reinterpret_cast<float2*>(g.Y + o + j + k) = make_float2(y0, y1);
                        }
                    }
                } else {
                    float b[8], x[8];
                    if (EPI == kEpiDgrad) tc::ld_global32(g.Z + o + j, r);
                    else if (EPI == kEpiOutTrain) tc::ld_global32(g.T + o + j, r);
                    if (EPI != kEpiDgrad) {  // the same address in every lane
                        const float4 b0 = *reinterpret_cast<const float4*>(g.bias + n0 + j);
                        const float4 b1 = *reinterpret_cast<const float4*>(g.bias + n0 + j + 4);
                        b[0] = b0.x, b[1] = b0.y, b[2] = b0.z, b[3] = b0.w;
                        b[4] = b1.x, b[5] = b1.y, b[6] = b1.z, b[7] = b1.w;
                    }
#pragma unroll
                    for (int k = 0; k < 8; ++k) {
                        if (EPI == kEpiHidden || EPI == kEpiHiddenInfer) {
                            const float z = v[j + k] + b[k];
                            r[k] = __float_as_uint(z);
                            x[k] = gelu_f(z);
                        } else if (EPI == kEpiOutTrain) {
                            const float d = (v[j + k] + b[k]) - __uint_as_float(r[k]);
                            lsum = fmaf(d, d, lsum);
                            x[k] = g.gscale * d;
                        } else {
                            x[k] = v[j + k] * gelu_grad_f(__uint_as_float(r[k]));
                        }
                    }
                    if (EPI == kEpiHidden) tc::st_global32(g.Z + o + j, r);
#pragma unroll
                    for (int k = 0; k < 8; k += 2) a[q / 2 + k / 2] = bf16_pair(x[k], x[k + 1]);
                }
            }
            if (EPI != kEpiWgrad && EPI != kEpiOutInfer) tc::st_global32(g.Aout + o + j0, a);
        }
    }

    __device__ __forceinline__ void finish()
    {
        if (EPI != kEpiOutTrain) return;
        __shared__ float sloss[tc::kThreads / 32];
        const float w = warp_sum_f(lsum);
        if ((threadIdx.x & 31) == 0) sloss[threadIdx.x >> 5] = w;
        __syncthreads();
        if (threadIdx.x == 0) {
            float t = 0.0f;
            for (int k = 0; k < tc::kThreads / 32; ++k) t += sloss[k];
            g.loss_part[blockIdx.y * gridDim.x + blockIdx.x] = t;
        }
    }
};

// Layer of a small batch (at most kSmallBatch rows; the gated macro step evaluates one): the
// product with its roles exchanged, C^T[n][b] = sum_k W[n][k] x[b][k], 128 outputs per block as the
// MMA's rows and the batch as its 32 columns. A thread then finishes one output, where the other
// form leaves the whole epilogue of a row to two lanes of the block. Same sums as the other form
// (the accumulation runs over k in the same order).
//
// The weights are loaded before the wait for the previous layer, so whatever writes them (Adam, a
// parameter upload) must have ended before the first layer starts. k_prep, the first kernel of every
// evaluation, sees to that: it releases the first layer only after its own wait. The layers
// themselves may release at once: nothing between k_prep and the last of them writes weights.
constexpr int kSmallBatch = 32;
constexpr int kSmallStages = 8;  // K = 512 in flight at once
constexpr int kSmallABytes = 128 * tc::kBK * 2, kSmallBBytes = kSmallBatch * tc::kBK * 2;
constexpr int kSmallStageBytes = kSmallABytes + kSmallBBytes;
constexpr int kSmallSmem = kSmallStages * kSmallStageBytes + 1024 + 8 * (2 * kSmallStages + 1) + 16;

template <bool LAST>
__global__ void __launch_bounds__(128, 1) k_mlp_small(const __grid_constant__ CUtensorMap tw,
                                                      const __grid_constant__ CUtensorMap tx, GemmArgs g,
                                                      uint32_t* status)
{
    using namespace tc;
    extern __shared__ uint8_t smem_raw[];
    uint8_t* smem = reinterpret_cast<uint8_t*>((reinterpret_cast<uintptr_t>(smem_raw) + 1023) & ~uintptr_t(1023));
    uint64_t* full = reinterpret_cast<uint64_t*>(smem + kSmallStages * kSmallStageBytes);
    uint64_t* empty = full + kSmallStages;
    uint64_t* done = empty + kSmallStages;
    uint32_t* tmem_slot = reinterpret_cast<uint32_t*>(done + 1);
    __shared__ int s_fail;
    const int tid = threadIdx.x, warp = tid >> 5, lane = tid & 31;
    const int n0 = (int)blockIdx.x * 128;
    const int ktiles = (g.K + kBK - 1) / kBK, pro = ktiles < kSmallStages ? ktiles : kSmallStages;
    if (tid == 0) {
        for (int s = 0; s < kSmallStages; ++s) {
            mbar_init(&full[s], 1);
            mbar_init(&empty[s], 1);
        }
        mbar_init(done, 1);
        fence_mbar_init();
        s_fail = 0;
        for (int t = 0; t < pro; ++t) {
            mbar_expect_tx(&full[t], kSmallStageBytes);
            tma_load_2d(smem + t * kSmallStageBytes, &tw, &full[t], t * kBK, n0);
        }
    }
    if (warp == 0) tmem_alloc(tmem_slot, 32);
    tc_fence_before();
    __syncthreads();
    tc_fence_after();
    const uint32_t tmem = *tmem_slot;
    grid_release();
    grid_wait();
    if (tid == 0) {
        for (int t = 0; t < pro; ++t)
            tma_load_2d(smem + t * kSmallStageBytes + kSmallABytes, &tx, &full[t], t * kBK, 0);
        int issued = pro, consumed = 0;
        bool ok = true;
        for (int kt = 0; kt < ktiles; ++kt) {
            const int s = kt % kSmallStages;
            if (!mbar_wait(&full[s], (uint32_t)((kt / kSmallStages) & 1))) {
                ok = false;
                break;
            }
            consumed = kt + 1;
            tc_fence_after();
            const uint32_t a0 = saddr(smem + s * kSmallStageBytes), b0 = a0 + kSmallABytes;
#pragma unroll
            for (int k = 0; k < kBK / 16; ++k)
                umma_bf16(tmem, sw128_desc(a0 + 32 * k), sw128_desc(b0 + 32 * k), idesc_bf16(128, kSmallBatch),
                          (kt | k) ? 1u : 0u);
            umma_commit(&empty[s]);
            const int t = kt - 1 + kSmallStages;
            if (kt >= 1 && t < ktiles) {
                const int q = (kt - 1) % kSmallStages;
                if (!mbar_wait(&empty[q], (uint32_t)(((kt - 1) / kSmallStages) & 1))) {
                    ok = false;
                    break;
                }
                mbar_expect_tx(&full[q], kSmallStageBytes);
                tma_load_2d(smem + q * kSmallStageBytes, &tw, &full[q], t * kBK, n0);
                tma_load_2d(smem + q * kSmallStageBytes + kSmallABytes, &tx, &full[q], t * kBK, 0);
                ++issued;
            }
        }
        umma_commit(done);
        if (!ok) {
            s_fail = 1;
            for (int t = consumed; t < issued; ++t)
                mbar_wait(&full[t % kSmallStages], (uint32_t)((t / kSmallStages) & 1));
        }
    }
    __syncthreads();
    bool ok = mbar_wait(done, 0u) && !s_fail;
    ok = __all_sync(0xFFFFFFFFu, ok);
    if (!ok && lane == 0) atomicOr(status, PE_FLAG_TIMEOUT);
    tc_fence_after();
    if (ok) {
        const int n = n0 + warp * 32 + lane;
        float v[32];
        tmem_ld32(tmem + ((uint32_t)(warp * 32) << 16), v);
        if (n < g.N) {
            const float bias = g.bias[n];
            const float sd = LAST ? g.sd[n] : 0.0f, mu = LAST ? g.mu[n] : 0.0f;
#pragma unroll
            for (int b = 0; b < 32; ++b) {
                if (b < g.M) {
                    const float z = v[b] + bias;
                    const size_t o = (size_t)b * g.N + n;
                    if (!LAST) g.Aout[o] = __float2bfloat16_rn(gelu_f(z));
                    else if (g.Y64) g.Y64[o] = (double)fmaf(z, sd, mu);
                    else g.Y[o] = fmaf(z, sd, mu);
                }
            }
        }
    }
    tc_fence_before();
    __syncthreads();
    if (warp == 0) tmem_dealloc(tmem, 32);
}

// ------------------------------------------------------------------ small kernels

// Weight blocks of the flat parameter vector: layer l's W [rows = d_{l+1}][cols = d_l] at off;
// its BF16 transpose [d_l][d_{l+1}] sits at the same offset of the transposed mirror.
struct WeightTable {
    int64_t off[PE_MLP_MAX_LAYERS];
    int rows[PE_MLP_MAX_LAYERS], cols[PE_MLP_MAX_LAYERS];
    int L;
};

// Writes the BF16 value of flat parameter i into the mirror and, for a weight, into the
// transposed mirror.
__device__ __forceinline__ void put_bf16(const WeightTable& wt, int64_t i, float w, __nv_bfloat16* __restrict__ pb,
                                         __nv_bfloat16* __restrict__ pbT)
{
    const __nv_bfloat16 b = __float2bfloat16_rn(w);
    pb[i] = b;
    for (int l = 0; l < wt.L; ++l) {
        const int64_t r = i - wt.off[l];
        if (r >= 0 && r < (int64_t)wt.rows[l] * wt.cols[l]) {
            const int row = (int)(r / wt.cols[l]), col = (int)(r - (int64_t)row * wt.cols[l]);
            pbT[wt.off[l] + (int64_t)col * wt.rows[l] + row] = b;
            break;
        }
    }
}

struct ParamSeg {
    int64_t off, n;
    float bound;  // weight init bound (0 for biases)
};
struct ParamTable {
    ParamSeg seg[2 * PE_MLP_MAX_LAYERS];
    int nseg;
};

__device__ __forceinline__ uint64_t splitmix64_seq(uint64_t seed, uint64_t i)
{
    uint64_t z = seed + (i + 1) * 0x9E3779B97F4A7C15ULL;
    z = (z ^ (z >> 30)) * 0xBF58476D1CE4E5B9ULL;
    z = (z ^ (z >> 27)) * 0x94D049BB133111EBULL;
    return z ^ (z >> 31);
}

// W = (2u - 1) a with u = (s_i >> 40) 2^-24 from the splitmix64 sequence (flat index i);
// biases 0. Writes the FP32 master and its BF16 mirror.
__global__ void k_mlp_init(ParamTable tab, WeightTable wt, uint64_t seed, float* __restrict__ p,
                           __nv_bfloat16* __restrict__ pb, __nv_bfloat16* __restrict__ pbT)
{
    for (int s = 0; s < tab.nseg; ++s) {
        const ParamSeg sg = tab.seg[s];
        for (int64_t i = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; i < sg.n; i += (int64_t)gridDim.x * blockDim.x) {
            const int64_t idx = sg.off + i;
            float w = 0.0f;
            if (sg.bound > 0.0f) {
                const float u = (float)(splitmix64_seq(seed, (uint64_t)idx) >> 40) * 5.9604644775390625e-8f;
                w = (2.0f * u - 1.0f) * sg.bound;
            }
            p[idx] = w;
            put_bf16(wt, idx, w, pb, pbT);
        }
    }
}

// Per-component column sums of X [rows][D] over row block blockIdx.y (pass 0: sum x;
// pass 1: sum (x - mu)^2), FP64, fixed order; with period P > 0 component k is pooled
// with every k' = k (mod P)-position of its block of P (translation-invariant statistics).
template <typename T>
__global__ void k_norm_partial(const T* __restrict__ X, int64_t rows, int D, const double* __restrict__ mu,
                               double* __restrict__ part)
{
    const int k = blockIdx.x * blockDim.x + threadIdx.x;
    if (k >= D) return;
    const int64_t per = (rows + gridDim.y - 1) / gridDim.y;
    const int64_t r0 = blockIdx.y * per, r1 = min(rows, r0 + per);
    double s = 0.0;
    const double m = mu ? mu[k] : 0.0;
    for (int64_t r = r0; r < r1; ++r) {
        const double x = (double)X[r * D + k];
        s += mu ? (x - m) * (x - m) : x;
    }
    part[(size_t)blockIdx.y * D + k] = s;
}

// Folds the row-block partials (and, with P > 0, the P positions of each block) into
// mean (pass 0) or deviation (pass 1, with the 1e-6 max floor) in FP64 and FP32.
__global__ void k_norm_final(const double* __restrict__ part, int nparts, int D, int P, int64_t rows, int pass,
                             double* __restrict__ acc64, float* __restrict__ out32)
{
    __shared__ double red[32];
    __shared__ double smax;
    for (int k = threadIdx.x; k < D; k += blockDim.x) {
        double s = 0.0;
        int64_t cnt = rows;
        if (P > 0) {
            const int b0 = (k / P) * P;
            for (int j = 0; j < P; ++j)
                for (int q = 0; q < nparts; ++q) s += part[(size_t)q * D + b0 + j];
            cnt = rows * P;
        } else {
            for (int q = 0; q < nparts; ++q) s += part[(size_t)q * D + k];
        }
        acc64[D + k] = (pass == 0) ? s / (double)cnt : sqrt(s / (double)cnt);
    }
    __syncthreads();
    if (pass == 0) {
        for (int k = threadIdx.x; k < D; k += blockDim.x) {
            acc64[k] = acc64[D + k];
            out32[k] = (float)acc64[k];
        }
        return;
    }
    double mx = 0.0;
    for (int k = threadIdx.x; k < D; k += blockDim.x) mx = fmax(mx, acc64[D + k]);
    mx = warp_max(mx);
    if ((threadIdx.x & 31) == 0) red[threadIdx.x >> 5] = mx;
    __syncthreads();
    if (threadIdx.x == 0) {
        double m = 0.0;
        for (int w = 0; w < (int)(blockDim.x >> 5); ++w) m = fmax(m, red[w]);
        smax = 1e-6 * fmax(m, 1e-30);
    }
    __syncthreads();
    for (int k = threadIdx.x; k < D; k += blockDim.x) out32[k] = (float)fmax(acc64[D + k], smax);
}

// Normalised BF16 inputs (and FP32 targets) of a batch, one row per block: x'[k] = x[src(k)] with
// the circular shift s inside each block of P components, src(k) = b P + (j - s) mod P. The row
// and shift come from rows (shift 0), or, drawing a training batch (step not null), from the
// splitmix64 sequence of (seed, step): row = (h >> 32) npairs >> 32, shift = (h mod 2^32) P >> 32;
// else block i takes row i.
template <typename T>
__global__ void __launch_bounds__(128) k_prep(const T* __restrict__ X, const float* __restrict__ Y, int B, int D,
                                              int Dout, const int32_t* __restrict__ rows,
                                              const int64_t* __restrict__ step, uint64_t seed, int64_t npairs, int P,
                                              const float* __restrict__ mu, const float* __restrict__ sd,
                                              const float* __restrict__ mu_o, const float* __restrict__ sd_o,
                                              __nv_bfloat16* __restrict__ xz, float* __restrict__ tz)
{
    // in this order: a small evaluation's layers read the weights before their own wait, and Adam may
    // be the kernel that this one waits for
    grid_wait();
    grid_release();
    const int i = blockIdx.x;
    int64_t r = rows ? rows[i] : i;
    int s = 0;
    if (step) {
        const uint64_t h = splitmix64_seq(seed, (uint64_t)(*step) * (uint64_t)B + (uint64_t)i);
        r = (int32_t)(((h >> 32) * (uint64_t)npairs) >> 32);
        s = P > 0 ? (int32_t)(((h & 0xFFFFFFFFull) * (uint64_t)P) >> 32) : 0;
    }
    auto source = [&](int k) {
        if (P <= 0) return k;
        const int j = k % P;
        return k - j + (j >= s ? j - s : j - s + P);
    };
    // dims are multiples of 64: pairs of components, one 4-byte store each
    for (int k = 2 * threadIdx.x; k < D; k += 2 * blockDim.x) {
        const float x0 = (float)X[r * D + source(k)], x1 = (float)X[r * D + source(k + 1)];
        reinterpret_cast<uint32_t*>(xz + (size_t)i * D)[k >> 1] =
            bf16_pair((x0 - mu[k]) / sd[k], (x1 - mu[k + 1]) / sd[k + 1]);
    }
    if (Y)
        for (int k = threadIdx.x; k < Dout; k += blockDim.x)
            tz[(size_t)i * Dout + k] = (Y[r * Dout + source(k)] - mu_o[k]) / sd_o[k];
}

// Bias correction of Adam step t = *step + 1 into c[2], and the step counter advanced. The decay
// rates come in FP64 (0.999 is not a float); one thread, once per step: the FP64 powers cost
// microseconds on every thread that forms them.
__device__ __forceinline__ void adam_begin(int64_t* step, float* c, double b1, double b2)
{
    const int64_t t = *step + 1;
    c[0] = (float)(1.0 / (1.0 - pow(b1, (double)t)));
    c[1] = (float)(1.0 / (1.0 - pow(b2, (double)t)));
    *step = t;
}

__global__ void k_adam_begin(int64_t* step, float* c, double b1, double b2)
{
    if (threadIdx.x == 0 && blockIdx.x == 0) adam_begin(step, c, b1, b2);
}

// All weight and bias gradients of the network and the loss, one launch: they depend only on the
// forward and data-gradient passes, so the layers' tiles fill the GPU together (32 tiles of a
// 512 x 512 layer alone leave four fifths of it idle for the length of a batch's reduction).
// Blocks, in this order: per layer the tiles of dW_l [d_{l+1}][d_l] = G_l^T act_{l-1} (contraction
// over the batch, operands row-major), then per layer the 64-column blocks of db_l, then one
// block for the loss and, in a training step (adam), Adam's bias corrections.
struct WgradArgs {
    CUtensorMap a[PE_MLP_MAX_LAYERS], b[PE_MLP_MAX_LAYERS];  // G_l, act_{l-1}: dims {d, B}, boxes {64, 64}
    const __nv_bfloat16* G[PE_MLP_MAX_LAYERS];
    float* dW[PE_MLP_MAX_LAYERS];
    float* db[PE_MLP_MAX_LAYERS];
    int tile0[PE_MLP_MAX_LAYERS + 1], bias0[PE_MLP_MAX_LAYERS + 1];  // first block of each layer's tiles / columns
    int M[PE_MLP_MAX_LAYERS], N[PE_MLP_MAX_LAYERS];
    int L, B;
    const float* loss_part;
    int nloss;
    float loss_scale;
    float* loss;
    int adam;
    int64_t* step;
    float* corr;
    double b1, b2;
};

// Bias gradient db[n] = sum_m G[m][n] of 64 columns: 32 running sums per column (rows m = l mod 32,
// FP32, in row order), folded pairwise (l with l + 16, then + 8, ...): a fixed order.
__device__ __forceinline__ void bias_grad_block(const __nv_bfloat16* G, int B, int N, int n0, float* db, float* red)
{
    const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
    const uint32_t* G2 = reinterpret_cast<const uint32_t*>(G + n0) + lane;  // columns n0 + 2 lane, + 1
    float s0[4], s1[4];
#pragma unroll
    for (int k = 0; k < 4; ++k) s0[k] = s1[k] = 0.0f;
#pragma unroll 4
    for (int m = 4 * warp; m < B; m += 32) {  // B a multiple of 32
        uint32_t u[4];
#pragma unroll
        for (int k = 0; k < 4; ++k) u[k] = __ldg(G2 + (size_t)(m + k) * (N / 2));
#pragma unroll
        for (int k = 0; k < 4; ++k) {
            s0[k] += __uint_as_float(u[k] << 16);
            s1[k] += __uint_as_float(u[k] & 0xFFFF0000u);
        }
    }
#pragma unroll
    for (int k = 0; k < 4; ++k) {
        red[(4 * warp + k) * 64 + 2 * lane] = s0[k];
        red[(4 * warp + k) * 64 + 2 * lane + 1] = s1[k];
    }
    __syncthreads();
    for (int h = 16; h > 0; h >>= 1) {
        for (int t = threadIdx.x; t < h * 64; t += blockDim.x) red[t] += red[t + h * 64];
        __syncthreads();
    }
    if (threadIdx.x < 64) db[n0 + threadIdx.x] = red[threadIdx.x];
}

__global__ void __launch_bounds__(tc::kThreads, 1) k_mlp_wgrad(const __grid_constant__ WgradArgs w, uint32_t* status)
{
    extern __shared__ uint8_t smem_raw[];
    const int blk = blockIdx.x, L = w.L;
    if (blk < w.tile0[L]) {
        int l = 0;
        while (blk >= w.tile0[l + 1]) ++l;
        const int t = blk - w.tile0[l], nx = w.N[l] / 64;
        TcEpi<kEpiWgrad> e{};
        e.g.M = w.M[l];
        e.g.N = w.N[l];
        e.g.Y = w.dW[l];
        tc::gemm_tile<64, true>(&w.a[l], &w.b[l], (t / nx) * tc::kBM, (t % nx) * 64, w.B, e, status);
        return;
    }
    grid_release();
    grid_wait();
    if (blk < w.bias0[L]) {
        int l = 0;
        while (blk >= w.bias0[l + 1]) ++l;
        bias_grad_block(w.G[l], w.B, w.M[l], 64 * (blk - w.bias0[l]), w.db[l], reinterpret_cast<float*>(smem_raw));
        return;
    }
    __shared__ double red[32];
    double s = 0.0;
    for (int i = threadIdx.x; i < w.nloss; i += blockDim.x) s += (double)w.loss_part[i];
    s = warp_sum(s);
    if ((threadIdx.x & 31) == 0) red[threadIdx.x >> 5] = s;
    __syncthreads();
    if (threadIdx.x == 0) {
        double t = 0.0;
        for (int k = 0; k < (int)(blockDim.x >> 5); ++k) t += red[k];
        *w.loss = (float)(t * w.loss_scale);
        if (w.adam) adam_begin(w.step, w.corr, w.b1, w.b2);
    }
}

// Adam with bias correction (corr: adam_begin's factors; the step counter lives on the device, so
// graph replays advance it). theta, m, v FP32; the BF16 mirror and its transposes are rewritten.
// The decay rates and their complements come in FP64 (0.999 is not a float). Bound by memory (32
// bytes per parameter; L2 holds the arrays of the usual networks): a block takes a 64 x 64 tile of
// one layer's weights, so that the mirror's transpose leaves through shared memory in rows of 128
// bytes; the last blocks take the biases. (One thread per parameter at any index, with the
// transposed store at a stride and 64-bit divisions to find it: 51 us for 10^6 parameters, 9 us
// now.)
__global__ void __launch_bounds__(256) k_adam(float* __restrict__ p, __nv_bfloat16* __restrict__ pb,
                                              __nv_bfloat16* __restrict__ pbT, WeightTable wt,
                                              const float* __restrict__ grad, float* __restrict__ m,
                                              float* __restrict__ v, const float* __restrict__ corr, float lr, double b1,
                                              double b2, float eps)
{
    __shared__ __nv_bfloat16 tile[64][66];
    grid_release();
    grid_wait();
    const float c1 = corr[0], c2 = corr[1];
    const float fb1 = (float)b1, fb2 = (float)b2, ob1 = (float)(1.0 - b1), ob2 = (float)(1.0 - b2);
    auto update = [&](float& w, float& mi, float& vi, float gi) {
        mi = fmaf(fb1, mi, ob1 * gi);
        vi = fmaf(fb2, vi, ob2 * gi * gi);
        w = w - lr * (mi * c1) / (sqrtf(vi * c2) + eps);
    };
    int blk = blockIdx.x, l = 0;
    for (; l < wt.L; ++l) {
        const int n = (wt.rows[l] / 64) * (wt.cols[l] / 64);
        if (blk < n) break;
        blk -= n;
    }
    if (l == wt.L) {  // biases, 256 per block
        for (l = 0; l < wt.L; ++l) {
            const int n = (wt.rows[l] + 255) / 256;
            if (blk < n) break;
            blk -= n;
        }
        const int k = 256 * blk + threadIdx.x;
        if (l < wt.L && k < wt.rows[l]) {
            const int64_t i = wt.off[l] + (int64_t)wt.rows[l] * wt.cols[l] + k;
            float w = p[i], mi = m[i], vi = v[i];
            update(w, mi, vi, grad[i]);
            m[i] = mi;
            v[i] = vi;
            p[i] = w;
            pb[i] = __float2bfloat16_rn(w);
        }
        return;
    }
    const int rows = wt.rows[l], cols = wt.cols[l], nx = cols / 64;
    const int r0 = 64 * (blk / nx), c0 = 64 * (blk % nx);
    const int tr = threadIdx.x >> 4, tc4 = 4 * (threadIdx.x & 15);
#pragma unroll
    for (int q = 0; q < 4; ++q) {
        const int r = tr + 16 * q;
        const int64_t i = wt.off[l] + (int64_t)(r0 + r) * cols + c0 + tc4;
        float4 w4 = *reinterpret_cast<const float4*>(p + i), m4 = *reinterpret_cast<const float4*>(m + i);
        float4 v4 = *reinterpret_cast<const float4*>(v + i);
        const float4 g4 = *reinterpret_cast<const float4*>(grad + i);
        update(w4.x, m4.x, v4.x, g4.x);
        update(w4.y, m4.y, v4.y, g4.y);
        update(w4.z, m4.z, v4.z, g4.z);
        update(w4.w, m4.w, v4.w, g4.w);
        *reinterpret_cast<float4*>(p + i) = w4;
        *reinterpret_cast<float4*>(m + i) = m4;
        *reinterpret_cast<float4*>(v + i) = v4;
        const uint2 b = make_uint2(bf16_pair(w4.x, w4.y), bf16_pair(w4.z, w4.w));
        *reinterpret_cast<uint2*>(pb + i) = b;
        uint32_t* t = reinterpret_cast<uint32_t*>(&tile[r][tc4]);
        t[0] = b.x;
        t[1] = b.y;
    }
    __syncthreads();
    // transpose: column c of the tile is a row piece of 64 elements, four threads per column
    const int c = threadIdx.x >> 2, k0 = 16 * (threadIdx.x & 3);
    uint32_t o[8];
#pragma unroll
    for (int k = 0; k < 8; ++k) {
        const __nv_bfloat162 t2 = __halves2bfloat162(tile[k0 + 2 * k][c], tile[k0 + 2 * k + 1][c]);
        o[k] = *reinterpret_cast<const uint32_t*>(&t2);
    }
    tc::st_global32(pbT + wt.off[l] + (int64_t)(c0 + c) * rows + r0 + k0, o);
}

}  // namespace
}  // namespace pe

// ------------------------------------------------------------------ host side

struct pe_mlp {
    int L;
    int dims[PE_MLP_MAX_LAYERS + 1];
    int dmax, max_batch;
    int64_t nparams;
    int64_t w_off[PE_MLP_MAX_LAYERS], b_off[PE_MLP_MAX_LAYERS];
    pe_mlp_layout lay;
    char* arena;
    cudaStream_t stream;
    float* p;
    __nv_bfloat16* pb;
    __nv_bfloat16* pbT;  // per-layer transposes of the BF16 weights (same offsets as pb)
    pe::WeightTable wt;
    float* grad;
    float* am;
    float* av;
    float* norm;        // [4][dmax]: mu_in, sd_in, mu_out, sd_out
    double* norm64;     // [2][dmax] scratch of the statistics
    double* normpart;   // [kNormBlocks][dmax]
    int64_t* step;      // Adam step counter (device)
    float* loss;        // last training loss (device)
    float* corr;        // [2] bias corrections of the current Adam step (device)
    float* loss_part;   // [kLossSlots]
    __nv_bfloat16* xz;  // [Bm][d0]
    float* z[PE_MLP_MAX_LAYERS];
    __nv_bfloat16* a[PE_MLP_MAX_LAYERS];
    float* tz;          // [Bm][dL]
    __nv_bfloat16* g[PE_MLP_MAX_LAYERS];  // [Bm][d_{l+1}] gradient at layer l's output
    uint32_t* status;    // device status word (PE_FLAG_TIMEOUT from the GEMM's bounded waits)
    int shift_period;   // period used by the statistics (for reference)
};

using namespace pe;

namespace {

size_t al256(size_t x) { return (x + 255) & ~size_t(255); }

int check_dims(int32_t nlayers, const int32_t* dims, int32_t max_batch)
{
    if (nlayers < 1 || nlayers > PE_MLP_MAX_LAYERS || !dims || max_batch < 1 || max_batch > 65536) return PE_EINVAL;
    for (int l = 0; l <= nlayers; ++l)
        if (dims[l] < 64 || dims[l] > 4096 || dims[l] % 64) return PE_EINVAL;
    return PE_OK;
}

struct WorkPlan {
    size_t xz, z[PE_MLP_MAX_LAYERS], a[PE_MLP_MAX_LAYERS], tz, g[PE_MLP_MAX_LAYERS], total;
};

WorkPlan plan_work(int L, const int32_t* dims, int Bm)
{
    WorkPlan w;
    size_t o = 0;
    auto take = [&](size_t bytes) {
        size_t at = o;
        o += al256(bytes);
        return at;
    };
    w.xz = take(2 * (size_t)Bm * dims[0]);
    for (int l = 0; l + 1 < L; ++l) {
        w.z[l] = take(4 * (size_t)Bm * dims[l + 1]);
        w.a[l] = take(2 * (size_t)Bm * dims[l + 1]);
    }
    w.tz = take(4 * (size_t)Bm * dims[L]);
    for (int l = 0; l < L; ++l) w.g[l] = take(2 * (size_t)Bm * dims[l + 1]);
    w.total = o;
    return w;
}

// C[M][N] = A[M][K] B[N][K]^T on the tensor cores with the epilogue EPI; A and B stored
// with K contiguous (row strides lda, ldb).
// Tile width: 128 columns, or 64 when N needs it or when 128-wide tiles would leave SMs idle.
int tile_n(int N, int M)
{
    if (N % 128 != 0) return 64;
    return (N / 128) * ((M + tc::kBM - 1) / tc::kBM) < sm_count() ? 64 : 128;
}

template <int EPI>
int tc_gemm(pe_mlp* h, const GemmArgs& g, cudaStream_t s)
{
    const int bn = tile_n(g.N, g.M);
    CUtensorMap ma, mb;
    PE_TRY(tc_operand_map(&ma, g.A, g.M, g.K, g.lda, tc::kBM));
    PE_TRY(tc_operand_map(&mb, g.B, g.N, g.K, g.ldb, bn));
    TcEpi<EPI> e{g, 0.0f};
    const dim3 grid(g.N / bn, (g.M + tc::kBM - 1) / tc::kBM);
    if (bn == 128)
        return launch_dependent(tc::k_tc_gemm<128, TcEpi<EPI>>, grid, tc::kThreads, tc::TileCfg<128>::kSmemBytes, s, ma, mb,
                                g.K, e, h->status);
    return launch_dependent(tc::k_tc_gemm<64, TcEpi<EPI>>, grid, tc::kThreads, tc::TileCfg<64>::kSmemBytes, s, ma, mb, g.K,
                            e, h->status);
}

// One layer of a small batch (inference): the product with its roles exchanged.
template <bool LAST>
int small_layer(pe_mlp* h, const GemmArgs& g, cudaStream_t s)
{
    CUtensorMap mw, mx;
    PE_TRY(tc_operand_map(&mw, g.B, g.N, g.K, g.ldb, 128));
    PE_TRY(tc_operand_map(&mx, g.A, g.M, g.K, g.lda, kSmallBatch));
    return launch_dependent(k_mlp_small<LAST>, dim3((g.N + 127) / 128), 128, kSmallSmem, s, mw, mx, g, h->status);
}

// Loss partials of the output layer's GEMM (one per tile).
int loss_tiles(int Dout, int B) { return (Dout / tile_n(Dout, B)) * ((B + tc::kBM - 1) / tc::kBM); }

GemmArgs args0() { GemmArgs g; memset(&g, 0, sizeof(g)); return g; }

// Forward through every layer from h->xz (rows B). Inference: output into y32 / y64
// de-normalised; training: output compared with h->tz.
int forward(pe_mlp* h, int B, int train, float* y32, double* y64, int* launches)
{
    cudaStream_t s = h->stream;
    const __nv_bfloat16* in = h->xz;
    // batches of up to 32 rows: one 128-row tile of the usual form would be mostly padding
    const bool small = !train && B <= kSmallBatch;
    for (int l = 0; l < h->L; ++l) {
        GemmArgs g = args0();
        g.A = in;
        g.B = h->pb + h->w_off[l];
        g.M = B;
        g.N = h->dims[l + 1];
        g.K = h->dims[l];
        g.lda = h->dims[l];
        g.ldb = h->dims[l];
        g.bias = h->p + h->b_off[l];
        if (l + 1 < h->L) {
            g.Z = h->z[l];
            g.Aout = h->a[l];
            if (small) PE_TRY(small_layer<false>(h, g, s));
            else if (train) PE_TRY(tc_gemm<kEpiHidden>(h, g, s));
            else PE_TRY(tc_gemm<kEpiHiddenInfer>(h, g, s));
            in = h->a[l];
        } else if (!train) {
            g.Y = y32;
            g.Y64 = y64;
            g.mu = h->norm + 2 * h->dmax;
            g.sd = h->norm + 3 * h->dmax;
            if (small) PE_TRY(small_layer<true>(h, g, s));
            else PE_TRY(tc_gemm<kEpiOutInfer>(h, g, s));
        } else {
            g.T = h->tz;
            g.Aout = h->g[l];
            g.loss_part = h->loss_part;
            g.gscale = 2.0f / ((float)B * (float)g.N);
            PE_TRY(tc_gemm<kEpiOutTrain>(h, g, s));
        }
        ++*launches;
    }
    return PE_OK;
}

// Backward from the output gradient in g[L-1]: data gradients (times GELU') down to layer 1, then
// the weight and bias gradients of every layer into h->grad, the loss, and with adam the bias
// corrections of the step.
int backward(pe_mlp* h, int B, bool adam, double b1, double b2, int* launches)
{
    cudaStream_t s = h->stream;
    const int L = h->L, Dout = h->dims[L];
    for (int l = L - 1; l > 0; --l) {
        GemmArgs d = args0();  // G_{l-1} = (G_l W_l) * GELU'(z_{l-1}): W_l read as its transpose
        d.A = h->g[l];
        d.B = h->pbT + h->w_off[l];
        d.M = B;
        d.N = h->dims[l];
        d.K = h->dims[l + 1];
        d.lda = h->dims[l + 1];
        d.ldb = h->dims[l + 1];
        d.Z = h->z[l - 1];
        d.Aout = h->g[l - 1];
        PE_TRY(tc_gemm<kEpiDgrad>(h, d, s));
        ++*launches;
    }
    WgradArgs w;
    memset(&w, 0, sizeof(w));
    w.L = L;
    w.B = B;
    int blk = 0;
    for (int l = 0; l < L; ++l) {
        w.M[l] = h->dims[l + 1];
        w.N[l] = h->dims[l];
        w.G[l] = h->g[l];
        w.dW[l] = h->grad + h->w_off[l];
        w.db[l] = h->grad + h->b_off[l];
        w.tile0[l] = blk;
        blk += (w.N[l] / 64) * ((w.M[l] + tc::kBM - 1) / tc::kBM);
        PE_TRY(tc_operand_map(&w.a[l], h->g[l], B, w.M[l], w.M[l], 64));
        PE_TRY(tc_operand_map(&w.b[l], l ? h->a[l - 1] : h->xz, B, w.N[l], w.N[l], 64));
    }
    w.tile0[L] = blk;
    for (int l = 0; l < L; ++l) {
        w.bias0[l] = blk;
        blk += w.M[l] / 64;
    }
    w.bias0[L] = blk;
    w.loss_part = h->loss_part;
    w.nloss = loss_tiles(Dout, B);
    w.loss_scale = 1.0f / ((float)B * (float)Dout);
    w.loss = h->loss;
    w.adam = adam ? 1 : 0;
    w.step = h->step;
    w.corr = h->corr;
    w.b1 = b1;
    w.b2 = b2;
    PE_TRY(launch_dependent(k_mlp_wgrad, dim3(blk + 1), tc::kThreads, tc::TileCfg<64>::kSmemBytes, s, w, h->status));
    ++*launches;
    return PE_OK;
}

// Gradients of the batch rows[0..B) (B pairs from row 0 when null), or, with draw, of the batch of
// the current step of the sequence of seed.
int grad_pass(pe_mlp* h, const float* X, const float* Y, int64_t npairs, const int32_t* rows, bool draw, uint64_t seed,
              int B, int P, double b1, double b2, int* launches)
{
    PE_TRY(launch_dependent(k_prep<float>, dim3(B), 128, 0, h->stream, X, Y, B, h->dims[0], h->dims[h->L], rows,
                            draw ? h->step : nullptr, seed, npairs, P, h->norm, h->norm + h->dmax,
                            h->norm + 2 * h->dmax, h->norm + 3 * h->dmax, h->xz, h->tz));
    ++*launches;
    PE_TRY(forward(h, B, 1, nullptr, nullptr, launches));
    return backward(h, B, draw, b1, b2, launches);
}

int adam_update(pe_mlp* h, float lr, double b1, double b2, float eps)
{
    int blk = 0;
    for (int l = 0; l < h->L; ++l)
        blk += (h->dims[l] / 64) * (h->dims[l + 1] / 64) + (h->dims[l + 1] + 255) / 256;
    return launch_dependent(k_adam, dim3(blk), 256, 0, h->stream, h->p, h->pb, h->pbT, h->wt, h->grad, h->am, h->av,
                            h->corr, lr, b1, b2, eps);
}

}  // namespace

extern "C" PE_API int pe_mlp_layout_for(int32_t nlayers, const int32_t* dims, int32_t max_batch, pe_mlp_layout* out)
{
    if (!out) return PE_EINVAL;
    PE_TRY(check_dims(nlayers, dims, max_batch));
    memset(out, 0, sizeof(*out));
    int64_t np = 0;
    int dmax = 0;
    for (int l = 0; l < nlayers; ++l) np += (int64_t)dims[l + 1] * dims[l] + dims[l + 1];
    for (int l = 0; l <= nlayers; ++l) dmax = std::max(dmax, (int)dims[l]);
    out->nparams = np;
    out->bytes[PE_MLP_PARAMS] = 4 * (size_t)np;
    out->bytes[PE_MLP_PARAMS_BF16] = 2 * 2 * (size_t)np;  // the mirror, then its per-layer transposes
    out->bytes[PE_MLP_GRADS] = 4 * (size_t)np;
    out->bytes[PE_MLP_ADAM_M] = 4 * (size_t)np;
    out->bytes[PE_MLP_ADAM_V] = 4 * (size_t)np;
    out->bytes[PE_MLP_NORM] = 4 * 4 * (size_t)dmax + 8 * 2 * (size_t)dmax + 8 * (size_t)kNormBlocks * dmax + 256 +
                              4 * (size_t)kLossSlots;
    out->bytes[PE_MLP_WORK] = plan_work(nlayers, dims, max_batch).total;
    size_t off = 0;
    for (int b = 0; b < PE_MLP_NBUF; ++b) {
        out->offset[b] = off;
        off += al256(out->bytes[b]);
    }
    out->total_bytes = off;
    return PE_OK;
}

extern "C" PE_API int pe_mlp_create(int32_t nlayers, const int32_t* dims, int32_t max_batch, void* arena,
                                    size_t arena_bytes, void* stream, pe_mlp** out)
{
    if (!out) return PE_EINVAL;
    *out = nullptr;
    pe_mlp_layout lay;
    PE_TRY(pe_mlp_layout_for(nlayers, dims, max_batch, &lay));
    if (!arena || ((uintptr_t)arena & 255u) || arena_bytes < lay.total_bytes) return PE_EINVAL;
    pe_mlp* h = (pe_mlp*)calloc(1, sizeof(pe_mlp));
    if (!h) return PE_EINVAL;
    h->L = nlayers;
    h->dmax = 0;
    for (int l = 0; l <= nlayers; ++l) {
        h->dims[l] = dims[l];
        h->dmax = std::max(h->dmax, (int)dims[l]);
    }
    h->max_batch = max_batch;
    h->nparams = lay.nparams;
    int64_t o = 0;
    for (int l = 0; l < nlayers; ++l) {
        h->w_off[l] = o;
        o += (int64_t)dims[l + 1] * dims[l];
        h->b_off[l] = o;
        o += dims[l + 1];
    }
    h->lay = lay;
    h->arena = (char*)arena;
    h->stream = (cudaStream_t)stream;
    h->p = (float*)(h->arena + lay.offset[PE_MLP_PARAMS]);
    h->pb = (__nv_bfloat16*)(h->arena + lay.offset[PE_MLP_PARAMS_BF16]);
    h->pbT = h->pb + h->nparams;
    h->wt.L = nlayers;
    for (int l = 0; l < nlayers; ++l) {
        h->wt.off[l] = h->w_off[l];
        h->wt.rows[l] = dims[l + 1];
        h->wt.cols[l] = dims[l];
    }
    h->grad = (float*)(h->arena + lay.offset[PE_MLP_GRADS]);
    h->am = (float*)(h->arena + lay.offset[PE_MLP_ADAM_M]);
    h->av = (float*)(h->arena + lay.offset[PE_MLP_ADAM_V]);
    char* nb = h->arena + lay.offset[PE_MLP_NORM];
    h->norm = (float*)nb;
    nb += 4 * 4 * (size_t)h->dmax;
    h->norm64 = (double*)nb;
    nb += 8 * 2 * (size_t)h->dmax;
    h->normpart = (double*)nb;
    nb += 8 * (size_t)kNormBlocks * h->dmax;
    h->step = (int64_t*)nb;
    h->loss = (float*)(nb + 8);
    h->status = (uint32_t*)(nb + 16);
    h->corr = (float*)(nb + 24);
    h->loss_part = (float*)(nb + 256);
    const WorkPlan w = plan_work(nlayers, dims, max_batch);
    char* wb = h->arena + lay.offset[PE_MLP_WORK];
    h->xz = (__nv_bfloat16*)(wb + w.xz);
    for (int l = 0; l + 1 < nlayers; ++l) {
        h->z[l] = (float*)(wb + w.z[l]);
        h->a[l] = (__nv_bfloat16*)(wb + w.a[l]);
    }
    h->tz = (float*)(wb + w.tz);
    for (int l = 0; l < nlayers; ++l) h->g[l] = (__nv_bfloat16*)(wb + w.g[l]);
    *out = h;
    return PE_OK;
}

extern "C" PE_API void pe_mlp_destroy(pe_mlp* h) { free(h); }

extern "C" PE_API int pe_mlp_init(pe_mlp* h, uint64_t seed)
{
    if (!h) return PE_EINVAL;
    ParamTable tab;
    memset(&tab, 0, sizeof(tab));
    for (int l = 0; l < h->L; ++l) {
        const bool last = l == h->L - 1;
        tab.seg[2 * l] = {h->w_off[l], (int64_t)h->dims[l + 1] * h->dims[l],
                          (float)sqrt((last ? 3.0 : 6.0) / h->dims[l])};
        tab.seg[2 * l + 1] = {h->b_off[l], h->dims[l + 1], 0.0f};
    }
    tab.nseg = 2 * h->L;
    cudaStream_t s = h->stream;
    k_mlp_init<<<2 * sm_count(), 256, 0, s>>>(tab, h->wt, seed, h->p, h->pb, h->pbT);
    const size_t nb = 4 * (size_t)h->nparams;
    if (cudaMemsetAsync(h->am, 0, nb, s) != cudaSuccess || cudaMemsetAsync(h->av, 0, nb, s) != cudaSuccess ||
        cudaMemsetAsync(h->grad, 0, nb, s) != cudaSuccess || cudaMemsetAsync(h->step, 0, 32, s) != cudaSuccess)
        return PE_ECUDA;
    // identity normalisation until pe_mlp_fit_norm
    std::vector<float> id(4 * (size_t)h->dmax, 0.0f);
    for (int k = 0; k < h->dmax; ++k) id[h->dmax + k] = id[3 * h->dmax + k] = 1.0f;
    if (cudaMemcpyAsync(h->norm, id.data(), 4 * id.size(), cudaMemcpyHostToDevice, s) != cudaSuccess) return PE_ECUDA;
    if (cudaStreamSynchronize(s) != cudaSuccess) return PE_ECUDA;  // host vector goes out of scope
    return launch_status(1);
}

extern "C" PE_API int pe_mlp_fit_norm(pe_mlp* h, const float* X, const float* Y, int64_t npairs, int32_t period)
{
    if (!h || !X || !Y || npairs < 1) return PE_EINVAL;
    const int D[2] = {h->dims[0], h->dims[h->L]};
    for (int q = 0; q < 2; ++q)
        if (period < 0 || (period > 0 && D[q] % period)) return PE_EINVAL;
    cudaStream_t s = h->stream;
    const int nparts = (int)std::min<int64_t>(kNormBlocks, npairs);
    for (int q = 0; q < 2; ++q) {
        const float* src = q ? Y : X;
        float* mu32 = h->norm + (2 * q) * h->dmax;
        float* sd32 = h->norm + (2 * q + 1) * h->dmax;
        dim3 grid((D[q] + 255) / 256, nparts);
        k_norm_partial<float><<<grid, 256, 0, s>>>(src, npairs, D[q], nullptr, h->normpart);
        k_norm_final<<<1, 1024, 0, s>>>(h->normpart, nparts, D[q], period, npairs, 0, h->norm64, mu32);
        k_norm_partial<float><<<grid, 256, 0, s>>>(src, npairs, D[q], h->norm64, h->normpart);
        k_norm_final<<<1, 1024, 0, s>>>(h->normpart, nparts, D[q], period, npairs, 1, h->norm64, sd32);
    }
    h->shift_period = period;
    return launch_status(8);
}

extern "C" PE_API int pe_mlp_forward(pe_mlp* h, const void* x, int32_t x_is_f64, int32_t B, void* y, int32_t y_is_f64)
{
    if (!h || !x || !y || B < 1 || B > h->max_batch) return PE_EINVAL;
    cudaStream_t s = h->stream;
    const int D = h->dims[0];
    const int32_t* no_rows = nullptr;
    const int64_t* no_step = nullptr;
    const float* no_f = nullptr;
    float* no_t = nullptr;
    if (x_is_f64)
        PE_TRY(launch_dependent(k_prep<double>, dim3(B), 128, 0, s, (const double*)x, no_f, B, D, 0, no_rows, no_step,
                                uint64_t(0), int64_t(0), 0, h->norm, h->norm + h->dmax, no_f, no_f, h->xz, no_t));
    else
        PE_TRY(launch_dependent(k_prep<float>, dim3(B), 128, 0, s, (const float*)x, no_f, B, D, 0, no_rows, no_step,
                                uint64_t(0), int64_t(0), 0, h->norm, h->norm + h->dmax, no_f, no_f, h->xz, no_t));
    int launches = 1;
    PE_TRY(forward(h, B, 0, y_is_f64 ? nullptr : (float*)y, y_is_f64 ? (double*)y : nullptr, &launches));
    return launch_status(launches);
}

extern "C" PE_API int pe_mlp_grad(pe_mlp* h, const float* X, const float* Y, int64_t npairs, const int32_t* rows,
                                  int32_t B, float* loss)
{
    if (!h || !X || !Y || B < 32 || B % 32 || B > h->max_batch || (!rows && npairs < B)) return PE_EINVAL;
    if (loss_tiles(h->dims[h->L], B) > kLossSlots) return PE_EINVAL;
    int launches = 0;
    PE_TRY(grad_pass(h, X, Y, npairs, rows, false, 0, B, 0, 0.0, 0.0, &launches));
    if (loss && cudaMemcpyAsync(loss, h->loss, 4, cudaMemcpyDeviceToDevice, h->stream) != cudaSuccess) return PE_ECUDA;
    return launch_status(launches);
}

extern "C" PE_API int pe_mlp_adam(pe_mlp* h, double lr, double beta1, double beta2, double eps)
{
    if (!h || !(lr >= 0.0) || !(beta1 >= 0.0 && beta1 < 1.0) || !(beta2 >= 0.0 && beta2 < 1.0) || !(eps > 0.0))
        return PE_EINVAL;
    cudaStream_t s = h->stream;
    k_adam_begin<<<1, 32, 0, s>>>(h->step, h->corr, beta1, beta2);
    PE_TRY(adam_update(h, (float)lr, beta1, beta2, (float)eps));
    return launch_status(2);
}

extern "C" PE_API int pe_mlp_train(pe_mlp* h, const float* X, const float* Y, int64_t npairs, int32_t B,
                                   int32_t shift_period, uint64_t seed, int32_t nsteps, float lr, float* loss)
{
    if (!h || !X || !Y || npairs < 1 || npairs >= (int64_t(1) << 31) || nsteps < 0 || B < 32 || B % 32 ||
        B > h->max_batch || !(lr >= 0.0f))
        return PE_EINVAL;
    const int D = h->dims[0], Dout = h->dims[h->L];
    if (shift_period < 0 || (shift_period > 0 && (D % shift_period || Dout % shift_period))) return PE_EINVAL;
    if (loss_tiles(Dout, B) > kLossSlots) return PE_EINVAL;
    cudaStream_t s = h->stream;
    (void)sm_count();  // cached before any capture
    int launches = 0, rc = PE_OK;
    auto one_step = [&]() {
        if (rc == PE_OK) rc = grad_pass(h, X, Y, npairs, nullptr, true, seed, B, shift_period, 0.9, 0.999, &launches);
        if (rc == PE_OK) rc = adam_update(h, lr, 0.9, 0.999, 1e-8f);
        ++launches;
    };
    // One step captured as a graph and replayed (the step counter on the device advances the
    // sampling and the bias correction); on the legacy default stream the steps run eagerly.
    cudaGraph_t graph = nullptr;
    cudaGraphExec_t exec = nullptr;
    bool captured = false;
    if (s != nullptr && nsteps > 1 && cudaStreamBeginCapture(s, cudaStreamCaptureModeThreadLocal) == cudaSuccess) {
        one_step();
        if (cudaStreamEndCapture(s, &graph) == cudaSuccess && graph && rc == PE_OK &&
            cudaGraphInstantiate(&exec, graph, 0) == cudaSuccess)
            captured = true;
        else
            cudaGetLastError();
    }
    rc = PE_OK;
    const int per_step = launches;
    if (captured) {
        for (int i = 0; i < nsteps; ++i)
            if (cudaGraphLaunch(exec, s) != cudaSuccess) {
                cudaGraphExecDestroy(exec);
                cudaGraphDestroy(graph);
                return PE_ECUDA;
            }
        cudaGraphExecDestroy(exec);
        cudaGraphDestroy(graph);
        note_launches(per_step * nsteps);
    } else {
        if (graph) cudaGraphDestroy(graph);
        launches = 0;
        for (int i = 0; i < nsteps && rc == PE_OK; ++i) one_step();
        if (rc != PE_OK) return rc;
        if (cudaGetLastError() != cudaSuccess) return PE_ECUDA;
        note_launches(launches);
    }
    if (loss && cudaMemcpyAsync(loss, h->loss, 4, cudaMemcpyDeviceToDevice, s) != cudaSuccess) return PE_ECUDA;
    return PE_OK;
}

extern "C" PE_API int pe_mlp_sync_status(pe_mlp* h)
{
    if (!h) return PE_EINVAL;
    uint32_t st = 0;
    if (cudaStreamSynchronize(h->stream) != cudaSuccess) return PE_ECUDA;
    if (cudaMemcpy(&st, h->status, sizeof(st), cudaMemcpyDeviceToHost) != cudaSuccess) return PE_ECUDA;
    if (cudaMemset(h->status, 0, sizeof(st)) != cudaSuccess) return PE_ECUDA;
    return (st & PE_FLAG_TIMEOUT) ? PE_ETIMEOUT : PE_OK;
}

extern "C" PE_API int pe_mlp_info(const pe_mlp* h, int64_t* nparams, int64_t* steps_device_ptr, void** params,
                                  void** grads)
{
    if (!h) return PE_EINVAL;
    if (nparams) *nparams = h->nparams;
    if (steps_device_ptr) *steps_device_ptr = (int64_t)(uintptr_t)h->step;
    if (params) *params = h->p;
    if (grads) *grads = h->grad;
    return PE_OK;
}

// ------------------------------------------------------------------ gated surrogate step

namespace pe {
namespace {

using GateResult = pe_gate_result;

// Probe slope s_p and standard error sigma_i of every coefficient (line fit of the samples
// c_0..c_Ks at t_p = p dt), the gate decision, and on acceptance the leap
// c <- c_Ks + (dT - Ks dt) s_mlp (slope <- s_mlp). The estimated error is the relative change
// of the projected state, e = leap ||s_mlp - s_p|| / ||c_Ks||, accepted when
// e <= max(tol, nsig leap ||sigma|| / ||c_Ks||). One block, fixed summation order.
__global__ void __launch_bounds__(1024) k_gate(const double* __restrict__ cs, int Ks, int n, double dt, double dT,
                                              const double* __restrict__ s_mlp, double tol, double nsig,
                                              double* __restrict__ coarse, double* __restrict__ slope,
                                              GateResult* __restrict__ res)
{
    __shared__ double red[4][32];
    __shared__ int acc;
    const double tbar = 0.5 * Ks * dt;
    const double leap = dT - Ks * dt;
    double sxx = 0.0;
    for (int p = 0; p <= Ks; ++p) sxx += (p * dt - tbar) * (p * dt - tbar);
    double e2 = 0.0, n2 = 0.0, v2 = 0.0, c2 = 0.0;
    for (int i = threadIdx.x; i < n; i += blockDim.x) {
        double ybar = 0.0;
        for (int p = 0; p <= Ks; ++p) ybar += cs[(size_t)p * n + i];
        ybar /= (double)(Ks + 1);
        double sxy = 0.0;
        for (int p = 0; p <= Ks; ++p) sxy += (p * dt - tbar) * (cs[(size_t)p * n + i] - ybar);
        const double sp = sxy / sxx;
        double r2 = 0.0;
        for (int p = 0; p <= Ks; ++p) {
            const double r = cs[(size_t)p * n + i] - (ybar + sp * (p * dt - tbar));
            r2 += r * r;
        }
        const double d = s_mlp[i] - sp;
        const double cl = cs[(size_t)Ks * n + i];
        e2 += d * d;
        n2 += sp * sp;
        v2 += r2 / (double)(Ks - 1) / sxx;
        c2 += cl * cl;
    }
    e2 = warp_sum(e2);
    n2 = warp_sum(n2);
    v2 = warp_sum(v2);
    c2 = warp_sum(c2);
    const int lane = threadIdx.x & 31, w = threadIdx.x >> 5;
    if (lane == 0) {
        red[0][w] = e2;
        red[1][w] = n2;
        red[2][w] = v2;
        red[3][w] = c2;
    }
    __syncthreads();
    if (threadIdx.x == 0) {
        double a = 0.0, b = 0.0, c = 0.0, d = 0.0;
        for (int k = 0; k < (int)(blockDim.x >> 5); ++k) {
            a += red[0][k];
            b += red[1][k];
            c += red[2][k];
            d += red[3][k];
        }
        const double cn = sqrt(d);
        GateResult r;
        r.err = cn > 0.0 ? leap * sqrt(a) / cn : INFINITY;
        r.floor = fmax(tol, cn > 0.0 ? nsig * leap * sqrt(c) / cn : 0.0);
        r.norm = sqrt(b);
        r.sigma = sqrt(c);
        r.accepted = (r.err <= r.floor) ? 1 : 0;
        r.pad = 0;
        *res = r;
        acc = r.accepted;
    }
    __syncthreads();
    if (acc) {
        for (int i = threadIdx.x; i < n; i += blockDim.x) {
            coarse[i] = fma(leap, s_mlp[i], cs[(size_t)Ks * n + i]);
            slope[i] = s_mlp[i];
        }
    }
}

__global__ void k_to_f32(const double* __restrict__ src, int n, float* __restrict__ dst)
{
    const int i = blockIdx.x * blockDim.x + threadIdx.x;
    if (i < n) dst[i] = (float)src[i];
}

}  // namespace
}  // namespace pe

extern "C" PE_API int pe_step_surrogate(pe_ctx* ctx, pe_mlp* h, const pe_gate_cfg* gc, pe_gate_stats* out)
{
    NvtxRange nvtx("pe_step_surrogate");
    if (!ctx || !h || !gc || !out) return PE_EINVAL;
    pe_ctx* x = ctx;
    const pe_config& c = x->cfg;
    const int n = 2 * x->nc, Ks = gc->K_probe;
    if (x->ps || x->pres) return PE_EINVAL;  // the surrogate maps the density and momentum coefficients
    if (x->te_active) return PE_EINVAL;  // an accepted leap would not project the electrons' energy
    if (h->dims[0] != n || h->dims[h->L] != n || Ks < 2 || Ks >= x->K_cur || !(gc->tol >= 0.0) ||
        !(gc->noise_sigmas >= 0.0))
        return PE_EINVAL;
    char* buf = x->arena + x->lay.offset[PE_BUF_SURROGATE];
    double* s_mlp = (double*)buf;
    GateResult* res = (GateResult*)(buf + al256(8 * (size_t)n));
    // the learned slope from the coarse state at the start of the step, on the context stream
    const cudaStream_t saved = h->stream;
    h->stream = x->stream;
    const int rc = pe_mlp_forward(h, x->coarse, 1, 1, s_mlp, 1);
    h->stream = saved;
    PE_TRY(rc);
    if (!x->fresh) PE_TRY(pe_lift(x));
    PE_TRY(pe_ctx_burst_range(x, 0, Ks, 1));
    PE_TRY(pe_coarsen(x->samples, Ks + 1, c.ncell, x->s_w, x->s_p, c.wavelet, x->nc, x->bin_shift, x->csamples,
                      x->stream));
    PE_TRY(pe_gate(x->csamples, Ks, n, c.dt, x->dT_cur, s_mlp, gc->tol, gc->noise_sigmas, x->coarse, x->slope, res,
                   x->stream));
    GateResult r;
    if (cudaMemcpyAsync(&r, res, sizeof(r), cudaMemcpyDeviceToHost, x->stream) != cudaSuccess ||
        cudaStreamSynchronize(x->stream) != cudaSuccess)
        return PE_ECUDA;
    memset(out, 0, sizeof(*out));
    out->accepted = r.accepted;
    out->err = r.err;
    out->floor = r.floor;
    out->norm = r.norm;
    out->sigma = r.sigma;
    if (r.accepted) {
        out->fine_steps = Ks;
        x->macro_steps += 1;
        x->coarse_state = 1;
        x->time += x->dT_cur;
        x->fresh = 0;
        return PE_OK;
    }
    out->fine_steps = x->K_cur;
    PE_TRY(pe_ctx_burst_range(x, Ks, x->K_cur, 1));
    PE_TRY(pe_restrict(x));
    return pe_project(x);
}

extern "C" PE_API int pe_gate(const double* samples, int32_t K_probe, int32_t ncoef, double dt, double dT,
                               const double* s_mlp, double tol, double noise_sigmas, double* coarse, double* slope,
                               pe_gate_result* result, void* stream)
{
    if (!samples || !s_mlp || !coarse || !slope || !result || K_probe < 2 || ncoef < 1 || !(dt > 0.0) ||
        !(tol >= 0.0) || !(noise_sigmas >= 0.0))
        return PE_EINVAL;
    k_gate<<<1, 1024, 0, (cudaStream_t)stream>>>(samples, K_probe, ncoef, dt, dT, s_mlp, tol, noise_sigmas, coarse,
                                                 slope, result);
    return launch_status(1);
}

extern "C" PE_API int pe_export_f32(pe_ctx* ctx, int32_t what, float* out)
{
    if (!ctx || !out || (what != 0 && what != 1)) return PE_EINVAL;
    const int n = (int)ctx->ncoef;
    k_to_f32<<<(n + 255) / 256, 256, 0, ctx->stream>>>(what ? ctx->slope : ctx->coarse, n, out);
    return launch_status(1);
}

namespace pe {
namespace {
__global__ void k_set_params(const float* __restrict__ src, int64_t n, float* __restrict__ p,
                             __nv_bfloat16* __restrict__ pb, __nv_bfloat16* __restrict__ pbT, WeightTable wt)
{
    for (int64_t i = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; i < n; i += (int64_t)gridDim.x * blockDim.x) {
        const float w = src[i];
        p[i] = w;
        put_bf16(wt, i, w, pb, pbT);
    }
}
}  // namespace
}  // namespace pe

extern "C" PE_API int pe_mlp_set_params(pe_mlp* h, const float* params)
{
    if (!h || !params) return PE_EINVAL;
    k_set_params<<<2 * sm_count(), 256, 0, h->stream>>>(params, h->nparams, h->p, h->pb, h->pbT, h->wt);
    return launch_status(1);
}
