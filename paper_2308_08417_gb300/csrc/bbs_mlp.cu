// Learned initial guess for time-stepped batches: a small MLP that predicts
// each system's change of solution from its diagonal, right-hand side and
// previous solution, trained and run on the GPU by this file's kernels
// (BF16 tensor-core GEMMs with FP32 accumulation -- tcgen05 MMAs with the
// accumulator in tensor memory by default, mma.sync as the alternative --
// FP32 master weights, Adam).
// The paper has no such network; it motivates it: the solver accepts an
// initial guess (Sec. 2.1), and a better guess means fewer iterations.
//
// Network: 3n inputs (standardised diag(A), b, x_prev) -> H -> H -> H -> n,
// GELU (tanh form) after each hidden layer; output = standardised dx; the
// predicted initial guess is x_prev + dx * sigma + mu. Loss: mean squared
// error over the outputs. Weights W_l are [out, in] (y = x W^T + b).
//
// Storage (all owned by the bbs_mlp object):
//   master FP32 parameters, flat: W1 b1 W2 b2 W3 b3 W4 b4 (W row-major)
//   BF16 copies W_l [out, in_pad] (K-major, forward) and W_l^T [in, out_pad]
//   (K-major for the input-gradient GEMM), zero-padded to multiples of 32
//   activations of a minibatch: row-major and transposed BF16 copies (the
//   transposed ones feed the weight-gradient GEMMs, which reduce over rows)
#include <algorithm>
#include <cmath>
#include <cstdarg>
#include <cstdio>
#include <cstring>
#include <vector>

#include <cuda.h>
#include <cuda_bf16.h>
#include <cuda_runtime.h>
#include <cudaTypedefs.h>

#include "../../include/bbs.h"
#include "bbs_internal.h"
#include "bbs_mlp_gemm.cuh"
#include "bbs_umma.cuh"

namespace bbs {
namespace mlp {

constexpr int kLayers = 4;
constexpr float kGeluC = 0.044715f;
constexpr float kSqrt2OverPi = 0.7978845608028654f;

__device__ __forceinline__ float gelu(float z) {
    return 0.5f * z * (1.0f + tanhf(kSqrt2OverPi * (z + kGeluC * z * z * z)));
}
__device__ __forceinline__ float gelu_grad(float z) {
    const float t = tanhf(kSqrt2OverPi * (z + kGeluC * z * z * z));
    const float du = kSqrt2OverPi * (1.0f + 3.0f * kGeluC * z * z);
    return 0.5f * (1.0f + t) + 0.5f * z * (1.0f - t * t) * du;
}

// Sum over a block of 256 threads, in a tree; thread 0 has it.
__device__ __forceinline__ float block_tree_sum(float s) {
    for (int k = 16; k; k >>= 1) s += __shfl_xor_sync(0xffffffffu, s, k);
    __shared__ float ws[8];
    if ((threadIdx.x & 31) == 0) ws[threadIdx.x >> 5] = s;
    __syncthreads();
    return ((ws[0] + ws[1]) + (ws[2] + ws[3])) + ((ws[4] + ws[5]) + (ws[6] + ws[7]));
}

// ---------------------------------------------------------- epilogues

enum EpiMode { EPI_F32 = 0, EPI_BIAS_GELU = 1, EPI_BIAS = 2, EPI_GELU_BWD = 3, EPI_LOSS = 4 };

struct Epi {
    int mode;
    float* c;                 // EPI_F32 / EPI_BIAS: output; EPI_BIAS_GELU: pre-activation store
    int ldc;
    size_t zstride;           // EPI_F32: split-K part z goes to c + z * zstride
    const float* bias;        // EPI_BIAS_GELU / EPI_BIAS
    __nv_bfloat16* y;         // BF16 row-major output (EPI_BIAS_GELU, EPI_GELU_BWD)
    int ldy;
    __nv_bfloat16* yt;        // BF16 transposed output, may be null
    int ldyt;
    const float* z;           // EPI_GELU_BWD: pre-activation of the layer below; EPI_LOSS: targets
    int ldz;
    float* loss;              // EPI_LOSS: the tile's sum of squared errors, one per block

    // One element; the mma.sync GEMM calls it (no split, no EPI_LOSS).
    __device__ __forceinline__ void operator()(int m, int n, float v) const {
        switch (mode) {
            case EPI_F32:
                c[(size_t)m * ldc + n] = v;
                break;
            case EPI_BIAS:
                c[(size_t)m * ldc + n] = v + bias[n];
                break;
            case EPI_BIAS_GELU: {
                const float zz = v + bias[n];
                c[(size_t)m * ldc + n] = zz;
                const __nv_bfloat16 h = __float2bfloat16_rn(gelu(zz));
                y[(size_t)m * ldy + n] = h;
                if (yt) yt[(size_t)n * ldyt + m] = h;
                break;
            }
            default: {  // EPI_GELU_BWD
                const __nv_bfloat16 g = __float2bfloat16_rn(v * gelu_grad(z[(size_t)m * ldz + n]));
                y[(size_t)m * ldy + n] = g;
                if (yt) yt[(size_t)n * ldyt + m] = g;
                break;
            }
        }
    }

    // Rows r0, r0 + step, ... of one column of the tile (lanes are
    // neighbouring columns), eight rows' loads in flight at a time. With yt
    // the BF16 result takes the accumulator's place in the tile.
    template <int MODE>
    __device__ __forceinline__ float column(float* t, int ld, int r0, int step, int c0, int m0, int n0, int M,
                                            int bz) const {
        constexpr int kU = 8;
        const int n = n0 + c0;
        const float bn = MODE == EPI_F32 || MODE == EPI_GELU_BWD ? 0.0f : bias[n];
        const float scale = MODE == EPI_LOSS ? 2.0f / ((float)M * (float)ldc) : 0.0f;
        float acc = 0.0f;
        for (int i = r0; i < umma::kBM; i += kU * step) {
            float in[kU];
            if (MODE == EPI_GELU_BWD || MODE == EPI_LOSS) {
#pragma unroll
                for (int u = 0; u < kU; ++u) {
                    const int m = m0 + i + u * step;
                    in[u] = m < M ? __ldg(z + (size_t)m * ldz + n) : 0.0f;
                }
            }
#pragma unroll
            for (int u = 0; u < kU; ++u) {
                const int r = i + u * step, m = m0 + r;
                if (m >= M) continue;
                float* at = t + r * ld + c0;
                float v = *at + bn;
                if (MODE == EPI_F32) {
                    c[(size_t)bz * zstride + (size_t)m * ldc + n] = v;
                } else if (MODE == EPI_BIAS) {
                    c[(size_t)m * ldc + n] = v;
                } else {
                    if (MODE == EPI_BIAS_GELU) {
                        c[(size_t)m * ldc + n] = v;
                        v = gelu(v);
                    } else if (MODE == EPI_GELU_BWD) {
                        v *= gelu_grad(in[u]);
                    } else {
                        const float diff = v - in[u];
                        acc += diff * diff;
                        v = diff * scale;
                    }
                    const __nv_bfloat16 h = __float2bfloat16_rn(v);
                    y[(size_t)m * ldy + n] = h;
                    if (yt) *reinterpret_cast<__nv_bfloat16*>(at) = h;
                }
            }
        }
        return acc;
    }

    // The epilogue of a whole 128 x BN tile t (row stride BN + 1), by all
    // threads of the block.
    __device__ __forceinline__ void tile(float* t, int BN, int m0, int n0, int M, int N, int bz) const {
        const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31, ld = BN + 1;
        float acc = 0.0f;
        const bool pair = BN == 16;  // a warp then takes two rows at a time
        const int r0 = pair ? 2 * warp + (lane >> 4) : warp, step = (pair ? 2 : 1) * (umma::kThreads / 32);
        for (int c0 = pair ? lane & 15 : lane; c0 < BN && n0 + c0 < N; c0 += 32) {
            switch (mode) {
                case EPI_F32: column<EPI_F32>(t, ld, r0, step, c0, m0, n0, M, bz); break;
                case EPI_BIAS: column<EPI_BIAS>(t, ld, r0, step, c0, m0, n0, M, bz); break;
                case EPI_BIAS_GELU: column<EPI_BIAS_GELU>(t, ld, r0, step, c0, m0, n0, M, bz); break;
                case EPI_GELU_BWD: column<EPI_GELU_BWD>(t, ld, r0, step, c0, m0, n0, M, bz); break;
                default: acc += column<EPI_LOSS>(t, ld, r0, step, c0, m0, n0, M, bz); break;
            }
        }
        if (mode == EPI_LOSS) {
            acc = block_tree_sum(acc);
            if (threadIdx.x == 0) loss[blockIdx.y * gridDim.x + blockIdx.x] = acc;
        }
        if (yt == nullptr) return;  // the same for every thread
        __syncthreads();
        const int wide = (ldyt & 1) == 0;  // pairs of rows are then 4-byte aligned (m0 and r are even)
        for (int j = warp; j < BN && n0 + j < N; j += umma::kThreads / 32)
            for (int r = 2 * lane; r < umma::kBM && m0 + r < M; r += 64) {
                const __nv_bfloat16 lo = *reinterpret_cast<const __nv_bfloat16*>(t + r * ld + j);
                const __nv_bfloat16 hi = *reinterpret_cast<const __nv_bfloat16*>(t + (r + 1) * ld + j);
                __nv_bfloat16* to = yt + (size_t)(n0 + j) * ldyt + m0 + r;
                if (wide && m0 + r + 1 < M) {
                    *reinterpret_cast<__nv_bfloat162*>(to) = __nv_bfloat162(lo, hi);
                } else {
                    to[0] = lo;
                    if (m0 + r + 1 < M) to[1] = hi;
                }
            }
    }
};

__global__ void __launch_bounds__(256) gemm_kernel(const __nv_bfloat16* __restrict__ A, int lda,
                                                   const __nv_bfloat16* __restrict__ B, int ldb, int M,
                                                   int N, int K, Epi epi) {
    gemm_tn_mma<Epi>(A, lda, B, ldb, M, N, K, epi);
}

// [4096 x 256] from K = 256 with GELU: 36 -> 10 us; with the GELU gradient
// 28 -> 11 us (one launch from cold caches). What is left is latency: launch,
// copies, one wave of 256 blocks' epilogues. Launches overlap in a step (the
// next kernel sets up while this one runs): 138 -> 103 us with the narrower
// tiles and the sums below.
__global__ void __launch_bounds__(umma::kThreads, 2) gemm_umma_kernel(const __grid_constant__ CUtensorMap ta,
                                                                      const __grid_constant__ CUtensorMap tb, int M,
                                                                      int N, int K, int BN, int ktiles_per_split,
                                                                      Epi epi, int* err) {
    umma::gemm_tn_tma<Epi>(&ta, &tb, M, N, K, BN, blockIdx.x, blockIdx.y, blockIdx.z, ktiles_per_split, epi, err);
}

// The weight gradients of all layers, C_l = A_l B_l^T over the same K (the
// minibatch), in one launch: each alone is 8 to 14 tiles and was split 16-fold
// only to fill the chip for 11 to 20 us a layer. They wait for nothing but the
// output gradients, which are all there by the end of the backward chain.
// The splits are those of the single GEMM, so the sums are the same. 57 us of
// GEMMs and 24 us of sums -> 17 and 12 us.
struct WeightGrads {
    CUtensorMap a[kLayers], b[kLayers];
    int M[kLayers], N[kLayers], BN[kLayers], kps[kLayers], nt[kLayers], mt[kLayers];
    int first[kLayers + 1];  // first block of each
    Epi epi[kLayers];
};

__global__ void __launch_bounds__(umma::kThreads, 2) weight_grads_kernel(const __grid_constant__ WeightGrads w, int K,
                                                                         int* err) {
    int l = 0;
    while (l + 1 < kLayers && (int)blockIdx.x >= w.first[l + 1]) ++l;
    int t = blockIdx.x - w.first[l];
    const int bx = t % w.nt[l];
    t /= w.nt[l];
    umma::gemm_tn_tma<Epi>(&w.a[l], &w.b[l], w.M[l], w.N[l], K, w.BN[l], bx, t % w.mt[l], t / w.mt[l], w.kps[l],
                           w.epi[l], err);
}

// c[m][n] = sum over the splits of part[z][m][n] (split-K, fixed order).
__global__ void splitk_reduce_kernel(int M, int N, int splits, const float* __restrict__ part, float* __restrict__ c,
                                     int ldc) {
    const size_t total = (size_t)M * N;
    for (size_t i = (size_t)blockIdx.x * blockDim.x + threadIdx.x; i < total; i += (size_t)gridDim.x * blockDim.x) {
        float s = 0.0f;
        for (int z = 0; z < splits; ++z) s += part[(size_t)z * total + i];
        c[(i / N) * ldc + i % N] = s;
    }
}

struct Layers {
    int off_W[kLayers], off_b[kLayers], out[kLayers], in[kLayers], in_pad[kLayers], out_pad[kLayers];
    __nv_bfloat16 *Wb[kLayers], *WTb[kLayers];
};

struct Adam {
    float *p, *m, *v;
    float lr, b1, b2, eps, c1, c2;
};

// One parameter's step and, of a weight, the BF16 copies of what it becomes
// (their pads stay zero). Element e of layer l, parameter i in all.
__device__ __forceinline__ void adam_update(const Adam& a, const Layers& w, int l, int e, int i, float gi) {
    const float mi = a.b1 * a.m[i] + (1.0f - a.b1) * gi;
    const float vi = a.b2 * a.v[i] + (1.0f - a.b2) * gi * gi;
    a.m[i] = mi;
    a.v[i] = vi;
    const float pi = a.p[i] - a.lr * (mi / a.c1) / (sqrtf(vi / a.c2) + a.eps);
    a.p[i] = pi;
    if (i < w.off_b[l]) {
        const int r = e / w.in[l], k = e - r * w.in[l];
        const __nv_bfloat16 h = __float2bfloat16_rn(pi);
        w.Wb[l][(size_t)r * w.in_pad[l] + k] = h;
        w.WTb[l][(size_t)k * w.out_pad[l] + r] = h;
    }
}

// What is left of all layers' gradients, in one launch, and with ADAM the
// step that they are for:
//   * blocks below first[0]: one thread per weight adds its split-K parts
//     (splits <= 1: the GEMM has left the gradient in g);
//   * then one block per output: the bias gradient db[j] = sum of row j of dT
//     [N, M]. One warp a row with 2-byte loads took 10 us a layer, most of it
//     waiting; a block reads the row in one or two 16-byte loads per thread
//     (M is a multiple of 64) and adds in a tree, so its chains are shorter;
//   * with loss_parts, a last block that adds the tiles' losses, in a tree too
//     (an atomic per row into one FP32 sum was less exact, and its last bits
//     changed from run to run).
// As eight launches of sums, one of Adam and four that packed the BF16 weights
// this took 81 us a step of n = 144, hidden 256, M = 4096, nearly all of it
// launches and latency: 12 us now, from cold caches.
struct GradSums {
    Layers w;
    float* g;
    int count;
    const float* part[kLayers];
    int splits[kLayers];
    const __nv_bfloat16* dT[kLayers];
    int first[kLayers + 1];  // first bias block of each layer
    const float* loss_part;
    int loss_parts;
    float* loss;
};

template <bool ADAM>
__global__ void __launch_bounds__(256) grad_sums_kernel(const __grid_constant__ GradSums g, int M, Adam a) {
    umma::grid_wait();
    if ((int)blockIdx.x < g.first[0]) {
        for (int i = blockIdx.x * blockDim.x + threadIdx.x; i < g.count; i += g.first[0] * blockDim.x) {
            int l = 0;
            while (l + 1 < kLayers && i >= g.w.off_W[l + 1]) ++l;
            if (i >= g.w.off_b[l]) continue;
            const int e = i - g.w.off_W[l], total = g.w.off_b[l] - g.w.off_W[l], splits = g.splits[l];
            float s = 0.0f;
            if (splits > 1) {
                const float* __restrict__ part = g.part[l] + e;
#pragma unroll 8
                for (int z = 0; z < splits; ++z) s += __ldg(part + (size_t)z * total);
                g.g[i] = s;
            } else if (ADAM) {
                s = g.g[i];
            }
            if (ADAM) adam_update(a, g.w, l, e, i, s);
        }
        return;
    }
    if ((int)blockIdx.x >= g.first[kLayers]) {
        float s = 0.0f;
        for (int i = threadIdx.x; i < g.loss_parts; i += blockDim.x) s += g.loss_part[i];
        s = block_tree_sum(s);
        if (threadIdx.x == 0) *g.loss = s / ((float)M * (float)g.w.out[kLayers - 1]);
        return;
    }
    int l = 0;
    while (l + 1 < kLayers && (int)blockIdx.x >= g.first[l + 1]) ++l;
    const int j = blockIdx.x - g.first[l];
    const uint4* row = reinterpret_cast<const uint4*>(g.dT[l] + (size_t)j * M);
    float s = 0.0f;
    for (int i = threadIdx.x; i < M / 8; i += blockDim.x) {
        const uint4 q = __ldg(row + i);
        const uint32_t w[4] = {q.x, q.y, q.z, q.w};
        float p[4];
#pragma unroll
        for (int k = 0; k < 4; ++k) {
            const float2 f = __bfloat1622float2(reinterpret_cast<const __nv_bfloat162&>(w[k]));
            p[k] = f.x + f.y;
        }
        s += (p[0] + p[1]) + (p[2] + p[3]);
    }
    s = block_tree_sum(s);
    if (threadIdx.x == 0) {
        const int i = g.w.off_b[l] + j;
        g.g[i] = s;
        if (ADAM) adam_update(a, g.w, l, 0, i, s);
    }
}

// ---------------------------------------------------- small kernels

// Per-feature (3n inputs) and per-output (n) first and second moments of one
// time step's samples, accumulated in FP64: inputs diag(A), b, x_prev;
// outputs x_next - x_prev.
__global__ void observe_kernel(int num_batch, int n, const int32_t* __restrict__ row_ptrs,
                               const int32_t* __restrict__ cols, const double* __restrict__ values,
                               int nnz, const double* __restrict__ b, const double* __restrict__ xp,
                               const double* __restrict__ xn, double* __restrict__ sums,
                               double* __restrict__ sumsq) {
    const int F = 4 * n;
    const int f = blockIdx.x * blockDim.x + threadIdx.x;
    if (f >= F) return;
    double s = 0.0, s2 = 0.0;
    for (int i = blockIdx.y; i < num_batch; i += gridDim.y) {
        double v;
        if (f < n) {
            v = 0.0;
            for (int e = row_ptrs[f]; e < row_ptrs[f + 1]; ++e)
                if (cols[e] == f) v = values[(size_t)i * nnz + e];
        } else if (f < 2 * n) {
            v = b[(size_t)i * n + f - n];
        } else if (f < 3 * n) {
            v = xp[(size_t)i * n + f - 2 * n];
        } else {
            v = xn[(size_t)i * n + f - 3 * n] - xp[(size_t)i * n + f - 3 * n];
        }
        s += v;
        s2 += v * v;
    }
    atomicAdd(sums + f, s);
    atomicAdd(sumsq + f, s2);
}

__global__ void finalize_stats_kernel(int F, double count, const double* sums, const double* sumsq,
                                      float* mean, float* inv_std, float* stdv) {
    const int f = blockIdx.x * blockDim.x + threadIdx.x;
    if (f >= F) return;
    const double mu = sums[f] / count;
    const double var = fmax(sumsq[f] / count - mu * mu, 0.0);
    // a (numerically) constant quantity is centred but not scaled
    const double sd = var > 1e-12 * (mu * mu) + 1e-300 ? sqrt(var) : 1.0;
    mean[f] = (float)mu;
    stdv[f] = (float)sd;
    inv_std[f] = (float)(1.0 / sd);
}

// Standardised BF16 features [M, in_pad] (columns >= 3n zero) and, when xn is
// given, standardised FP32 targets [M, n].
__global__ void samples_kernel(int num_batch, int n, int in_pad, const int32_t* __restrict__ row_ptrs,
                               const int32_t* __restrict__ cols, const double* __restrict__ values, int nnz,
                               const double* __restrict__ b, const double* __restrict__ xp,
                               const double* __restrict__ xn, const float* __restrict__ mean,
                               const float* __restrict__ inv_std, __nv_bfloat16* __restrict__ feats,
                               float* __restrict__ targets) {
    const int i = blockIdx.x;
    for (int f = threadIdx.x; f < in_pad; f += blockDim.x) {
        float out = 0.0f;
        if (f < 3 * n) {
            double v;
            if (f < n) {
                v = 0.0;
                for (int e = row_ptrs[f]; e < row_ptrs[f + 1]; ++e)
                    if (cols[e] == f) v = values[(size_t)i * nnz + e];
            } else if (f < 2 * n) {
                v = b[(size_t)i * n + f - n];
            } else {
                v = xp[(size_t)i * n + f - 2 * n];
            }
            out = (float)((v - (double)mean[f]) * (double)inv_std[f]);
        }
        feats[(size_t)i * in_pad + f] = __float2bfloat16_rn(out);
    }
    if (xn != nullptr)
        for (int k = threadIdx.x; k < n; k += blockDim.x) {
            const int f = 3 * n + k;
            const double d = xn[(size_t)i * n + k] - xp[(size_t)i * n + k];
            targets[(size_t)i * n + k] = (float)((d - (double)mean[f]) * (double)inv_std[f]);
        }
}

// Minibatch gather: rows idx[r] of the sample store into X [M, in_pad] and
// X^T [in_pad, M], targets into T [M, n]; clears the loss. One block moves 64
// rows by 64 features through shared memory (M and in_pad are multiples of
// 64), so that both copies are written in whole lines: a block per row wrote
// X^T two bytes a line, 21 us for 4096 x 448 (now 8). The store is the
// caller's; `wide` says that it is 16-byte aligned.
__global__ void __launch_bounds__(256) gather_kernel(int M, int in_pad, int n, const int32_t* __restrict__ idx,
                                                     const __nv_bfloat16* __restrict__ feats,
                                                     const float* __restrict__ targets, bool wide,
                                                     __nv_bfloat16* __restrict__ X, __nv_bfloat16* __restrict__ XT,
                                                     float* __restrict__ T, float* __restrict__ loss) {
    __shared__ __nv_bfloat16 t[64][66];
    umma::grid_release();
    const int tid = threadIdx.x, f0 = blockIdx.x * 64, r0 = blockIdx.y * 64;
    if (blockIdx.x == 0 && blockIdx.y == 0 && tid == 0) *loss = 0.0f;
    const int c = (tid & 7) * 8;
#pragma unroll
    for (int h = 0; h < 2; ++h) {
        const int r = h * 32 + (tid >> 3);
        const __nv_bfloat16* from = feats + (size_t)idx[r0 + r] * in_pad + f0 + c;
        alignas(16) __nv_bfloat16 v[8];
        if (wide) {
            *reinterpret_cast<uint4*>(v) = __ldg(reinterpret_cast<const uint4*>(from));
        } else {
#pragma unroll
            for (int k = 0; k < 8; ++k) v[k] = from[k];
        }
        *reinterpret_cast<uint4*>(X + (size_t)(r0 + r) * in_pad + f0 + c) = *reinterpret_cast<uint4*>(v);
#pragma unroll
        for (int k = 0; k < 8; ++k) t[r][c + k] = v[k];
    }
    for (int i = blockIdx.x * 256 + tid; i < 64 * n; i += gridDim.x * 256)
        T[(size_t)r0 * n + i] = targets[(size_t)idx[r0 + i / n] * n + i % n];
    __syncthreads();
    const int r = (tid & 31) * 2;
    for (int f = tid >> 5; f < 64; f += 8)
        *reinterpret_cast<__nv_bfloat162*>(XT + (size_t)(f0 + f) * M + r0 + r) = __nv_bfloat162(t[r][f], t[r + 1][f]);
}

// dOut = 2 (out - t) / (M n) as BF16 [M, n_pad] and [n_pad, M]; loss sum.
// For the mma.sync GEMM; the tcgen05 one has it in its epilogue (EPI_LOSS).
__global__ void loss_kernel(int M, int n, int n_pad, const float* __restrict__ out,
                            const float* __restrict__ t, __nv_bfloat16* __restrict__ d,
                            __nv_bfloat16* __restrict__ dT, float* __restrict__ loss) {
    const int r = blockIdx.x;
    const float scale = 2.0f / ((float)M * (float)n);
    float acc = 0.0f;
    for (int k = threadIdx.x; k < n_pad; k += blockDim.x) {
        float g = 0.0f;
        if (k < n) {
            const float diff = out[(size_t)r * n + k] - t[(size_t)r * n + k];
            acc += diff * diff;
            g = diff * scale;
        }
        const __nv_bfloat16 gb = __float2bfloat16_rn(g);
        d[(size_t)r * n_pad + k] = gb;
        dT[(size_t)k * M + r] = gb;
    }
    for (int m = 16; m; m >>= 1) acc += __shfl_xor_sync(0xffffffffu, acc, m);
    __shared__ float part[32];
    if ((threadIdx.x & 31) == 0) part[threadIdx.x >> 5] = acc;
    __syncthreads();
    if (threadIdx.x == 0) {
        float s = 0.0f;
        for (int w = 0; w < (int)(blockDim.x >> 5); ++w) s += part[w];
        atomicAdd(loss, s / ((float)M * (float)n));
    }
}

// BF16 copies of one layer: W [out, in_pad] and W^T [in, out_pad], zero pads.
__global__ void pack_kernel(int out, int in, int in_pad, int out_pad, const float* __restrict__ W,
                            __nv_bfloat16* __restrict__ Wb, __nv_bfloat16* __restrict__ WTb) {
    const int total = out_pad * in_pad;
    for (int i = blockIdx.x * blockDim.x + threadIdx.x; i < total; i += gridDim.x * blockDim.x) {
        const int r = i / in_pad, k = i % in_pad;  // r over out_pad, k over in_pad
        const float w = (r < out && k < in) ? W[(size_t)r * in + k] : 0.0f;
        const __nv_bfloat16 h = __float2bfloat16_rn(w);
        if (r < out) Wb[(size_t)r * in_pad + k] = h;
        if (k < in) WTb[(size_t)k * out_pad + r] = h;
    }
}

// Deterministic initialisation from a counter-based hash (splitmix64):
// uniform in [-bound, bound].
__device__ __forceinline__ uint64_t splitmix64(uint64_t x) {
    x += 0x9e3779b97f4a7c15ULL;
    x = (x ^ (x >> 30)) * 0xbf58476d1ce4e5b9ULL;
    x = (x ^ (x >> 27)) * 0x94d049bb133111ebULL;
    return x ^ (x >> 31);
}

__global__ void init_kernel(size_t count, float* __restrict__ p, uint64_t seed, size_t offset, float bound) {
    for (size_t i = (size_t)blockIdx.x * blockDim.x + threadIdx.x; i < count;
         i += (size_t)gridDim.x * blockDim.x) {
        const uint64_t r = splitmix64(seed ^ splitmix64(offset + i));
        const double u = (double)(r >> 11) * (1.0 / 9007199254740992.0);  // [0, 1)
        p[i] = (float)((2.0 * u - 1.0) * bound);
    }
}

// x0 = x_prev + gamma * (predicted change), the change de-standardised.
__global__ void predict_epilogue_kernel(int num_batch, int n, const float* __restrict__ out,
                                        const double* __restrict__ xp, const float* __restrict__ mean,
                                        const float* __restrict__ stdv, const double* __restrict__ gamma,
                                        double* __restrict__ x0) {
    const size_t total = (size_t)num_batch * n;
    const double g = *gamma;
    for (size_t i = (size_t)blockIdx.x * blockDim.x + threadIdx.x; i < total;
         i += (size_t)gridDim.x * blockDim.x) {
        const int k = (int)(i % n);
        x0[i] = xp[i] + g * ((double)out[i] * (double)stdv[3 * n + k] + (double)mean[3 * n + k]);
    }
}

// Gate statistics of one time step: sums over the batch of c.d and c.c, with
// c the predicted change (de-standardised network output) and d the true
// change x_next - x_prev, accumulated in FP64 (acc[0], acc[1]).
__global__ void gate_observe_kernel(int num_batch, int n, const float* __restrict__ out,
                                    const double* __restrict__ xp, const double* __restrict__ xn,
                                    const float* __restrict__ mean, const float* __restrict__ stdv,
                                    double* __restrict__ acc) {
    const size_t total = (size_t)num_batch * n;
    double cd = 0.0, cc = 0.0;
    for (size_t i = (size_t)blockIdx.x * blockDim.x + threadIdx.x; i < total;
         i += (size_t)gridDim.x * blockDim.x) {
        const int k = (int)(i % n);
        const double c = (double)out[i] * (double)stdv[3 * n + k] + (double)mean[3 * n + k];
        cd += c * (xn[i] - xp[i]);
        cc += c * c;
    }
    for (int m = 16; m; m >>= 1) {
        cd += __shfl_xor_sync(0xffffffffu, cd, m);
        cc += __shfl_xor_sync(0xffffffffu, cc, m);
    }
    if ((threadIdx.x & 31) == 0) {
        atomicAdd(acc, cd);
        atomicAdd(acc + 1, cc);
    }
}

// gamma = acc[0] / acc[1], the least-squares scale of the predicted change,
// limited to [0, 1]; 0 when no change was predicted. Clears the sums.
__global__ void gate_finalize_kernel(double* __restrict__ acc, double* __restrict__ gamma) {
    const double num = acc[0], den = acc[1];
    double g = den > 0.0 ? num / den : 0.0;
    g = isfinite(g) ? fmin(fmax(g, 0.0), 1.0) : 0.0;
    *gamma = g;
    acc[0] = 0.0;
    acc[1] = 0.0;
}

}  // namespace mlp
}  // namespace bbs

#include "bbs_mlp_infer.cuh"

// ------------------------------------------------------------------ host

using bbs::mlp::Epi;

struct bbs_mlp {
    int device = 0;
    int n = 0, hidden = 0, in = 0, in_pad = 0, n_pad = 0, max_batch = 0;
    int dims_in[4], dims_out[4], pad_in[4], pad_out[4];
    size_t off_W[4], off_b[4], count = 0;
    float *p = nullptr, *g = nullptr, *m = nullptr, *v = nullptr;
    __nv_bfloat16* Wb[4] = {};
    __nv_bfloat16* WTb[4] = {};
    int adam_t = 0;
    // statistics
    double *sums = nullptr, *sumsq = nullptr;
    double observed = 0.0;
    float *mean = nullptr, *inv_std = nullptr, *stdv = nullptr;
    // minibatch activations (max_batch rows)
    __nv_bfloat16 *X = nullptr, *XT = nullptr;
    float* T = nullptr;
    float* Z[3] = {};
    __nv_bfloat16* Y[3] = {};
    __nv_bfloat16* YT[3] = {};
    float* out = nullptr;
    __nv_bfloat16 *D = nullptr, *DT = nullptr;
    __nv_bfloat16* DZ[3] = {};
    __nv_bfloat16* DZT[3] = {};
    int* err = nullptr;     // set by a tensor-core GEMM whose waits ran out
    double* gate = nullptr;  // [gamma, sum c.d, sum c.c] (see bbs_mlp_gate_observe)
    float* loss_part = nullptr;  // one per tile of the output layer
    float* part = nullptr;  // split-K partial sums of the weight-gradient GEMMs
    size_t part_cap = 0;    // floats one layer may take of it
    int sms = 0;
    int gemm_kind = BBS_GEMM_TCGEN05;  // or BBS_GEMM_MMA_SYNC
    // fused inference (bbs_mlp_infer.cuh): TMA maps of the BF16 weights, the
    // padded output width and the kernel's shared memory; fused = usable
    CUtensorMap infer_maps[4];
    int n_mma = 0;
    size_t infer_smem = 0;
    bool fused = false;
    std::vector<void*> allocs;
};

namespace {

bbs_status errf(bbs_status s, const char* fmt, ...) {
    char msg[512];
    va_list ap;
    va_start(ap, fmt);
    vsnprintf(msg, sizeof msg, fmt, ap);
    va_end(ap);
    return bbs::record_error(s, msg);
}

int round_up(int v, int a) { return (v + a - 1) / a * a; }

template <typename T>
bool dev_alloc(bbs_mlp* m, T** ptr, size_t count) {
    void* p = nullptr;
    if (cudaMalloc(&p, std::max<size_t>(count, 1) * sizeof(T)) != cudaSuccess) return false;
    cudaMemset(p, 0, std::max<size_t>(count, 1) * sizeof(T));
    m->allocs.push_back(p);
    *ptr = static_cast<T*>(p);
    return true;
}

// cuTensorMapEncodeTiled from the driver, through the runtime (no -lcuda).
PFN_cuTensorMapEncodeTiled_v12000 tensor_map_encoder() {
    static PFN_cuTensorMapEncodeTiled_v12000 fn = nullptr;
    static bool tried = false;
    if (!tried) {
        tried = true;
        void* p = nullptr;
        cudaDriverEntryPointQueryResult q;
        if (cudaGetDriverEntryPointByVersion("cuTensorMapEncodeTiled", &p, 12000, cudaEnableDefault, &q) ==
                cudaSuccess &&
            q == cudaDriverEntryPointSuccess)
            fn = reinterpret_cast<PFN_cuTensorMapEncodeTiled_v12000>(p);
    }
    return fn;
}

// TMA map of a K-major BF16 operand [rows, K] (row stride ld elements) read
// in boxes of box_k K-elements by box_rows rows: 8 (16 bytes) without a
// swizzle, or 64 (128 bytes) in the 128-byte swizzle. Rows past the end read
// as zeros.
bool make_operand_map(CUtensorMap* map, const __nv_bfloat16* ptr, int rows, int K, int ld, int box_rows,
                      int box_k = 8) {
    PFN_cuTensorMapEncodeTiled_v12000 enc = tensor_map_encoder();
    if (enc == nullptr) return false;
    const cuuint64_t dims[2] = {(cuuint64_t)K, (cuuint64_t)rows};
    const cuuint64_t strides[1] = {(cuuint64_t)ld * 2};
    const cuuint32_t box[2] = {(cuuint32_t)box_k, (cuuint32_t)box_rows};
    const cuuint32_t estr[2] = {1, 1};
    return enc(map, CU_TENSOR_MAP_DATA_TYPE_BFLOAT16, 2, const_cast<__nv_bfloat16*>(ptr), dims, strides, box, estr,
               CU_TENSOR_MAP_INTERLEAVE_NONE, box_k == 64 ? CU_TENSOR_MAP_SWIZZLE_128B : CU_TENSOR_MAP_SWIZZLE_NONE,
               CU_TENSOR_MAP_L2_PROMOTION_L2_128B,
               CU_TENSOR_MAP_FLOAT_OOB_FILL_NONE) == CUDA_SUCCESS;
}

// Tiles and splits of a tcgen05 GEMM: 128 rows x BN columns, BN <= 64 so that
// the layer GEMMs over thousands of samples launch hundreds of blocks, and
// narrower while a GEMM that is not split leaves SMs without a block: its
// epilogue is most of it, and halves with the tile (12 -> 10 us for [4096 x
// 256] from K = 256, BN 64 -> 32). An
// FP32-output GEMM with few tiles and a long K (the weight gradients, K =
// samples) is split over K when part_cap floats have room: each split writes
// its partial tile, which are then added in a fixed order.
struct Tiles {
    int BN, mt, nt, splits, kps;
};

// Grows with the number of k-tiles nk; 1 where the tiles fill the chip.
int max_splits(const Tiles& t, int nk, size_t total, size_t part_cap, int sms) {
    const int want = 2 * sms, tiles = t.mt * t.nt;  // two blocks per SM fit (96 KB of stages each)
    if (tiles >= want || nk < 8 || total == 0) return 1;
    const size_t s = std::min<size_t>((size_t)std::min((want + tiles - 1) / tiles, nk / 4), part_cap / total);
    return (int)std::max<size_t>(s, 1);
}

Tiles gemm_tiles(int M, int N, int K, bool split, size_t part_cap, int sms) {
    Tiles t;
    const int ntile = (N + 63) / 64;
    t.BN = std::max(16, round_up((N + ntile - 1) / ntile, 16));
    t.mt = (M + bbs::umma::kBM - 1) / bbs::umma::kBM;
    t.nt = (N + t.BN - 1) / t.BN;
    const int nk = K / bbs::umma::kBK;
    t.splits = 1, t.kps = nk;
    while (!split && t.BN > 16 && t.mt * t.nt < sms) {
        t.BN = round_up(t.BN / 2, 16);
        t.nt = (N + t.BN - 1) / t.BN;
    }
    if (split) {
        t.splits = max_splits(t, nk, (size_t)M * N, part_cap, sms);
        if (t.splits > 1) {
            t.kps = (nk + t.splits - 1) / t.splits;
            t.splits = (nk + t.kps - 1) / t.kps;  // every split has k-tiles
        }
    }
    return t;
}

// Launch that may begin before the stream's last kernel ends (umma::grid_wait).
template <class... P, class... A>
cudaError_t launch_early(void (*k)(P...), dim3 grid, int threads, size_t smem, cudaStream_t st, const A&... args) {
    cudaLaunchConfig_t c{};
    cudaLaunchAttribute at{};
    at.id = cudaLaunchAttributeProgrammaticStreamSerialization;
    at.val.programmaticStreamSerializationAllowed = 1;
    c.gridDim = grid;
    c.blockDim = dim3(threads);
    c.dynamicSmemBytes = smem;
    c.stream = st;
    c.attrs = &at;
    c.numAttrs = 1;
    return cudaLaunchKernelEx(&c, k, args...);
}

bool gemm_maps(CUtensorMap* ta, CUtensorMap* tb, const __nv_bfloat16* A, int lda, const __nv_bfloat16* B, int ldb,
               int M, int N, int K, int BN) {
    return make_operand_map(ta, A, M, K, lda, bbs::umma::kBM, bbs::umma::kBK) &&
           make_operand_map(tb, B, N, K, ldb, BN, bbs::umma::kBK);
}

// What the tcgen05 GEMMs need of the current device (once per object: the launches
// of a step do not look again).
cudaError_t allow_gemms() {
    const size_t smem = bbs::umma::smem_bytes(64);
    const cudaError_t e = bbs::allow_smem((const void*)bbs::mlp::gemm_umma_kernel, smem);
    return e != cudaSuccess ? e : bbs::allow_smem((const void*)bbs::mlp::weight_grads_kernel, smem);
}

// C = A B^T through the chosen tensor-core path (kind 1: tcgen05 with the
// accumulator in tensor memory, K a multiple of 64; kind 0: mma.sync).
cudaError_t gemm_any(int kind, const __nv_bfloat16* A, int lda, const __nv_bfloat16* B, int ldb, int M, int N,
                     int K, const Epi& e, int* err, cudaStream_t st, float* part = nullptr, size_t part_cap = 0,
                     int sms = 152) {
    if (kind == BBS_GEMM_TCGEN05) {
        const Tiles t = gemm_tiles(M, N, K, e.mode == bbs::mlp::EPI_F32 && part != nullptr, part_cap, sms);
        CUtensorMap ta, tb;
        if (!gemm_maps(&ta, &tb, A, lda, B, ldb, M, N, K, t.BN)) return cudaErrorInvalidValue;
        dim3 grid(t.nt, t.mt, t.splits);
        const size_t smem = bbs::umma::smem_bytes(t.BN);
        if (t.splits == 1) {
            return launch_early(bbs::mlp::gemm_umma_kernel, grid, bbs::umma::kThreads, smem, st, ta, tb, M, N, K, t.BN,
                                t.kps, e, err);
        }
        Epi pe = e;
        pe.c = part;
        pe.ldc = N;
        pe.zstride = (size_t)M * N;
        bbs::mlp::gemm_umma_kernel<<<grid, bbs::umma::kThreads, smem, st>>>(ta, tb, M, N, K, t.BN, t.kps, pe, err);
        const size_t total = (size_t)M * N;
        const int blocks = (int)std::min<size_t>((total + 255) / 256, (size_t)sms * 8);
        bbs::mlp::splitk_reduce_kernel<<<blocks, 256, 0, st>>>(M, N, t.splits, part, e.c, e.ldc);
        return cudaGetLastError();
    }
    dim3 grid((N + bbs::mlp::kBN - 1) / bbs::mlp::kBN, (M + bbs::mlp::kBM - 1) / bbs::mlp::kBM);
    bbs::mlp::gemm_kernel<<<grid, 256, 0, st>>>(A, lda, B, ldb, M, N, K, e);
    return cudaGetLastError();
}

cudaError_t gemm(bbs_mlp* m, const __nv_bfloat16* A, int lda, const __nv_bfloat16* B, int ldb, int M, int N,
                 int K, const Epi& e, cudaStream_t st) {
    return gemm_any(m->gemm_kind, A, lda, B, ldb, M, N, K, e, m->err, st, nullptr, 0, m->sms);
}

Epi epi_f32(float* c, int ldc) {
    Epi e{};
    e.mode = bbs::mlp::EPI_F32;
    e.c = c;
    e.ldc = ldc;
    return e;
}

void pack_all(bbs_mlp* m, cudaStream_t st) {
    for (int l = 0; l < bbs::mlp::kLayers; ++l) {
        const int total = m->pad_out[l] * m->pad_in[l];
        bbs::mlp::pack_kernel<<<(total + 255) / 256, 256, 0, st>>>(m->dims_out[l], m->dims_in[l], m->pad_in[l],
                                                                   m->pad_out[l], m->p + m->off_W[l], m->Wb[l],
                                                                   m->WTb[l]);
    }
}

// Forward pass of M rows of X [M, in_pad]; activations kept for backward.
// With loss parts (tcgen05 only) the last layer writes the output gradient D
// and D^T and a sum of squared errors per tile instead of its output.
cudaError_t forward(bbs_mlp* m, const __nv_bfloat16* X, int M, bool keep_transposed, cudaStream_t st,
                    float* loss = nullptr) {
    const __nv_bfloat16* h = X;
    int ldh = m->in_pad;
    cudaError_t e = cudaSuccess;
    for (int l = 0; l < 3 && e == cudaSuccess; ++l) {
        Epi ep{};
        ep.mode = bbs::mlp::EPI_BIAS_GELU;
        ep.c = m->Z[l];
        ep.ldc = m->hidden;
        ep.bias = m->p + m->off_b[l];
        ep.y = m->Y[l];
        ep.ldy = m->hidden;
        ep.yt = keep_transposed ? m->YT[l] : nullptr;
        ep.ldyt = M;
        e = gemm(m, h, ldh, m->Wb[l], m->pad_in[l], M, m->hidden, m->pad_in[l], ep, st);
        h = m->Y[l];
        ldh = m->hidden;
    }
    if (e != cudaSuccess) return e;
    Epi ep{};
    ep.mode = bbs::mlp::EPI_BIAS;
    ep.c = m->out;
    ep.ldc = m->n;
    ep.bias = m->p + m->off_b[3];
    if (loss != nullptr) {
        ep.mode = bbs::mlp::EPI_LOSS;
        ep.z = m->T;
        ep.ldz = m->n;
        ep.y = m->D;  // its pad columns stay zero
        ep.ldy = m->n_pad;
        ep.yt = m->DT;
        ep.ldyt = M;
        ep.loss = loss;
    }
    return gemm(m, h, ldh, m->Wb[3], m->pad_in[3], M, m->n, m->pad_in[3], ep, st);
}

// Loss (cleared by the caller) and gradients of the minibatch in X/XT/T (M
// rows) into m->g: forward, then the chain of the layers' output gradients,
// then every weight gradient, which only reads them, and the optimiser's step
// if there is one.
cudaError_t backward(bbs_mlp* m, int M, float* loss, const bbs::mlp::Adam* adam, cudaStream_t st) {
    using namespace bbs::mlp;
    const bool tc = m->gemm_kind == BBS_GEMM_TCGEN05;
    cudaError_t e = forward(m, m->X, M, true, st, tc ? m->loss_part : nullptr);
    if (e != cudaSuccess) return e;
    if (!tc) loss_kernel<<<M, 160, 0, st>>>(M, m->n, m->n_pad, m->out, m->T, m->D, m->DT, loss);
    const __nv_bfloat16 *dT[kLayers], *d = m->D;  // [out, M] and [M, out_pad]
    int ld_d = m->n_pad;
    dT[kLayers - 1] = m->DT;
    for (int l = kLayers - 1; l > 0; --l) {
        // d_{l-1} = (d . W_l) * gelu'(z_{l-1}):  [M, in] = d [M, out_pad] . W_l^T [in, out_pad]^T
        Epi ep{};
        ep.mode = EPI_GELU_BWD;
        ep.z = m->Z[l - 1];
        ep.ldz = m->hidden;
        ep.y = m->DZ[l - 1];
        ep.ldy = m->hidden;
        ep.yt = m->DZT[l - 1];
        ep.ldyt = M;
        if ((e = gemm(m, d, ld_d, m->WTb[l], m->pad_out[l], M, m->dims_in[l], m->pad_out[l], ep, st)) != cudaSuccess)
            return e;
        d = m->DZ[l - 1];
        dT[l - 1] = m->DZT[l - 1];
        ld_d = m->hidden;
    }
    // dW_l = d_l^T [out, M] . h_{l-1}^T [in, M]^T, the partial sums of the
    // layers one after the other in m->part
    WeightGrads w{};
    GradSums g{};
    g.g = m->g;
    g.count = (int)m->count;
    if (tc) {
        const Tiles t = gemm_tiles(M, m->n, m->pad_in[kLayers - 1], false, 0, m->sms);  // the last layer's
        g.loss_part = m->loss_part;
        g.loss_parts = t.mt * t.nt;
        g.loss = loss;
    }
    size_t used = 0;
    bool walk = adam != nullptr;  // over the weights
    for (int l = 0; l < kLayers; ++l) {
        const int out = m->dims_out[l], in = m->dims_in[l];
        const size_t total = (size_t)out * in;
        float* dW = m->g + m->off_W[l];
        const __nv_bfloat16* hT = l == 0 ? m->XT : m->YT[l - 1];
        g.w.off_W[l] = (int)m->off_W[l], g.w.off_b[l] = (int)m->off_b[l];
        g.w.out[l] = out, g.w.in[l] = in, g.w.in_pad[l] = m->pad_in[l], g.w.out_pad[l] = m->pad_out[l];
        g.w.Wb[l] = m->Wb[l], g.w.WTb[l] = m->WTb[l];
        g.splits[l] = 1;
        g.dT[l] = dT[l];
        g.first[l + 1] = g.first[l] + out;
        if (!tc) {
            if ((e = gemm(m, dT[l], M, hT, M, out, in, M, epi_f32(dW, in), st)) != cudaSuccess) return e;
            continue;
        }
        const Tiles t = gemm_tiles(out, in, M, true, m->part_cap, m->sms);
        if (!gemm_maps(&w.a[l], &w.b[l], dT[l], M, hT, M, out, in, M, t.BN)) return cudaErrorInvalidValue;
        w.M[l] = out, w.N[l] = in, w.BN[l] = t.BN, w.kps[l] = t.kps, w.nt[l] = t.nt, w.mt[l] = t.mt;
        w.first[l + 1] = w.first[l] + t.nt * t.mt * t.splits;
        w.epi[l] = epi_f32(dW, in);
        g.splits[l] = t.splits;
        if (t.splits > 1) {
            w.epi[l].c = m->part + used;
            w.epi[l].zstride = total;
            g.part[l] = m->part + used;
            used += (size_t)t.splits * total;
            walk = true;
        }
    }
    if (tc) {
        if ((e = launch_early(weight_grads_kernel, dim3(w.first[kLayers]), bbs::umma::kThreads,
                              bbs::umma::smem_bytes(64), st, w, M, m->err)) != cudaSuccess)
            return e;
    }
    const int rb = walk ? (int)std::min<size_t>((m->count + 255) / 256, (size_t)m->sms * 16) : 0;
    for (int l = 0; l <= kLayers; ++l) g.first[l] += rb;
    return launch_early(adam ? grad_sums_kernel<true> : grad_sums_kernel<false>, dim3(g.first[kLayers] + (tc ? 1 : 0)), 256, 0, st, g,
                        M, adam ? *adam : Adam{});
}

}  // namespace

extern "C" {

bbs_status bbs_mlp_create(bbs_handle* h, int32_t n, int32_t hidden, uint64_t seed, int32_t max_batch,
                          bbs_mlp** out) {
    if (h == nullptr || out == nullptr) return errf(BBS_ERR_INVALID_ARG, "null handle or output");
    *out = nullptr;
    if (n < 1 || n > 2048 || hidden < 64 || hidden % 64 != 0 || hidden > 4096)
        return errf(BBS_ERR_INVALID_ARG, "need 1 <= n <= 2048 and hidden a multiple of 64 in [64, 4096]");
    if (max_batch < 64 || max_batch % 64 != 0)
        return errf(BBS_ERR_INVALID_ARG, "max_batch must be a positive multiple of 64");
    cudaSetDevice(bbs::handle_device(h));
    bbs_mlp* m = new bbs_mlp();
    m->device = bbs::handle_device(h);
    m->n = n;
    m->hidden = hidden;
    m->in = 3 * n;
    m->in_pad = round_up(3 * n, 64);
    m->n_pad = round_up(n, 64);
    m->max_batch = max_batch;
    const int ins[4] = {3 * n, hidden, hidden, hidden}, outs[4] = {hidden, hidden, hidden, n};
    size_t o = 0;
    for (int l = 0; l < 4; ++l) {
        m->dims_in[l] = ins[l];
        m->dims_out[l] = outs[l];
        m->pad_in[l] = round_up(ins[l], 64);
        m->pad_out[l] = round_up(outs[l], 64);
        m->off_W[l] = o;
        o += (size_t)ins[l] * outs[l];
        m->off_b[l] = o;
        o += outs[l];
    }
    m->count = o;
    bool ok = dev_alloc(m, &m->p, o) && dev_alloc(m, &m->g, o) && dev_alloc(m, &m->m, o) &&
              dev_alloc(m, &m->v, o);
    for (int l = 0; l < 4 && ok; ++l)
        ok = dev_alloc(m, &m->Wb[l], (size_t)outs[l] * m->pad_in[l]) &&
             dev_alloc(m, &m->WTb[l], (size_t)ins[l] * m->pad_out[l]);
    const int F = 4 * n;
    ok = ok && dev_alloc(m, &m->sums, F) && dev_alloc(m, &m->sumsq, F) && dev_alloc(m, &m->mean, F) &&
         dev_alloc(m, &m->inv_std, F) && dev_alloc(m, &m->stdv, F);
    const size_t MB = (size_t)max_batch;
    ok = ok && dev_alloc(m, &m->X, MB * m->in_pad) && dev_alloc(m, &m->XT, MB * m->in_pad) &&
         dev_alloc(m, &m->T, MB * n) && dev_alloc(m, &m->out, MB * n) &&
         dev_alloc(m, &m->D, MB * m->n_pad) && dev_alloc(m, &m->DT, MB * m->n_pad) &&
         dev_alloc(m, &m->err, 1) && dev_alloc(m, &m->gate, 3);
    for (int l = 0; l < 3 && ok; ++l)
        ok = dev_alloc(m, &m->Z[l], MB * hidden) && dev_alloc(m, &m->Y[l], MB * hidden) &&
             dev_alloc(m, &m->YT[l], MB * hidden) && dev_alloc(m, &m->DZ[l], MB * hidden) &&
             dev_alloc(m, &m->DZT[l], MB * hidden);
    // split-K partials of the weight gradients: a layer takes up to 32 splits of the largest [out, in]
    size_t wmax = 0;
    for (int l = 0; l < 4; ++l) wmax = std::max(wmax, (size_t)outs[l] * ins[l]);
    m->part_cap = 32 * wmax;
    cudaDeviceGetAttribute(&m->sms, cudaDevAttrMultiProcessorCount, m->device);
    if (m->sms <= 0) m->sms = 152;
    // all layers' at a time; a smaller minibatch is never split further
    size_t psum = 0;
    for (int l = 0; l < 4; ++l) {
        const size_t total = (size_t)outs[l] * ins[l];
        psum += max_splits(gemm_tiles(outs[l], ins[l], 0, true, 0, m->sms), max_batch / bbs::umma::kBK, total,
                           m->part_cap, m->sms) *
                total;
    }
    ok = ok && dev_alloc(m, &m->part, psum);
    ok = ok && dev_alloc(m, &m->loss_part, (size_t)((max_batch + bbs::umma::kBM - 1) / bbs::umma::kBM) * ((n + 15) / 16));
    if (!ok) {
        bbs_mlp_destroy(m);
        return errf(BBS_ERR_NO_MEMORY, "MLP buffers");
    }
    // init: weights U(-1/sqrt(in), 1/sqrt(in)), the output layer scaled by 0.1 so
    // the first predictions stay near the mean change; biases zero
    for (int l = 0; l < 4; ++l) {
        const float bound = (float)(1.0 / std::sqrt((double)ins[l])) * (l == 3 ? 0.1f : 1.0f);
        const size_t cnt = (size_t)ins[l] * outs[l];
        bbs::mlp::init_kernel<<<(unsigned)std::min<size_t>((cnt + 255) / 256, 4096), 256>>>(
            cnt, m->p + m->off_W[l], seed, m->off_W[l], bound);
    }
    // standardisation defaults to identity until statistics are finalised
    std::vector<float> ones(F, 1.0f);
    cudaMemcpy(m->inv_std, ones.data(), F * sizeof(float), cudaMemcpyHostToDevice);
    cudaMemcpy(m->stdv, ones.data(), F * sizeof(float), cudaMemcpyHostToDevice);
    const double gamma_one = 1.0;  // ungated until bbs_mlp_gate_finalize
    cudaMemcpy(m->gate, &gamma_one, sizeof(double), cudaMemcpyHostToDevice);
    pack_all(m, nullptr);
    // fused inference (one kernel for the whole network) when its tiles fit:
    // hidden and the 16-padded output width up to 256 (one MMA's N and the
    // tensor-memory columns), the activation tile and weight ring in shared
    // memory
    m->n_mma = round_up(n, 16);
    const bbs::mlp::InferSmem L = bbs::mlp::infer_smem(n, m->in_pad, hidden, m->n_mma);
    m->infer_smem = L.total;
    int optin = 0;
    cudaDeviceGetAttribute(&optin, cudaDevAttrMaxSharedMemoryPerBlockOptin, m->device);
    m->fused = hidden <= 256 && m->n_mma <= 256 && L.total <= (size_t)optin;
    for (int l = 0; l < 4 && m->fused; ++l)
        m->fused = make_operand_map(&m->infer_maps[l], m->Wb[l], outs[l], m->pad_in[l], m->pad_in[l],
                                    l < 3 ? hidden : m->n_mma);
    if (m->fused)
        m->fused = bbs::allow_smem((const void*)bbs::mlp::mlp_infer_kernel<false>, L.total) == cudaSuccess &&
                   bbs::allow_smem((const void*)bbs::mlp::mlp_infer_kernel<true>, L.total) == cudaSuccess;
    cudaError_t e = allow_gemms();
    if (e == cudaSuccess) e = cudaDeviceSynchronize();
    if (e != cudaSuccess) {
        bbs_mlp_destroy(m);
        return errf(BBS_ERR_CUDA, "MLP init: %s", cudaGetErrorString(e));
    }
    *out = m;
    return BBS_OK;
}

bbs_status bbs_mlp_destroy(bbs_mlp* m) {
    if (m == nullptr) return BBS_OK;
    cudaSetDevice(m->device);
    for (void* p : m->allocs) cudaFree(p);
    delete m;
    return BBS_OK;
}

bbs_status bbs_mlp_param_count(const bbs_mlp* m, int64_t* count) {
    if (m == nullptr || count == nullptr) return errf(BBS_ERR_INVALID_ARG, "null argument");
    *count = (int64_t)m->count;
    return BBS_OK;
}

bbs_status bbs_mlp_get_params(bbs_mlp* m, float* params, void* stream) {
    if (m == nullptr || params == nullptr) return errf(BBS_ERR_INVALID_ARG, "null argument");
    cudaError_t e = cudaMemcpyAsync(params, m->p, m->count * sizeof(float), cudaMemcpyDeviceToDevice,
                                    reinterpret_cast<cudaStream_t>(stream));
    return e == cudaSuccess ? BBS_OK : errf(BBS_ERR_CUDA, "%s", cudaGetErrorString(e));
}

bbs_status bbs_mlp_set_params(bbs_mlp* m, const float* params, void* stream) {
    if (m == nullptr || params == nullptr) return errf(BBS_ERR_INVALID_ARG, "null argument");
    cudaStream_t st = reinterpret_cast<cudaStream_t>(stream);
    cudaError_t e = cudaMemcpyAsync(m->p, params, m->count * sizeof(float), cudaMemcpyDeviceToDevice, st);
    if (e != cudaSuccess) return errf(BBS_ERR_CUDA, "%s", cudaGetErrorString(e));
    pack_all(m, st);
    e = cudaGetLastError();
    return e == cudaSuccess ? BBS_OK : errf(BBS_ERR_CUDA, "%s", cudaGetErrorString(e));
}

static bbs_status check_csr_batch(const bbs_mlp* m, const bbs_batch_matrix* A) {
    if (A == nullptr || A->fmt != BBS_FMT_CSR || A->n != m->n || !A->row_ptrs || !A->col_idxs || !A->values)
        return errf(BBS_ERR_INVALID_ARG, "the MLP reads a BatchCsr matrix with n = %d", m->n);
    return BBS_OK;
}

bbs_status bbs_mlp_observe(bbs_mlp* m, const bbs_batch_matrix* A, const double* b, const double* x_prev,
                           const double* x_next, void* stream) {
    if (m == nullptr || !b || !x_prev || !x_next) return errf(BBS_ERR_INVALID_ARG, "null argument");
    bbs_status s = check_csr_batch(m, A);
    if (s != BBS_OK) return s;
    if (A->num_batch == 0) return BBS_OK;
    const int F = 4 * m->n;
    dim3 grid((F + 127) / 128, std::min(A->num_batch, 256));
    bbs::mlp::observe_kernel<<<grid, 128, 0, reinterpret_cast<cudaStream_t>(stream)>>>(
        A->num_batch, m->n, A->row_ptrs, A->col_idxs, A->values, A->nnz, b, x_prev, x_next, m->sums, m->sumsq);
    m->observed += A->num_batch;
    cudaError_t e = cudaGetLastError();
    return e == cudaSuccess ? BBS_OK : errf(BBS_ERR_CUDA, "%s", cudaGetErrorString(e));
}

bbs_status bbs_mlp_finalize_stats(bbs_mlp* m, void* stream) {
    if (m == nullptr || m->observed <= 0) return errf(BBS_ERR_INVALID_ARG, "no samples observed");
    const int F = 4 * m->n;
    bbs::mlp::finalize_stats_kernel<<<(F + 127) / 128, 128, 0, reinterpret_cast<cudaStream_t>(stream)>>>(
        F, m->observed, m->sums, m->sumsq, m->mean, m->inv_std, m->stdv);
    cudaError_t e = cudaGetLastError();
    return e == cudaSuccess ? BBS_OK : errf(BBS_ERR_CUDA, "%s", cudaGetErrorString(e));
}

bbs_status bbs_mlp_make_samples(bbs_mlp* m, const bbs_batch_matrix* A, const double* b, const double* x_prev,
                                const double* x_next, uint16_t* feats, float* targets, void* stream) {
    if (m == nullptr || !b || !x_prev || !feats || (x_next && !targets))
        return errf(BBS_ERR_INVALID_ARG, "null argument");
    bbs_status s = check_csr_batch(m, A);
    if (s != BBS_OK) return s;
    if (A->num_batch == 0) return BBS_OK;
    bbs::mlp::samples_kernel<<<A->num_batch, 128, 0, reinterpret_cast<cudaStream_t>(stream)>>>(
        A->num_batch, m->n, m->in_pad, A->row_ptrs, A->col_idxs, A->values, A->nnz, b, x_prev, x_next, m->mean,
        m->inv_std, reinterpret_cast<__nv_bfloat16*>(feats), targets);
    cudaError_t e = cudaGetLastError();
    return e == cudaSuccess ? BBS_OK : errf(BBS_ERR_CUDA, "%s", cudaGetErrorString(e));
}

static bbs_status gradients(bbs_mlp* m, const uint16_t* feats, const float* targets, const int32_t* rows, int32_t M,
                            float* loss, const bbs::mlp::Adam* adam, void* stream) {
    if (m == nullptr || !feats || !targets || !rows || !loss) return errf(BBS_ERR_INVALID_ARG, "null argument");
    if (M < 64 || M > m->max_batch || M % 64 != 0)
        return errf(BBS_ERR_INVALID_ARG, "minibatch must be a multiple of 64 up to %d", m->max_batch);
    cudaStream_t st = reinterpret_cast<cudaStream_t>(stream);
    bbs::mlp::gather_kernel<<<dim3(m->in_pad / 64, M / 64), 256, 0, st>>>(
        M, m->in_pad, m->n, rows, reinterpret_cast<const __nv_bfloat16*>(feats), targets,
        reinterpret_cast<uintptr_t>(feats) % 16 == 0, m->X, m->XT, m->T, loss);
    cudaError_t e = cudaGetLastError();
    if (e == cudaSuccess) e = backward(m, M, loss, adam, st);
    return e == cudaSuccess ? BBS_OK : errf(BBS_ERR_CUDA, "%s", cudaGetErrorString(e));
}

bbs_status bbs_mlp_gradients(bbs_mlp* m, const uint16_t* feats, const float* targets, const int32_t* rows,
                             int32_t M, float* loss, void* stream) {
    return gradients(m, feats, targets, rows, M, loss, nullptr, stream);
}

bbs_status bbs_mlp_train_step(bbs_mlp* m, const uint16_t* feats, const float* targets, const int32_t* rows,
                              int32_t M, float lr, float* loss, void* stream) {
    if (m == nullptr) return errf(BBS_ERR_INVALID_ARG, "null argument");
    const float t = (float)(m->adam_t + 1);
    const bbs::mlp::Adam adam{m->p, m->m, m->v, lr, 0.9f, 0.999f, 1e-8f, 1.0f - powf(0.9f, t), 1.0f - powf(0.999f, t)};
    bbs_status s = gradients(m, feats, targets, rows, M, loss, &adam, stream);
    if (s == BBS_OK) m->adam_t += 1;
    return s;
}

bbs_status bbs_mlp_set_gemm(bbs_mlp* m, int32_t kind) {
    if (m == nullptr || (kind != BBS_GEMM_MMA_SYNC && kind != BBS_GEMM_TCGEN05))
        return errf(BBS_ERR_INVALID_ARG, "unknown GEMM kind");
    m->gemm_kind = kind;
    return BBS_OK;
}

bbs_status bbs_mlp_check(bbs_mlp* m) {
    if (m == nullptr) return errf(BBS_ERR_INVALID_ARG, "null network");
    int flag = 0;
    cudaError_t e = cudaMemcpy(&flag, m->err, sizeof(int), cudaMemcpyDeviceToHost);
    if (e != cudaSuccess) return errf(BBS_ERR_CUDA, "%s", cudaGetErrorString(e));
    return flag ? errf(BBS_ERR_CUDA, "a tensor-core GEMM gave up waiting for its MMAs") : BBS_OK;
}

bbs_status bbs_gemm_bf16(bbs_handle* h, int32_t kind, const uint16_t* A, int32_t lda, const uint16_t* B,
                         int32_t ldb, int32_t M, int32_t N, int32_t K, float* C, int32_t ldc) {
    if (h == nullptr || !A || !B || !C || M < 0 || N < 0 || K < 0)
        return errf(BBS_ERR_INVALID_ARG, "null pointer or negative size");
    if (kind != BBS_GEMM_MMA_SYNC && kind != BBS_GEMM_TCGEN05) return errf(BBS_ERR_INVALID_ARG, "unknown GEMM kind");
    const int kmul = kind == BBS_GEMM_TCGEN05 ? 64 : 32;
    if (K % kmul != 0 || lda % 8 != 0 || ldb % 8 != 0 || lda < K || ldb < K || ldc < N)
        return errf(BBS_ERR_INVALID_ARG, "K must be a multiple of %d, lda/ldb multiples of 8 and >= K", kmul);
    if (M == 0 || N == 0) return BBS_OK;
    cudaSetDevice(bbs::handle_device(h));
    int* err = nullptr;
    cudaError_t e = cudaMalloc(&err, sizeof(int));
    if (e != cudaSuccess) return errf(BBS_ERR_NO_MEMORY, "%s", cudaGetErrorString(e));
    cudaMemset(err, 0, sizeof(int));
    Epi ep = epi_f32(C, ldc);
    if (K == 0) {
        cudaFree(err);
        return errf(BBS_ERR_INVALID_ARG, "K must be positive");
    }
    float* part = nullptr;
    const size_t part_cap = (size_t)32 * M * N;
    if (kind == BBS_GEMM_TCGEN05 && cudaMalloc(&part, part_cap * sizeof(float)) != cudaSuccess) part = nullptr;
    int sms = 0;
    cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, bbs::handle_device(h));
    e = allow_gemms();
    if (e == cudaSuccess)
        e = gemm_any(kind, reinterpret_cast<const __nv_bfloat16*>(A), lda, reinterpret_cast<const __nv_bfloat16*>(B),
                     ldb, M, N, K, ep, err, nullptr, part, part ? part_cap : 0, sms > 0 ? sms : 152);
    int flag = 0;
    if (e == cudaSuccess) e = cudaDeviceSynchronize();
    if (e == cudaSuccess) e = cudaMemcpy(&flag, err, sizeof(int), cudaMemcpyDeviceToHost);
    cudaFree(err);
    if (part) cudaFree(part);
    if (e != cudaSuccess) return errf(BBS_ERR_CUDA, "%s", cudaGetErrorString(e));
    return flag ? errf(BBS_ERR_CUDA, "the tensor-core GEMM gave up waiting for its MMAs") : BBS_OK;
}

bbs_status bbs_mlp_get_grads(bbs_mlp* m, float* grads, void* stream) {
    if (m == nullptr || grads == nullptr) return errf(BBS_ERR_INVALID_ARG, "null argument");
    cudaError_t e = cudaMemcpyAsync(grads, m->g, m->count * sizeof(float), cudaMemcpyDeviceToDevice,
                                    reinterpret_cast<cudaStream_t>(stream));
    return e == cudaSuccess ? BBS_OK : errf(BBS_ERR_CUDA, "%s", cudaGetErrorString(e));
}

bbs_status bbs_mlp_forward(bbs_mlp* m, const uint16_t* feats, int32_t M, float* out, void* stream) {
    if (m == nullptr || !feats || !out) return errf(BBS_ERR_INVALID_ARG, "null argument");
    cudaStream_t st = reinterpret_cast<cudaStream_t>(stream);
    for (int r0 = 0; r0 < M; r0 += m->max_batch) {
        const int rows = std::min(m->max_batch, M - r0);
        cudaError_t e = forward(m, reinterpret_cast<const __nv_bfloat16*>(feats) + (size_t)r0 * m->in_pad, rows,
                                false, st);
        if (e == cudaSuccess)
            e = cudaMemcpyAsync(out + (size_t)r0 * m->n, m->out, sizeof(float) * rows * m->n,
                                cudaMemcpyDeviceToDevice, st);
        if (e != cudaSuccess) return errf(BBS_ERR_CUDA, "%s", cudaGetErrorString(e));
    }
    return BBS_OK;
}

}  // extern "C"

// The tcgen05 path runs predictions and gate statistics through the fused
// kernel when the network's tiles fit it.
static bool uses_fused(const bbs_mlp* m) { return m->fused && m->gemm_kind == BBS_GEMM_TCGEN05; }

// One launch of the fused network over the batch (128 systems per block):
// x0 = x_prev + gamma * change (x_next == nullptr), or the gate statistics of
// the change against x_next - x_prev.
static bbs_status infer_fused(bbs_mlp* m, const bbs_batch_matrix* A, const double* b, const double* x_prev,
                              const double* x_next, double* x0, cudaStream_t st) {
    if (A->num_batch == 0) return BBS_OK;
    bbs::mlp::InferParams p{};
    p.num_batch = A->num_batch;
    p.n = m->n;
    p.nnz = A->nnz;
    p.in_pad = m->in_pad;
    p.hidden = m->hidden;
    p.n_mma = m->n_mma;
    p.row_ptrs = A->row_ptrs;
    p.cols = A->col_idxs;
    p.values = A->values;
    p.b = b;
    p.xp = x_prev;
    p.xn = x_next;
    p.x0 = x0;
    p.acc = m->gate + 1;
    for (int l = 0; l < 4; ++l) p.bias[l] = m->p + m->off_b[l];
    p.mean = m->mean;
    p.inv_std = m->inv_std;
    p.stdv = m->stdv;
    p.gamma = m->gate;
    p.err = m->err;
    const unsigned grid = (unsigned)((A->num_batch + bbs::mlp::kInferRows - 1) / bbs::mlp::kInferRows);
    const auto& w = m->infer_maps;
    if (x_next != nullptr)
        bbs::mlp::mlp_infer_kernel<true><<<grid, bbs::mlp::kInferThreads, m->infer_smem, st>>>(w[0], w[1], w[2], w[3], p);
    else
        bbs::mlp::mlp_infer_kernel<false><<<grid, bbs::mlp::kInferThreads, m->infer_smem, st>>>(w[0], w[1], w[2], w[3],
                                                                                              p);
    cudaError_t e = cudaGetLastError();
    return e == cudaSuccess ? BBS_OK : errf(BBS_ERR_CUDA, "%s", cudaGetErrorString(e));
}

// The network over a batch, max_batch rows at a time; `tail(r0, rows)`
// consumes each piece's output in m->out.
template <class Tail>
static bbs_status run_batch(bbs_mlp* m, const bbs_batch_matrix* A, const double* b, const double* x_prev,
                            cudaStream_t st, Tail tail) {
    const int n = m->n;
    for (int r0 = 0; r0 < A->num_batch; r0 += m->max_batch) {
        const int rows = std::min(m->max_batch, A->num_batch - r0);
        bbs::mlp::samples_kernel<<<rows, 128, 0, st>>>(
            rows, n, m->in_pad, A->row_ptrs, A->col_idxs, A->values + (size_t)r0 * A->nnz, A->nnz,
            b + (size_t)r0 * n, x_prev + (size_t)r0 * n, nullptr, m->mean, m->inv_std, m->X, nullptr);
        cudaError_t e = forward(m, m->X, rows, false, st);
        if (e != cudaSuccess) return errf(BBS_ERR_CUDA, "%s", cudaGetErrorString(e));
        tail(r0, rows);
    }
    cudaError_t e = cudaGetLastError();
    return e == cudaSuccess ? BBS_OK : errf(BBS_ERR_CUDA, "%s", cudaGetErrorString(e));
}

extern "C" {

bbs_status bbs_mlp_predict(bbs_mlp* m, const bbs_batch_matrix* A, const double* b, const double* x_prev,
                           double* x0, void* stream) {
    if (m == nullptr || !b || !x_prev || !x0) return errf(BBS_ERR_INVALID_ARG, "null argument");
    bbs_status s = check_csr_batch(m, A);
    if (s != BBS_OK) return s;
    cudaStream_t st = reinterpret_cast<cudaStream_t>(stream);
    if (uses_fused(m)) return infer_fused(m, A, b, x_prev, nullptr, x0, st);
    const int n = m->n;
    return run_batch(m, A, b, x_prev, st, [&](int r0, int rows) {
        bbs::mlp::predict_epilogue_kernel<<<std::min((rows * n + 255) / 256, 4096), 256, 0, st>>>(
            rows, n, m->out, x_prev + (size_t)r0 * n, m->mean, m->stdv, m->gate, x0 + (size_t)r0 * n);
    });
}

bbs_status bbs_mlp_gate_observe(bbs_mlp* m, const bbs_batch_matrix* A, const double* b, const double* x_prev,
                                const double* x_next, void* stream) {
    if (m == nullptr || !b || !x_prev || !x_next) return errf(BBS_ERR_INVALID_ARG, "null argument");
    bbs_status s = check_csr_batch(m, A);
    if (s != BBS_OK) return s;
    cudaStream_t st = reinterpret_cast<cudaStream_t>(stream);
    if (uses_fused(m)) return infer_fused(m, A, b, x_prev, x_next, nullptr, st);
    const int n = m->n;
    return run_batch(m, A, b, x_prev, st, [&](int r0, int rows) {
        bbs::mlp::gate_observe_kernel<<<std::min((rows * n + 255) / 256, 1024), 256, 0, st>>>(
            rows, n, m->out, x_prev + (size_t)r0 * n, x_next + (size_t)r0 * n, m->mean, m->stdv, m->gate + 1);
    });
}

bbs_status bbs_mlp_gate_finalize(bbs_mlp* m, void* stream) {
    if (m == nullptr) return errf(BBS_ERR_INVALID_ARG, "null argument");
    bbs::mlp::gate_finalize_kernel<<<1, 1, 0, reinterpret_cast<cudaStream_t>(stream)>>>(m->gate + 1, m->gate);
    cudaError_t e = cudaGetLastError();
    return e == cudaSuccess ? BBS_OK : errf(BBS_ERR_CUDA, "%s", cudaGetErrorString(e));
}

bbs_status bbs_mlp_get_gate(bbs_mlp* m, double* gamma) {
    if (m == nullptr || gamma == nullptr) return errf(BBS_ERR_INVALID_ARG, "null argument");
    cudaError_t e = cudaMemcpy(gamma, m->gate, sizeof(double), cudaMemcpyDeviceToHost);
    return e == cudaSuccess ? BBS_OK : errf(BBS_ERR_CUDA, "%s", cudaGetErrorString(e));
}

}  // extern "C"
