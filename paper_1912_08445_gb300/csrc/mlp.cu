// Learned initial level populations: a 4 -> 128 -> 128 -> 128 -> n_out network (ReLU,
// log-softmax output) mapping four local features of a cell to its log fractional level
// populations, trained on populations the ALI itself converged to.
//
// Kernels:
//   k_features     FP64 features per cell (log n, log T, log |grad v|, log Sobolev tau)
//   k_mlp_tile     one CTA of 16 warps per 64 rows: the 128-wide layers, the back-propagated
//                  deltas and the weight gradients run on the tensor cores (mma.sync
//                  m16n8k16, BF16 operands, FP32 accumulation), operands in shared memory;
//                  the gradients are per-CTA FP32 partial sums, summed over CTAs in a fixed
//                  order
//   k_count        number of targets of a batch (the loss is their mean)
//   k_grad_reduce  fixed-order sum of the per-CTA partials
//   k_adam         Adam on FP32 master weights, refreshing the BF16 copies
#include <cuda_bf16.h>
#include <chrono>
#include <cmath>
#include <cstring>
#include <algorithm>
#include <mutex>
#include <random>
#include <cstdio>
#include "common.cuh"

using namespace mg;

namespace {

constexpr int kHid = 128;          // hidden width
constexpr int kIn = 4;           // features
constexpr int kRows = 64;        // rows per CTA
constexpr int kMaxOut = 32;      // padded output width
constexpr float kFracMin = 1e-12f;

struct Layout {
    int n_out, npad;
    // offsets into the flat FP32 parameter vector
    int64_t W1, b1, W2, b2, W3, b3, W4, b4, total;
};

Layout make_layout(int n_out) {
    Layout L{};
    L.n_out = n_out;
    L.npad = n_out <= 16 ? 16 : 32;
    int64_t k = 0;
    L.W1 = k; k += kIn * kHid;
    L.b1 = k; k += kHid;
    L.W2 = k; k += kHid * kHid;
    L.b2 = k; k += kHid;
    L.W3 = k; k += kHid * kHid;
    L.b3 = k; k += kHid;
    L.W4 = k; k += kHid * n_out;
    L.b4 = k; k += n_out;
    L.total = k;
    return L;
}

// Floats per CTA of gradient partials: the parameters and the loss, rounded up so that every
// CTA's share starts on a 16-byte boundary.
__host__ __device__ inline int64_t partial_stride(const Layout &L) { return (L.total + 4) & ~(int64_t)3; }

// BF16 weight copies stored [out][in], W4 padded to npad outputs with zeros (the backward
// products read them transposed).
struct BfWeights {
    __nv_bfloat16 *W2T, *W3T, *W4T;   // [128][128], [128][128], [npad][128]
};

__device__ __forceinline__ void mma_bf16(float (&c)[4], const uint32_t (&a)[4], uint32_t b0, uint32_t b1) {
    asm volatile("mma.sync.aligned.m16n8k16.row.col.f32.bf16.bf16.f32 {%0,%1,%2,%3}, {%4,%5,%6,%7}, {%8,%9}, "
                 "{%0,%1,%2,%3};"
                 : "+f"(c[0]), "+f"(c[1]), "+f"(c[2]), "+f"(c[3])
                 : "r"(a[0]), "r"(a[1]), "r"(a[2]), "r"(a[3]), "r"(b0), "r"(b1));
}

// Four 8 x 8 BF16 blocks of shared memory into a fragment, as stored or transposed; lane l
// gives the address of row l % 8 of block l / 8.
__device__ __forceinline__ void ldsm4(uint32_t (&r)[4], const __nv_bfloat16 *p) {
    asm volatile("ldmatrix.sync.aligned.m8n8.x4.shared.b16 {%0,%1,%2,%3}, [%4];"
                 : "=r"(r[0]), "=r"(r[1]), "=r"(r[2]), "=r"(r[3])
                 : "r"((unsigned)__cvta_generic_to_shared(p))
                 : "memory");
}
__device__ __forceinline__ void ldsm4t(uint32_t (&r)[4], const __nv_bfloat16 *p) {
    asm volatile("ldmatrix.sync.aligned.m8n8.x4.trans.shared.b16 {%0,%1,%2,%3}, [%4];"
                 : "=r"(r[0]), "=r"(r[1]), "=r"(r[2]), "=r"(r[3])
                 : "r"((unsigned)__cvta_generic_to_shared(p))
                 : "memory");
}

// acc[16 x 8 NT] (+)= A[16 x 16 KT] times B. A: rows of shared memory (stride lda), or with TA
// columns (A[m][k] stored at [k][m]). B: stored [n][k] (stride ldb), or with TB [k][n]. Fragment
// layouts of mma.m16n8k16: lane = 4 g + c holds rows g and g+8, columns 2c, 2c+1 (+8).
template <int KT, int NT, bool TA, bool TB>
__device__ __forceinline__ void warp_gemm(const __nv_bfloat16 *A, int lda, const __nv_bfloat16 *B, int ldb,
                                          float (&acc)[NT][4]) {
    static_assert(NT % 2 == 0, "two column blocks per load of B");
    const int lane = threadIdx.x & 31, r = lane & 7, m = lane >> 3;
#pragma unroll
    for (int nt = 0; nt < NT; nt++) acc[nt][0] = acc[nt][1] = acc[nt][2] = acc[nt][3] = 0.f;
#pragma unroll
    for (int kt = 0; kt < KT; kt++) {
        uint32_t a[4];
        if (TA) ldsm4t(a, A + (16 * kt + r + 8 * (m >> 1)) * lda + 8 * (m & 1));
        else ldsm4(a, A + (r + 8 * (m & 1)) * lda + 16 * kt + 8 * (m >> 1));
#pragma unroll
        for (int nt = 0; nt < NT; nt += 2) {
            uint32_t b[4];
            if (TB) ldsm4t(b, B + (16 * kt + r + 8 * (m & 1)) * ldb + 8 * nt + 8 * (m >> 1));
            else ldsm4(b, B + (8 * nt + r + 8 * (m >> 1)) * ldb + 16 * kt + 8 * (m & 1));
            mma_bf16(acc[nt], a, b[0], b[1]);
            mma_bf16(acc[nt + 1], a, b[2], b[3]);
        }
    }
}

struct TileArgs {
    int64_t rows;
    const float *X;            // [rows][4] raw features
    const int32_t *index;      // optional row permutation
    const float *Y;            // [rows][n_out] target fractions (training) or nullptr
    const float *theta;        // FP32 master (W1, biases)
    BfWeights w;
    Layout L;
    float mean[kIn], istd[kIn];
    const int *count;          // number of (row, level) targets >= 1e-12 in the batch (training)
    float *logp;               // [rows][n_out] output (forward) or nullptr
    float *partial;            // [tiles][partial_stride] gradient partials and loss (training)
};

constexpr int kLd = kHid + 8;       // row stride in shared memory: 8 rows of 16 bytes hit all banks once
constexpr int kLdz = kMaxOut + 8;
constexpr int kTileThreads = 512;

// Shared memory per CTA: weights as [out][in], activations h1, h2, h3, two delta buffers
// (bf16) and inputs.
struct TileSmem {
    __nv_bfloat16 w2[kHid][kLd], w3[kHid][kLd], w4[kMaxOut][kLd];
    __nv_bfloat16 h1[kRows][kLd], h2[kRows][kLd], h3[kRows][kLd];
    __nv_bfloat16 da[kRows][kLd], db[kRows][kLd];
    __nv_bfloat16 dz[kRows][kLdz];
    float x[kRows][kIn];
    float loss[4];
};

// Stores an accumulator block (16 rows from r0, columns from c0) plus bias into bf16 rows
// with ReLU.
template <int NT>
__device__ __forceinline__ void store_relu(float (&acc)[NT][4], const float *bias, __nv_bfloat16 (*dst)[kLd], int r0,
                                           int c0) {
    const int lane = threadIdx.x & 31, g = lane >> 2, c = lane & 3;
#pragma unroll
    for (int nt = 0; nt < NT; nt++) {
        const int col = c0 + 8 * nt + 2 * c;
        const float b0 = bias[col], b1 = bias[col + 1];
        *reinterpret_cast<__nv_bfloat162 *>(&dst[r0 + g][col]) =
            __floats2bfloat162_rn(fmaxf(acc[nt][0] + b0, 0.f), fmaxf(acc[nt][1] + b1, 0.f));
        *reinterpret_cast<__nv_bfloat162 *>(&dst[r0 + g + 8][col]) =
            __floats2bfloat162_rn(fmaxf(acc[nt][2] + b0, 0.f), fmaxf(acc[nt][3] + b1, 0.f));
    }
}

// Delta through a ReLU layer: dst = acc masked by (h > 0).
template <int NT>
__device__ __forceinline__ void store_masked(float (&acc)[NT][4], __nv_bfloat16 (*h)[kLd], __nv_bfloat16 (*dst)[kLd],
                                             int r0, int c0) {
    const int lane = threadIdx.x & 31, g = lane >> 2, c = lane & 3;
#pragma unroll
    for (int nt = 0; nt < NT; nt++) {
        const int col = c0 + 8 * nt + 2 * c;
#pragma unroll
        for (int s = 0; s < 2; s++) {
            const float2 hv = __bfloat1622float2(*reinterpret_cast<__nv_bfloat162 *>(&h[r0 + g + 8 * s][col]));
            *reinterpret_cast<__nv_bfloat162 *>(&dst[r0 + g + 8 * s][col]) = __floats2bfloat162_rn(
                hv.x > 0.f ? acc[nt][2 * s] : 0.f, hv.y > 0.f ? acc[nt][2 * s + 1] : 0.f);
        }
    }
}

// dW[i][j] = sum_rows a[r][i] d[r][j] over this CTA's rows, i in [i0, i0 + 16), j in [j0, j0 + 8 NT),
// j < nj: on the tensor cores, K = rows.
template <int NT>
__device__ __forceinline__ void weight_grad(const __nv_bfloat16 *a, const __nv_bfloat16 *d, int ldd, int i0, int j0,
                                            int nj, float *out) {
    const int lane = threadIdx.x & 31, g = lane >> 2, c = lane & 3;
    float acc[NT][4];
    warp_gemm<kRows / 16, NT, true, true>(a + i0, kLd, d + j0, ldd, acc);
#pragma unroll
    for (int nt = 0; nt < NT; nt++)
#pragma unroll
        for (int s = 0; s < 2; s++) {
            const int i = i0 + g + 8 * s, j = j0 + 8 * nt + 2 * c;
            if (nj == kHid) {   // (the layers' rows start on even offsets)
                *reinterpret_cast<float2 *>(&out[i * kHid + j]) = make_float2(acc[nt][2 * s], acc[nt][2 * s + 1]);
            } else {
                if (j < nj) out[i * nj + j] = acc[nt][2 * s];
                if (j + 1 < nj) out[i * nj + j + 1] = acc[nt][2 * s + 1];
            }
        }
}

// Copies n rows of 128 bf16 from global memory into padded rows.
__device__ __forceinline__ void load_rows(__nv_bfloat16 (*dst)[kLd], const __nv_bfloat16 *src, int n) {
    for (int t = threadIdx.x; t < n * (kHid / 8); t += kTileThreads) {
        const int r = t / (kHid / 8), k = t - r * (kHid / 8);
        *reinterpret_cast<uint4 *>(&dst[r][8 * k]) = *reinterpret_cast<const uint4 *>(src + r * kHid + 8 * k);
    }
}

// One CTA per 64 rows (without gradients the CTAs take several tiles and load the weights
// once). The products are small (64 x 128 x 128) and what bounded them was the latency of
// their operands: weights gathered four bytes at a time from global memory by 4 warps, weight
// gradients one output and 64 dependent shared-memory loads at a time. Sixteen warps now
// share each product (16 x 32 outputs each) with all operands in shared memory (ldmatrix),
// and the gradients are tensor-core products over the rows. 4096 rows: 151 -> 26 us.
__global__ void __launch_bounds__(kTileThreads) k_mlp_tile(TileArgs a) {
    extern __shared__ __align__(16) unsigned char smem_raw[];
    TileSmem &S = *reinterpret_cast<TileSmem *>(smem_raw);
    const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31, g = lane >> 2, c = lane & 3;
    const int r0 = (warp & 3) * 16, c0 = (warp >> 2) * 32;
    const int n_out = a.L.n_out, npad = a.L.npad;
    const float *th = a.theta;
    load_rows(S.w2, a.w.W2T, kHid);
    load_rows(S.w3, a.w.W3T, kHid);
    load_rows(S.w4, a.w.W4T, npad);
    const int64_t tiles = (a.rows + kRows - 1) / kRows;
    for (int64_t tile = blockIdx.x; tile < tiles; tile += gridDim.x) {
        const int64_t row0 = tile * kRows;
        // inputs (normalised); rows beyond the end are zero and carry no loss
        for (int t = threadIdx.x; t < kRows * kIn; t += kTileThreads) {
            const int r = t / kIn, i = t - r * kIn;
            const int64_t gr = row0 + r;
            float v = 0.f;
            if (gr < a.rows) {
                const int64_t src = a.index ? a.index[gr] : gr;
                v = (a.X[src * kIn + i] - a.mean[i]) * a.istd[i];
            }
            S.x[r][i] = v;
        }
        __syncthreads();
        // layer 1 (K = 4) on the CUDA cores
        for (int t = threadIdx.x; t < kRows * kHid; t += kTileThreads) {
            const int r = t / kHid, j = t - r * kHid;
            float s = th[a.L.b1 + j];
#pragma unroll
            for (int i = 0; i < kIn; i++) s += S.x[r][i] * th[a.L.W1 + i * kHid + j];
            S.h1[r][j] = __float2bfloat16(fmaxf(s, 0.f));
        }
        __syncthreads();
        {   // layers 2 and 3
            float acc[4][4];
            warp_gemm<8, 4, false, false>(&S.h1[r0][0], kLd, &S.w2[c0][0], kLd, acc);
            store_relu<4>(acc, th + a.L.b2, S.h2, r0, c0);
            __syncthreads();
            warp_gemm<8, 4, false, false>(&S.h2[r0][0], kLd, &S.w3[c0][0], kLd, acc);
            store_relu<4>(acc, th + a.L.b3, S.h3, r0, c0);
            __syncthreads();
        }
        // output layer and log-softmax, the first four warps; lanes 4g..4g+3 hold rows r0+g
        // and r0+g+8
        if (warp < 4) {
            float z[4][4];
            float lp[4][4];
            {
                float acc[4][4];
                if (npad == 16) {
                    float a2[2][4];
                    warp_gemm<8, 2, false, false>(&S.h3[r0][0], kLd, &S.w4[0][0], kLd, a2);
                    for (int nt = 0; nt < 4; nt++)
                        for (int k = 0; k < 4; k++) acc[nt][k] = nt < 2 ? a2[nt][k] : 0.f;
                } else {
                    warp_gemm<8, 4, false, false>(&S.h3[r0][0], kLd, &S.w4[0][0], kLd, acc);
                }
                float mx[2] = {-INFINITY, -INFINITY};
                for (int nt = 0; nt < 4; nt++)
                    for (int k = 0; k < 4; k++) {
                        const int col = 8 * nt + 2 * c + (k & 1);
                        z[nt][k] = col < n_out ? acc[nt][k] + th[a.L.b4 + col] : -INFINITY;
                        mx[k >> 1] = fmaxf(mx[k >> 1], z[nt][k]);
                    }
                for (int s = 0; s < 2; s++) {
                    mx[s] = fmaxf(mx[s], __shfl_xor_sync(0xffffffffu, mx[s], 1));
                    mx[s] = fmaxf(mx[s], __shfl_xor_sync(0xffffffffu, mx[s], 2));
                }
                float se[2] = {0.f, 0.f};
                for (int nt = 0; nt < 4; nt++)
                    for (int k = 0; k < 4; k++)
                        se[k >> 1] += (z[nt][k] == -INFINITY) ? 0.f : expf(z[nt][k] - mx[k >> 1]);
                for (int s = 0; s < 2; s++) {
                    se[s] += __shfl_xor_sync(0xffffffffu, se[s], 1);
                    se[s] += __shfl_xor_sync(0xffffffffu, se[s], 2);
                }
                for (int nt = 0; nt < 4; nt++)
                    for (int k = 0; k < 4; k++) lp[nt][k] = z[nt][k] - mx[k >> 1] - logf(se[k >> 1]);
            }
            if (a.logp) {
                for (int nt = 0; nt < 4; nt++)
                    for (int k = 0; k < 4; k++) {
                        const int col = 8 * nt + 2 * c + (k & 1);
                        const int64_t gr = row0 + r0 + g + 8 * (k >> 1);
                        if (col < n_out && gr < a.rows) a.logp[gr * n_out + col] = lp[nt][k];
                    }
            }
            if (a.partial) {
                // dL/dlogp, through log-softmax
                const int cnt = *a.count;
                const float inv_count = cnt ? 1.f / (float)cnt : 0.f;
                float lsum = 0.f;
                float gsum[2] = {0.f, 0.f};
                float gv[4][4];
                for (int nt = 0; nt < 4; nt++)
                    for (int k = 0; k < 4; k++) {
                        const int col = 8 * nt + 2 * c + (k & 1);
                        const int64_t gr = row0 + r0 + g + 8 * (k >> 1);
                        float gg = 0.f;
                        if (col < n_out && gr < a.rows) {
                            const int64_t src = a.index ? a.index[gr] : gr;
                            const float y = a.Y[src * n_out + col];
                            if (y >= kFracMin) {
                                const float d = lp[nt][k] - logf(y);
                                lsum += d * d;
                                gg = 2.f * d * inv_count;
                            }
                        }
                        gv[nt][k] = gg;
                        gsum[k >> 1] += gg;
                    }
                for (int s = 0; s < 2; s++) {
                    gsum[s] += __shfl_xor_sync(0xffffffffu, gsum[s], 1);
                    gsum[s] += __shfl_xor_sync(0xffffffffu, gsum[s], 2);
                }
                for (int nt = 0; nt < 4; nt++)
                    for (int k = 0; k < 4; k++) {
                        const int col = 8 * nt + 2 * c + (k & 1);
                        const float dzv = col < n_out ? gv[nt][k] - expf(lp[nt][k]) * gsum[k >> 1] : 0.f;
                        S.dz[r0 + g + 8 * (k >> 1)][col] = __float2bfloat16(dzv);
                    }
                for (int d = 16; d; d >>= 1) lsum += __shfl_xor_sync(0xffffffffu, lsum, d);
                if (lane == 0) S.loss[warp] = lsum;
            }
        }
        __syncthreads();
        if (!a.partial) continue;
        // ---- training: back through the layers
        {   // dh3 = (dz W4^T) masked by h3 > 0; dh2 = (dh3 W3^T) masked by h2 > 0
            float acc[4][4];
            if (npad == 16) warp_gemm<1, 4, false, true>(&S.dz[r0][0], kLdz, &S.w4[0][c0], kLd, acc);
            else warp_gemm<2, 4, false, true>(&S.dz[r0][0], kLdz, &S.w4[0][c0], kLd, acc);
            store_masked<4>(acc, S.h3, S.da, r0, c0);
            __syncthreads();
            warp_gemm<8, 4, false, true>(&S.da[r0][0], kLd, &S.w3[0][c0], kLd, acc);
            store_masked<4>(acc, S.h2, S.db, r0, c0);
        }
        __syncthreads();
        float *P = a.partial + (size_t)tile * partial_stride(a.L);
        // weight gradients of layers 4 and 3 (need dz, h3, dh3 = da, h2)
        if (warp < 8) {
            if (npad == 16) weight_grad<2>(&S.h3[0][0], &S.dz[0][0], kLdz, 16 * warp, 0, n_out, P + a.L.W4);
            else weight_grad<4>(&S.h3[0][0], &S.dz[0][0], kLdz, 16 * warp, 0, n_out, P + a.L.W4);
        } else {
            for (int j = threadIdx.x - 256; j < n_out + kHid; j += 256) {
                float s = 0.f;
                if (j < n_out)
                    for (int r = 0; r < kRows; r++) s += __bfloat162float(S.dz[r][j]);
                else
                    for (int r = 0; r < kRows; r++) s += __bfloat162float(S.da[r][j - n_out]);
                P[j < n_out ? a.L.b4 + j : a.L.b3 + j - n_out] = s;
            }
        }
        for (int q = 0; q < 2; q++)
            weight_grad<4>(&S.h2[0][0], &S.da[0][0], kLd, 16 * (2 * (warp & 3) + q), c0, kHid, P + a.L.W3);
        __syncthreads();
        {   // dh1 = dh2 W2^T, masked by h1 > 0 (into da, which is free now)
            float acc[4][4];
            warp_gemm<8, 4, false, true>(&S.db[r0][0], kLd, &S.w2[0][c0], kLd, acc);
            store_masked<4>(acc, S.h1, S.da, r0, c0);
        }
        __syncthreads();
        for (int q = 0; q < 2; q++)
            weight_grad<4>(&S.h1[0][0], &S.db[0][0], kLd, 16 * (2 * (warp & 3) + q), c0, kHid, P + a.L.W2);
        for (int t = threadIdx.x; t < (kIn + 2) * kHid; t += kTileThreads) {
            const int i = t / kHid, j = t - i * kHid;
            float s = 0.f;
            if (i < kIn) {
                for (int r = 0; r < kRows; r++) s += S.x[r][i] * __bfloat162float(S.da[r][j]);
                P[a.L.W1 + t] = s;
            } else if (i == kIn) {
                for (int r = 0; r < kRows; r++) s += __bfloat162float(S.db[r][j]);
                P[a.L.b2 + j] = s;
            } else {
                for (int r = 0; r < kRows; r++) s += __bfloat162float(S.da[r][j]);
                P[a.L.b1 + j] = s;
            }
        }
        if (threadIdx.x == 0) P[a.L.total] = S.loss[0] + S.loss[1] + S.loss[2] + S.loss[3];
        __syncthreads();
    }
}

// Targets of at least kFracMin among the rows of a batch, into *count (zeroed before).
__global__ void k_count(int64_t rows, int n_out, const float *Y, const int32_t *index, int *count) {
    int n = 0;
    for (int64_t t = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; t < rows * n_out; t += (int64_t)gridDim.x * blockDim.x) {
        const int64_t r = t / n_out;
        n += Y[(index ? (int64_t)index[r] : r) * n_out + (t - r * n_out)] >= kFracMin;
    }
    n = __reduce_add_sync(0xffffffffu, n);
    if ((threadIdx.x & 31) == 0 && n) atomicAdd(count, n);
}

__global__ void __launch_bounds__(64) k_grad_reduce(const float *__restrict__ partial, int nblk, int64_t stride,
                                                      int64_t total, float *grad, double *loss) {
    const int64_t t = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
    if (t > total) return;
    double s = 0.0;
#pragma unroll 16
    for (int b = 0; b < nblk; b++) s += (double)partial[(size_t)b * stride + t];
    if (t == total) *loss = s;
    else grad[t] = (float)s;
}

__global__ void k_refresh_bf16(const float *theta, Layout L, BfWeights w) {
    const int t = blockIdx.x * blockDim.x + threadIdx.x;
    if (t < kHid * kHid) {
        const int i = t / kHid, j = t - (t / kHid) * kHid;   // W[i][j], i = in, j = out
        w.W2T[j * kHid + i] = __float2bfloat16(theta[L.W2 + t]);
        w.W3T[j * kHid + i] = __float2bfloat16(theta[L.W3 + t]);
    }
    if (t < kHid * L.npad) {
        const int i = t / L.npad, j = t - (t / L.npad) * L.npad;
        const float v = j < L.n_out ? theta[L.W4 + i * L.n_out + j] : 0.f;
        w.W4T[j * kHid + i] = __float2bfloat16(v);
    }
}

__global__ void k_adam(float *theta, float *m, float *v, const float *grad, int64_t n, float lr, float b1, float b2,
                       float eps, float c1, float c2) {
    const int64_t t = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
    if (t >= n) return;
    const float g = grad[t];
    const float mt = b1 * m[t] + (1.f - b1) * g;
    const float vt = b2 * v[t] + (1.f - b2) * g * g;
    m[t] = mt;
    v[t] = vt;
    theta[t] -= lr * (mt / c1) / (sqrtf(vt / c2) + eps);
}

// Features per cell (FP64): log10 n_coll, log10 T, log10 |grad v| (least-squares velocity
// gradient over the neighbours, regularised by 1e-6 tr/3), log10 of the Sobolev optical
// depth of line 0 at LTE populations with velocity scale max(|grad v|, b / l), l the mean
// neighbour distance.
__global__ void k_features(int64_t n, const double *pos, const double *vel, const int64_t *off, const int32_t *idx,
                           const double *T, const double *ncoll, const double *nspec, const double *b, int nlev,
                           const double *E, const double *g, LineConst l0, float *out) {
    const int64_t c = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
    if (c >= n) return;
    double M[3][3] = {{0, 0, 0}, {0, 0, 0}, {0, 0, 0}}, B[3][3] = {{0, 0, 0}, {0, 0, 0}, {0, 0, 0}};
    double ell = 0.0;
    const int64_t e0 = off[c], e1 = off[c + 1];
    for (int64_t e = e0; e < e1; e++) {
        const int64_t m = idx[e];
        double dx[3], dv[3];
        for (int k = 0; k < 3; k++) {
            dx[k] = pos[3 * m + k] - pos[3 * c + k];
            dv[k] = vel[3 * m + k] - vel[3 * c + k];
        }
        ell += sqrt(dx[0] * dx[0] + dx[1] * dx[1] + dx[2] * dx[2]);
        for (int i = 0; i < 3; i++)
            for (int j = 0; j < 3; j++) {
                M[i][j] += dx[i] * dx[j];
                B[i][j] += dv[i] * dx[j];
            }
    }
    double gv = 0.0;
    if (e1 > e0) {
        ell /= (double)(e1 - e0);
        const double reg = 1e-6 * (M[0][0] + M[1][1] + M[2][2]) / 3.0;
        for (int i = 0; i < 3; i++) M[i][i] += reg;
        // inverse of the symmetric 3x3 matrix by cofactors
        const double c00 = M[1][1] * M[2][2] - M[1][2] * M[2][1], c01 = M[1][2] * M[2][0] - M[1][0] * M[2][2],
                     c02 = M[1][0] * M[2][1] - M[1][1] * M[2][0];
        const double det = M[0][0] * c00 + M[0][1] * c01 + M[0][2] * c02;
        double Mi[3][3];
        Mi[0][0] = c00 / det; Mi[1][0] = c01 / det; Mi[2][0] = c02 / det;
        Mi[0][1] = (M[0][2] * M[2][1] - M[0][1] * M[2][2]) / det;
        Mi[1][1] = (M[0][0] * M[2][2] - M[0][2] * M[2][0]) / det;
        Mi[2][1] = (M[0][1] * M[2][0] - M[0][0] * M[2][1]) / det;
        Mi[0][2] = (M[0][1] * M[1][2] - M[0][2] * M[1][1]) / det;
        Mi[1][2] = (M[0][2] * M[1][0] - M[0][0] * M[1][2]) / det;
        Mi[2][2] = (M[0][0] * M[1][1] - M[0][1] * M[1][0]) / det;
        for (int i = 0; i < 3; i++)
            for (int j = 0; j < 3; j++) {
                const double G = B[i][0] * Mi[0][j] + B[i][1] * Mi[1][j] + B[i][2] * Mi[2][j];
                gv += G * G;
            }
        gv = sqrt(gv);
    } else {
        ell = 1.0;
    }
    const double ikT = 1.0 / (kKB * T[c]);
    double Z = 0.0;
    for (int i = 0; i < nlev; i++) Z += g[i] * exp(-E[i] * ikT);
    const double nl = nspec[c] * g[l0.lo] * exp(-E[l0.lo] * ikT) / Z;
    const double nu_ = nspec[c] * g[l0.up] * exp(-E[l0.up] * ikT) / Z;
    const double chi_int = l0.pre * (nl * l0.Blu - nu_ * l0.Bul);
    const double vs = fmax(gv, b[c] / ell);
    const double tau = chi_int * kC / (l0.nu * vs);
    out[4 * c + 0] = (float)log10(ncoll[c]);
    out[4 * c + 1] = (float)log10(T[c]);
    out[4 * c + 2] = (float)log10(fmax(gv, 1e-30));
    out[4 * c + 3] = (float)log10(fmax(tau, 1e-30));
}

// Populations n_i = n_species exp(log p_i); a row with a non-finite output keeps LTE.
__global__ void k_pops_from_logp(int64_t n, int nlev, const float *logp, const double *nspec, double *pops,
                                 unsigned long long *bad) {
    const int64_t c = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
    if (c >= n) return;
    bool ok = true;
    for (int i = 0; i < nlev; i++) ok = ok && isfinite(logp[c * nlev + i]);
    if (!ok) { atomicAdd(bad, 1ull); return; }
    double s = 0.0;
    for (int i = 0; i < nlev; i++) s += exp((double)logp[c * nlev + i]);
    for (int i = 0; i < nlev; i++) pops[c * nlev + i] = nspec[c] * exp((double)logp[c * nlev + i]) / s;
}

}  // namespace

struct mg_mlp {
    int device = 0;
    cudaStream_t stream = nullptr;
    Layout L{};
    float *theta = nullptr, *m = nullptr, *v = nullptr, *grad = nullptr;
    BfWeights w{};
    __nv_bfloat16 *wbuf = nullptr;
    float mean[kIn] = {0, 0, 0, 0}, istd[kIn] = {1, 1, 1, 1};
    int64_t step = 0;
    std::string err;
    // workspace of loss_grad and train, one at a time (`busy`), other threads wait: inputs,
    // targets, row indices, per-CTA partials, losses and target counts (kept up to 256 MB each)
    std::mutex busy;
    float *wX = nullptr, *wY = nullptr, *wP = nullptr;
    int32_t *wI = nullptr;
    double *wL = nullptr;
    int *wC = nullptr;
    size_t cX = 0, cY = 0, cP = 0, cI = 0, cL = 0, cC = 0;
};

static int mfail(mg_mlp *p, int code, const std::string &msg) {
    if (p) p->err = msg;
    return code;
}

#define M_CUDA(call)                                                                            \
    do {                                                                                        \
        cudaError_t e_ = (call);                                                                \
        if (e_ != cudaSuccess) return mfail(p, MG_ERR_CUDA, std::string(#call ": ") + cudaGetErrorString(e_)); \
    } while (0)

static void refresh(mg_mlp *p) {
    k_refresh_bf16<<<(kHid * kHid + 255) / 256, 256, 0, p->stream>>>(p->theta, p->L, p->w);
}

extern "C" int mg_mlp_create(mg_mlp **out, int32_t n_out, uint64_t seed, int32_t device) {
    if (!out || n_out < 2 || n_out > kMaxOut) return MG_ERR_ARG;
    mg_mlp *p = new mg_mlp();
    p->device = device;
    p->L = make_layout(n_out);
    if (cudaSetDevice(device) != cudaSuccess || cudaStreamCreateWithFlags(&p->stream, cudaStreamNonBlocking) != cudaSuccess) {
        delete p;
        return MG_ERR_CUDA;
    }
    const int64_t T = p->L.total;
    const size_t nbf = 2 * (size_t)kHid * kHid + (size_t)kHid * kMaxOut;
    if (cudaMalloc(&p->theta, 4 * T) || cudaMalloc(&p->m, 4 * T) || cudaMalloc(&p->v, 4 * T) ||
        cudaMalloc(&p->grad, 4 * T) || cudaMalloc(&p->wbuf, 2 * nbf)) {
        mg_mlp_destroy(p);
        return MG_ERR_OOM;
    }
    p->w.W2T = p->wbuf;
    p->w.W3T = p->w.W2T + kHid * kHid;
    p->w.W4T = p->w.W3T + kHid * kHid;
    // He-uniform initial weights from a seeded generator, zero biases
    std::mt19937_64 rng(seed);
    std::vector<float> th(T, 0.f);
    auto fill = [&](int64_t o, int fan_in, int64_t cnt) {
        std::uniform_real_distribution<double> U(-std::sqrt(6.0 / fan_in), std::sqrt(6.0 / fan_in));
        for (int64_t k = 0; k < cnt; k++) th[o + k] = (float)U(rng);
    };
    fill(p->L.W1, kIn, kIn * kHid);
    fill(p->L.W2, kHid, kHid * kHid);
    fill(p->L.W3, kHid, kHid * kHid);
    fill(p->L.W4, kHid, kHid * n_out);
    cudaMemcpyAsync(p->theta, th.data(), 4 * T, cudaMemcpyHostToDevice, p->stream);
    cudaMemsetAsync(p->m, 0, 4 * T, p->stream);
    cudaMemsetAsync(p->v, 0, 4 * T, p->stream);
    refresh(p);
    if (cudaStreamSynchronize(p->stream) != cudaSuccess) { mg_mlp_destroy(p); return MG_ERR_CUDA; }
    *out = p;
    return MG_OK;
}

extern "C" int mg_mlp_destroy(mg_mlp *p) {
    if (!p) return MG_OK;
    cudaSetDevice(p->device);
    if (p->stream) cudaStreamSynchronize(p->stream);
    cudaFree(p->wX); cudaFree(p->wY); cudaFree(p->wP); cudaFree(p->wI); cudaFree(p->wL); cudaFree(p->wC);
    cudaFree(p->theta); cudaFree(p->m); cudaFree(p->v); cudaFree(p->grad); cudaFree(p->wbuf);
    if (p->stream) cudaStreamDestroy(p->stream);
    delete p;
    return MG_OK;
}

extern "C" const char *mg_mlp_last_error(const mg_mlp *p) { return p ? p->err.c_str() : "null network"; }

extern "C" int mg_mlp_param_count(const mg_mlp *p, int64_t *count) {
    if (!p || !count) return MG_ERR_ARG;
    *count = p->L.total;
    return MG_OK;
}

extern "C" int mg_mlp_set_params(mg_mlp *p, const float *theta, int64_t count) {
    if (!p || !theta || count != p->L.total) return MG_ERR_ARG;
    cudaSetDevice(p->device);
    M_CUDA(cudaMemcpyAsync(p->theta, theta, 4 * count, cudaMemcpyHostToDevice, p->stream));
    M_CUDA(cudaMemsetAsync(p->m, 0, 4 * count, p->stream));
    M_CUDA(cudaMemsetAsync(p->v, 0, 4 * count, p->stream));
    p->step = 0;
    refresh(p);
    M_CUDA(cudaStreamSynchronize(p->stream));
    return MG_OK;
}

extern "C" int mg_mlp_get_params(const mg_mlp *cp, float *theta, int64_t count) {
    mg_mlp *p = const_cast<mg_mlp *>(cp);
    if (!p || !theta || count != p->L.total) return MG_ERR_ARG;
    cudaSetDevice(p->device);
    M_CUDA(cudaMemcpyAsync(theta, p->theta, 4 * count, cudaMemcpyDeviceToHost, p->stream));
    M_CUDA(cudaStreamSynchronize(p->stream));
    return MG_OK;
}

extern "C" int mg_mlp_set_normalisation(mg_mlp *p, const float *mean, const float *stdv) {
    if (!p || !mean || !stdv) return MG_ERR_ARG;
    for (int i = 0; i < kIn; i++) {
        if (!(stdv[i] > 0)) return mfail(p, MG_ERR_ARG, "normalisation: std must be > 0");
        p->mean[i] = mean[i];
        p->istd[i] = 1.f / stdv[i];
    }
    return MG_OK;
}

static TileArgs tile_args(mg_mlp *p, int64_t rows, const float *X, const int32_t *index, const float *Y, float *logp,
                          float *partial, const int *count) {
    TileArgs a{};
    a.rows = rows; a.X = X; a.index = index; a.Y = Y; a.theta = p->theta; a.w = p->w; a.L = p->L;
    for (int i = 0; i < kIn; i++) { a.mean[i] = p->mean[i]; a.istd[i] = p->istd[i]; }
    a.count = count; a.logp = logp; a.partial = partial;
    return a;
}

static int launch_tile(mg_mlp *p, const TileArgs &a) {
    int64_t blocks = (a.rows + kRows - 1) / kRows;
    // without gradients one CTA per SM takes several tiles
    if (!a.partial) blocks = std::min<int64_t>(blocks, 152);
    const size_t sm = sizeof(TileSmem);
    cudaFuncSetAttribute(k_mlp_tile, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)sm);
    k_mlp_tile<<<(unsigned)blocks, kTileThreads, sm, p->stream>>>(a);
    M_CUDA(cudaGetLastError());
    return MG_OK;
}

// Device-pointer forward pass: X [rows][4] raw features -> logp [rows][n_out].
int mg_mlp_forward_dev(mg_mlp *p, int64_t rows, const float *d_X, float *d_logp, cudaStream_t s) {
    cudaStream_t keep = p->stream;
    p->stream = s;
    int rc = launch_tile(p, tile_args(p, rows, d_X, nullptr, nullptr, d_logp, nullptr, nullptr));
    p->stream = keep;
    return rc;
}

// Grows a workspace buffer. (Buffers larger than 256 MB are not kept: see release.)
template <typename T>
static int reserve(mg_mlp *p, T *&buf, size_t &cap, size_t count) {
    if (cap >= count) return MG_OK;
    cudaFree(buf);
    buf = nullptr;
    cap = 0;
    M_CUDA(cudaMalloc(&buf, sizeof(T) * count));
    cap = count;
    return MG_OK;
}
template <typename T>
static void release(T *&buf, size_t &cap) {
    if (sizeof(T) * cap <= (256u << 20)) return;
    cudaFree(buf);
    buf = nullptr;
    cap = 0;
}
static int done(mg_mlp *p, int rc) {
    release(p->wX, p->cX);
    release(p->wY, p->cY);
    release(p->wP, p->cP);
    release(p->wI, p->cI);
    return rc;
}

extern "C" int mg_mlp_forward(mg_mlp *p, int64_t rows, const float *X, float *logp) {
    if (!p || rows < 1 || !X || !logp) return MG_ERR_ARG;
    cudaSetDevice(p->device);
    float *dX = nullptr, *dL = nullptr;   // (not the workspace: threads may share a network's forward pass)
    M_CUDA(cudaMalloc(&dX, 16 * rows));
    M_CUDA(cudaMalloc(&dL, 4 * rows * p->L.n_out));
    M_CUDA(cudaMemcpyAsync(dX, X, 16 * rows, cudaMemcpyHostToDevice, p->stream));
    int rc = launch_tile(p, tile_args(p, rows, dX, nullptr, nullptr, dL, nullptr, nullptr));
    if (!rc) {
        M_CUDA(cudaMemcpyAsync(logp, dL, 4 * rows * p->L.n_out, cudaMemcpyDeviceToHost, p->stream));
        M_CUDA(cudaStreamSynchronize(p->stream));
    }
    cudaFree(dX);
    cudaFree(dL);
    return rc;
}

// One gradient evaluation over device rows (index optional); leaves grad in p->grad, the sum
// of squares in *dloss and the number of targets in *dcount.
static int grad_dev(mg_mlp *p, int64_t rows, const float *dX, const int32_t *didx, const float *dY, float *dpart,
                    double *dloss, int *dcount) {
    const int64_t blocks = (rows + kRows - 1) / kRows, m = rows * p->L.n_out;
    M_CUDA(cudaMemsetAsync(dcount, 0, sizeof(int), p->stream));
    k_count<<<(unsigned)std::min<int64_t>(304, (m + 1023) / 1024), 256, 0, p->stream>>>(rows, p->L.n_out, dY, didx, dcount);
    int rc = launch_tile(p, tile_args(p, rows, dX, didx, dY, nullptr, dpart, dcount));
    if (rc) return rc;
    k_grad_reduce<<<(unsigned)(p->L.total / 64 + 1), 64, 0, p->stream>>>(dpart, (int)blocks, partial_stride(p->L),
                                                                       p->L.total, p->grad, dloss);
    M_CUDA(cudaGetLastError());
    return MG_OK;
}

static int loss_grad_host(mg_mlp *p, int64_t rows, const float *X, const float *Y, double *loss, float *grad) {
    const int n_out = p->L.n_out;
    const int64_t blocks = (rows + kRows - 1) / kRows, stride = partial_stride(p->L);
    int rc;
    if ((rc = reserve(p, p->wX, p->cX, 4 * rows)) || (rc = reserve(p, p->wY, p->cY, rows * n_out)) ||
        (rc = reserve(p, p->wP, p->cP, blocks * stride)) || (rc = reserve(p, p->wL, p->cL, 1)) ||
        (rc = reserve(p, p->wC, p->cC, 1)))
        return rc;
    M_CUDA(cudaMemcpyAsync(p->wX, X, 16 * rows, cudaMemcpyHostToDevice, p->stream));
    M_CUDA(cudaMemcpyAsync(p->wY, Y, 4 * rows * n_out, cudaMemcpyHostToDevice, p->stream));
    if ((rc = grad_dev(p, rows, p->wX, nullptr, p->wY, p->wP, p->wL, p->wC))) return rc;
    double lsum = 0.0;
    int cnt = 0;
    if (grad) M_CUDA(cudaMemcpyAsync(grad, p->grad, 4 * p->L.total, cudaMemcpyDeviceToHost, p->stream));
    M_CUDA(cudaMemcpyAsync(&lsum, p->wL, 8, cudaMemcpyDeviceToHost, p->stream));
    M_CUDA(cudaMemcpyAsync(&cnt, p->wC, 4, cudaMemcpyDeviceToHost, p->stream));
    M_CUDA(cudaStreamSynchronize(p->stream));
    if (loss) *loss = lsum * (cnt ? 1.f / (float)cnt : 0.f);
    return MG_OK;
}

extern "C" int mg_mlp_loss_grad(mg_mlp *p, int64_t rows, const float *X, const float *Y, double *loss, float *grad) {
    if (!p || rows < 1 || !X || !Y) return MG_ERR_ARG;
    std::lock_guard<std::mutex> own(p->busy);
    cudaSetDevice(p->device);
    return done(p, loss_grad_host(p, rows, X, Y, loss, grad));
}

static int train_host(mg_mlp *p, int64_t rows, const float *X, const float *Y, const mg_train_opts *o,
                      mg_train_report &r) {
    const int n_out = p->L.n_out;
    const int64_t B = o->batch, stride = partial_stride(p->L), blocks = (B + kRows - 1) / kRows;
    const int64_t steps = std::max<int64_t>(1, rows / B);   // per epoch
    int rc;
    if ((rc = reserve(p, p->wX, p->cX, 4 * rows)) || (rc = reserve(p, p->wY, p->cY, rows * n_out)) ||
        (rc = reserve(p, p->wI, p->cI, rows)) || (rc = reserve(p, p->wP, p->cP, blocks * stride)) ||
        (rc = reserve(p, p->wL, p->cL, steps)) || (rc = reserve(p, p->wC, p->cC, steps)))
        return rc;
    M_CUDA(cudaMemcpyAsync(p->wX, X, 16 * rows, cudaMemcpyHostToDevice, p->stream));
    M_CUDA(cudaMemcpyAsync(p->wY, Y, 4 * rows * n_out, cudaMemcpyHostToDevice, p->stream));
    std::vector<int32_t> idx(rows);
    std::vector<double> lsum(steps);
    std::vector<int> cnt(steps);
    std::mt19937_64 rng(o->seed);
    for (int ep = 0; ep < o->epochs; ep++) {
        for (int64_t i = 0; i < rows; i++) idx[i] = (int32_t)i;
        std::shuffle(idx.begin(), idx.end(), rng);
        M_CUDA(cudaMemcpyAsync(p->wI, idx.data(), 4 * rows, cudaMemcpyHostToDevice, p->stream));
        int64_t nb = 0;
        for (int64_t s = 0; s + B <= rows || (s == 0 && rows < B); s += B, nb++) {
            const int64_t nr = std::min<int64_t>(B, rows - s);
            if ((rc = grad_dev(p, nr, p->wX, p->wI + s, p->wY, p->wP, p->wL + nb, p->wC + nb))) return rc;
            p->step++;
            const float c1 = 1.f - std::pow(0.9f, (float)p->step), c2 = 1.f - std::pow(0.999f, (float)p->step);
            k_adam<<<(unsigned)((p->L.total + 255) / 256), 256, 0, p->stream>>>(p->theta, p->m, p->v, p->grad,
                                                                                 p->L.total, o->lr, 0.9f, 0.999f,
                                                                                 1e-8f, c1, c2);
            refresh(p);
            r.steps++;
        }
        // the epoch's losses (and the indices' buffer is free for the next shuffle)
        M_CUDA(cudaMemcpyAsync(lsum.data(), p->wL, 8 * nb, cudaMemcpyDeviceToHost, p->stream));
        M_CUDA(cudaMemcpyAsync(cnt.data(), p->wC, 4 * nb, cudaMemcpyDeviceToHost, p->stream));
        M_CUDA(cudaStreamSynchronize(p->stream));
        double ep_loss = 0.0;
        for (int64_t k = 0; k < nb; k++) ep_loss += lsum[k] * (cnt[k] ? 1.f / (float)cnt[k] : 0.f);
        if (nb) {
            if (r.first_loss < 0) r.first_loss = ep_loss / nb;
            r.last_loss = ep_loss / nb;
        }
    }
    return MG_OK;
}

extern "C" int mg_mlp_train(mg_mlp *p, int64_t rows, const float *X, const float *Y, const mg_train_opts *o,
                            mg_train_report *rep) {
    if (!p || rows < 1 || !X || !Y || !o || o->epochs < 1 || o->batch < kRows || !(o->lr > 0)) return MG_ERR_ARG;
    std::lock_guard<std::mutex> own(p->busy);
    cudaSetDevice(p->device);
    auto t0 = std::chrono::steady_clock::now();
    mg_train_report r{};
    r.first_loss = -1;
    const int rc = done(p, train_host(p, rows, X, Y, o, r));
    r.seconds = std::chrono::duration<double>(std::chrono::steady_clock::now() - t0).count();
    if (rep) *rep = r;
    return rc;
}

// ---------------------------------------------------------------- context side
extern "C" int mg_features(mg_ctx *ctx, float *out) {
    if (!ctx || !out) return MG_ERR_ARG;
    if (!ctx->have_mesh || !ctx->have_model || !ctx->have_species)
        return mg_fail(ctx, MG_ERR_STATE, "mg_features: needs mesh, model and species");
    cudaSetDevice(ctx->device);
    float *d = nullptr;
    int rc;
    if ((rc = mg_alloc(ctx, &d, 4 * ctx->n))) return rc;
    k_features<<<(unsigned)((ctx->n + 127) / 128), 128, 0, ctx->stream>>>(
        ctx->n, ctx->d_pos, ctx->d_vel, ctx->d_nbr_off, ctx->d_nbr_idx, ctx->d_T, ctx->d_ncoll, ctx->d_nspec, ctx->d_b,
        ctx->n_lev, ctx->d_E, ctx->d_g, ctx->h_lines[0], d);
    cudaError_t e = cudaMemcpyAsync(out, d, 16 * ctx->n, cudaMemcpyDeviceToHost, ctx->stream);
    if (e == cudaSuccess) e = cudaStreamSynchronize(ctx->stream);
    cudaFree(d);
    if (e != cudaSuccess) return mg_cuda_check(ctx, e, "mg_features");
    return MG_OK;
}

extern "C" int mg_init_populations_mlp(mg_ctx *ctx, mg_mlp *p) {
    if (!ctx || !p) return MG_ERR_ARG;
    if (!ctx->have_mesh || !ctx->have_model || !ctx->have_species)
        return mg_fail(ctx, MG_ERR_STATE, "mg_init_populations_mlp: needs mesh, model and species");
    if (p->L.n_out != ctx->n_lev) return mg_fail(ctx, MG_ERR_ARG, "mg_init_populations_mlp: network outputs != levels");
    cudaSetDevice(ctx->device);
    int rc;
    if ((rc = mg_init_populations(ctx, MG_INIT_LTE))) return rc;   // fallback for rows the network cannot give
    float *dF = nullptr, *dL = nullptr;
    if ((rc = mg_alloc(ctx, &dF, 4 * ctx->n))) return rc;
    if ((rc = mg_alloc(ctx, &dL, ctx->n * ctx->n_lev))) {
        cudaFree(dF);
        return rc;
    }
    k_features<<<(unsigned)((ctx->n + 127) / 128), 128, 0, ctx->stream>>>(
        ctx->n, ctx->d_pos, ctx->d_vel, ctx->d_nbr_off, ctx->d_nbr_idx, ctx->d_T, ctx->d_ncoll, ctx->d_nspec, ctx->d_b,
        ctx->n_lev, ctx->d_E, ctx->d_g, ctx->h_lines[0], dF);
    rc = mg_mlp_forward_dev(p, ctx->n, dF, dL, ctx->stream);
    if (!rc) {
        cudaMemsetAsync(ctx->d_scal + 5, 0, 8, ctx->stream);
        k_pops_from_logp<<<(unsigned)((ctx->n + 127) / 128), 128, 0, ctx->stream>>>(ctx->n, ctx->n_lev, dL,
                                                                                   ctx->d_nspec, ctx->d_pops,
                                                                                   ctx->d_scal + 5);
        unsigned long long bad = 0;
        cudaMemcpyAsync(&bad, ctx->d_scal + 5, 8, cudaMemcpyDeviceToHost, ctx->stream);
        cudaStreamSynchronize(ctx->stream);
        ctx->last_fallback = (int64_t)bad;
    }
    cudaFree(dF);
    cudaFree(dL);
    mg_band_restart(ctx);
    ctx->have_pops = true;
    ctx->have_rad = false;
    return rc;
}

extern "C" int mg_attach_mlp(mg_ctx *ctx, mg_mlp *p) {
    if (!ctx) return MG_ERR_ARG;
    if (p && ctx->have_species && p->L.n_out != ctx->n_lev)
        return mg_fail(ctx, MG_ERR_ARG, "mg_attach_mlp: network outputs != levels");
    ctx->mlp = p;
    return MG_OK;
}

// ------------------------------------------------------------------ file format
static const char kMagic[8] = {'M', 'G', 'M', 'L', 'P', '0', '0', '1'};

extern "C" int mg_mlp_save(const mg_mlp *cp, const char *path) {
    mg_mlp *p = const_cast<mg_mlp *>(cp);
    if (!p || !path) return MG_ERR_ARG;
    std::vector<float> th(p->L.total);
    int rc = mg_mlp_get_params(p, th.data(), p->L.total);
    if (rc) return rc;
    FILE *f = std::fopen(path, "wb");
    if (!f) return mfail(p, MG_ERR_ARG, std::string("mg_mlp_save: cannot open ") + path);
    const int32_t hdr[2] = {p->L.n_out, 0};
    const int64_t np = p->L.total;
    float mean[kIn], sd[kIn];
    for (int i = 0; i < kIn; i++) { mean[i] = p->mean[i]; sd[i] = 1.f / p->istd[i]; }
    bool ok = std::fwrite(kMagic, 1, 8, f) == 8 && std::fwrite(hdr, 4, 2, f) == 2 && std::fwrite(&np, 8, 1, f) == 1 &&
              std::fwrite(mean, 4, kIn, f) == (size_t)kIn && std::fwrite(sd, 4, kIn, f) == (size_t)kIn &&
              std::fwrite(th.data(), 4, th.size(), f) == th.size();
    ok = (std::fclose(f) == 0) && ok;
    return ok ? MG_OK : mfail(p, MG_ERR_ARG, std::string("mg_mlp_save: short write to ") + path);
}

extern "C" int mg_mlp_load(mg_mlp **out, const char *path, int32_t device) {
    if (!out || !path) return MG_ERR_ARG;
    *out = nullptr;
    FILE *f = std::fopen(path, "rb");
    if (!f) return MG_ERR_ARG;
    char magic[8];
    int32_t hdr[2];
    int64_t np = 0;
    float mean[kIn], sd[kIn];
    bool ok = std::fread(magic, 1, 8, f) == 8 && std::memcmp(magic, kMagic, 8) == 0 &&
              std::fread(hdr, 4, 2, f) == 2 && std::fread(&np, 8, 1, f) == 1 &&
              std::fread(mean, 4, kIn, f) == (size_t)kIn && std::fread(sd, 4, kIn, f) == (size_t)kIn &&
              hdr[0] >= 2 && hdr[0] <= kMaxOut && np == make_layout(hdr[0]).total;
    std::vector<float> th(ok ? (size_t)np : 0);
    ok = ok && std::fread(th.data(), 4, th.size(), f) == th.size();
    std::fclose(f);
    if (!ok) return MG_ERR_ARG;
    mg_mlp *p = nullptr;
    int rc = mg_mlp_create(&p, hdr[0], 0, device);
    if (rc) return rc;
    if ((rc = mg_mlp_set_params(p, th.data(), np)) || (rc = mg_mlp_set_normalisation(p, mean, sd))) {
        mg_mlp_destroy(p);
        return rc;
    }
    *out = p;
    return MG_OK;
}
