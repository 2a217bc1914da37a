// mlp.cu -- the force/torque surrogate network of the particle predictor:
// 34 inputs -> three hidden layers of 128 exact-GELU units -> 6 outputs, on
// standardised inputs and outputs, trained on trajectories the solver logs.
// (Not in the paper, whose only predictor is the orientation
// predictor-corrector of Sec. 2.3; it predicts F(t+1), T(t+1) for the marker
// velocities of the immersed-boundary step, Sec. 2.2.)
//
// Kernels (precision 0, BF16 tensor cores, mma.sync m16n8k16 with FP32
// accumulation; the products are at most 4096x128x128, where the rate of the
// matrix unit does not show):
//   k_rows        32 rows per block (outputs of many rows: 128): the four layers
//                 with the BF16 weights and all activations in shared memory;
//                 with training also the loss, and the backward pass down to
//                 the first layer
//   k_wgrad       weight and bias gradients of one 256-row slice per block row
//   k_update      sum of the slices in order, AdamW and the BF16 copy
// The predictor in the step runs up to 16 samples per block (mlp_infer_rows).
// Precision 1 (an FP32 check mode): k_gemm, k_mlp_infer and the layer-by-layer
// passes.
// Fixed summation orders, no atomics on data: deterministic.
#include <cuda_bf16.h>
#include <cuda_runtime.h>
#include <math.h>
#include <string.h>

#include <string>
#include <vector>

#include "../../include/turret.h"
#include "turret_internal.cuh"

using namespace turret;

namespace turret {

__device__ __forceinline__ float gelu_f(float x) { return 0.5f * x * (1.0f + erff(x * 0.70710678118654752f)); }
__device__ __forceinline__ float gelu_prime_f(float x) {
    return 0.5f * (1.0f + erff(x * 0.70710678118654752f)) + x * 0.39894228040143268f * expf(-0.5f * x * x);
}

__device__ __forceinline__ void mma_bf16(float (&d)[4], const uint32_t (&a)[4], const uint32_t (&b)[2]) {
    asm volatile(
        "mma.sync.aligned.m16n8k16.row.col.f32.bf16.bf16.f32 {%0,%1,%2,%3}, {%4,%5,%6,%7}, {%8,%9}, "
        "{%0,%1,%2,%3};\n"
        : "+f"(d[0]), "+f"(d[1]), "+f"(d[2]), "+f"(d[3])
        : "r"(a[0]), "r"(a[1]), "r"(a[2]), "r"(a[3]), "r"(b[0]), "r"(b[1]));
}

__device__ __forceinline__ uint32_t ld_pair(const __nv_bfloat16 *p) { return *reinterpret_cast<const uint32_t *>(p); }

// ---------------------------------------------------------------------------
// GEMM of the FP32 check mode.  A(m, k) = ta ? A[k * lda + m] : A[m * lda + k];
//        B(k, n) = tb ? B[k * ldb + n] : B[n * ldb + k]   (tb = 0: weights [N][K]).
struct GemmArgs {
    const float *A;
    const float *B;
    float *C;
    const float *bias;  // [N], added when non-null
    float *Aout;        // EPI_GELU: gelu of the result
    const float *Zg;    // EPI_DGELU: the result times gelu'(Zg)
    int lda, ldb, ldc, ldo, ldz;
    int ta, tb;
    int M, N, K;
    int kslice;         // > 0: block z sums K range [z kslice, (z+1) kslice) into part[z][M][N]
    float *part;
};
enum { EPI_STORE = 0, EPI_GELU = 1, EPI_DGELU = 2 };
// split-K of the weight-gradient products (reductions over the batch): slices
// of KSLICE rows, partial sums added in slice order by k_sum_slices
constexpr int KSLICE = 256, MAX_SLICES = 64;
constexpr int GBM = 64, GBN = 64, GBK = 32, GTHREADS = 128;

__device__ __forceinline__ void epilogue(const GemmArgs &g, int epi, int m, int n, float acc) {
    if (m >= g.M || n >= g.N) return;
    if (g.kslice > 0) {  // partial sum of this block's K slice
        g.part[((size_t)blockIdx.z * g.M + m) * g.N + n] = acc;
        return;
    }
    float v = acc + (g.bias ? g.bias[n] : 0.0f);
    if (epi == EPI_DGELU) v *= gelu_prime_f(g.Zg[(size_t)m * g.ldz + n]);
    g.C[(size_t)m * g.ldc + n] = v;
    if (epi == EPI_GELU) g.Aout[(size_t)m * g.ldo + n] = gelu_f(v);
}

__global__ void __launch_bounds__(GTHREADS) k_gemm(GemmArgs g, int epi) {
    __shared__ float As[GBM][GBK + 1];
    __shared__ float Bs[GBN][GBK + 1];
    const int tid = threadIdx.x;
    const int m0 = blockIdx.x * GBM, n0 = blockIdx.y * GBN;
    const int tr = tid >> 3, tc = tid & 7;  // rows 4 tr + i, columns tc + 8 j
    float sacc[4][8];
#pragma unroll
    for (int i = 0; i < 4; ++i)
#pragma unroll
        for (int j = 0; j < 8; ++j) sacc[i][j] = 0.0f;
    const int kbeg = g.kslice > 0 ? blockIdx.z * g.kslice : 0;
    const int kend = g.kslice > 0 ? min(g.K, kbeg + g.kslice) : g.K;
    for (int k0 = kbeg; k0 < kend; k0 += GBK) {
        // stage the A and B tiles (any layout -> [row][k]), zero outside the matrices
#pragma unroll 4
        for (int e = tid; e < GBM * GBK; e += GTHREADS) {
            int m, k;
            if (g.ta) { k = e / GBM; m = e % GBM; } else { m = e / GBK; k = e % GBK; }
            const int gm = m0 + m, gk = k0 + k;
            float v = 0.0f;
            if (gm < g.M && gk < kend) v = g.ta ? g.A[(size_t)gk * g.lda + gm] : g.A[(size_t)gm * g.lda + gk];
            As[m][k] = v;
        }
#pragma unroll 4
        for (int e = tid; e < GBN * GBK; e += GTHREADS) {
            int n, k;
            if (g.tb) { k = e / GBN; n = e % GBN; } else { n = e / GBK; k = e % GBK; }
            const int gn = n0 + n, gk = k0 + k;
            float v = 0.0f;
            if (gn < g.N && gk < kend) v = g.tb ? g.B[(size_t)gk * g.ldb + gn] : g.B[(size_t)gn * g.ldb + gk];
            Bs[n][k] = v;
        }
        __syncthreads();
#pragma unroll 4
        for (int k = 0; k < GBK; ++k)
#pragma unroll
            for (int i = 0; i < 4; ++i)
#pragma unroll
                for (int j = 0; j < 8; ++j) sacc[i][j] = fmaf(As[4 * tr + i][k], Bs[tc + 8 * j][k], sacc[i][j]);
        __syncthreads();
    }
#pragma unroll
    for (int i = 0; i < 4; ++i)
#pragma unroll
        for (int j = 0; j < 8; ++j) epilogue(g, epi, m0 + 4 * tr + i, n0 + tc + 8 * j, sacc[i][j]);
}

// ---------------------------------------------------------------------------
// Standardisation: x_s = (x - mean) / std (inputs and targets), and back.
__global__ void k_standardise(const float *__restrict__ x, int n, int d, const float *__restrict__ mean,
                              const float *__restrict__ stdv, float *__restrict__ out) {
    const int i = blockIdx.x * blockDim.x + threadIdx.x;
    if (i >= n * d) return;
    const int c = i % d;
    out[i] = (x[i] - mean[c]) / stdv[c];
}

__global__ void k_unstandardise(const float *__restrict__ y, int n, const float *__restrict__ mean,
                                const float *__restrict__ stdv, float *__restrict__ out) {
    const int i = blockIdx.x * blockDim.x + threadIdx.x;
    if (i >= n * MLP_OUT) return;
    const int c = i % MLP_OUT;
    out[i] = fmaf(y[i], stdv[c], mean[c]);
}

// Loss = mean over samples and outputs of (y - t)^2 (accumulated in FP64 in a
// fixed order) and dL/dy = 2 (y - t) / (6 n).
constexpr int LOSS_THREADS = 256;
__global__ void __launch_bounds__(LOSS_THREADS) k_loss(const float *__restrict__ y, const float *__restrict__ t,
                                                       int n, float *__restrict__ dy, double *__restrict__ loss) {
    __shared__ double part[LOSS_THREADS];
    const int total = n * MLP_OUT;
    const float sc = 2.0f / (float)total;
    double s = 0.0;
    for (int i = threadIdx.x; i < total; i += LOSS_THREADS) {
        const float e = y[i] - t[i];
        s += (double)e * (double)e;
        dy[i] = sc * e;
    }
    part[threadIdx.x] = s;
    __syncthreads();
    for (int w = LOSS_THREADS / 2; w > 0; w >>= 1) {
        if (threadIdx.x < w) part[threadIdx.x] += part[threadIdx.x + w];
        __syncthreads();
    }
    if (threadIdx.x == 0) *loss = part[0] / (double)total;
}

// Bias gradient, first pass: column sums of dZ [n][ld] over the rows of
// slice blockIdx.y (KSLICE rows, in row order) into part[slice][ncol].
__global__ void k_colsum(const float *__restrict__ dz, int n, int ncol, int ld, float *__restrict__ part) {
    const int c = blockIdx.x * blockDim.x + threadIdx.x;
    if (c >= ncol) return;
    const int r0 = blockIdx.y * KSLICE, r1 = min(n, r0 + KSLICE);
    float s = 0.0f;
    for (int r = r0; r < r1; ++r) s += dz[(size_t)r * ld + c];
    part[(size_t)blockIdx.y * ncol + c] = s;
}

// Sum of nsl partial results part[z][count] in slice order z = 0, 1, ...
__global__ void k_sum_slices(const float *__restrict__ part, int nsl, int count, float *__restrict__ out) {
    const int i = blockIdx.x * blockDim.x + threadIdx.x;
    if (i >= count) return;
    float s = part[i];
    for (int z = 1; z < nsl; ++z) s += part[(size_t)z * count + i];
    out[i] = s;
}

// Offsets of the flat parameter vector (W1 b1 W2 b2 W3 b3 W4 b4).
constexpr int OFF_W1 = 0, OFF_B1 = OFF_W1 + MLP_H * MLP_IN, OFF_W2 = OFF_B1 + MLP_H, OFF_B2 = OFF_W2 + MLP_H * MLP_H,
              OFF_W3 = OFF_B2 + MLP_H, OFF_B3 = OFF_W3 + MLP_H * MLP_H, OFF_W4 = OFF_B3 + MLP_H,
              OFF_B4 = OFF_W4 + MLP_OUT * MLP_H, OFF_END = OFF_B4 + MLP_OUT;
static_assert(OFF_END == MLP_NPARAM, "parameter layout");

__device__ __forceinline__ bool is_weight(int i) {
    return i < OFF_B1 || (i >= OFF_W2 && i < OFF_B2) || (i >= OFF_W3 && i < OFF_B3) || (i >= OFF_W4 && i < OFF_B4);
}

// BF16 copies of the weight matrices in the padded layout of the inference
// kernel: W1 [128][48] (columns 34..47 zero), W2, W3 [128][128], W4 [8][128]
// (rows 6, 7 zero).
constexpr int WB1 = 0, WB2 = WB1 + MLP_H * MLP_INP, WB3 = WB2 + MLP_H * MLP_H, WB4 = WB3 + MLP_H * MLP_H,
              WB_END = WB4 + MLP_OUTP * MLP_H;

__global__ void k_refresh_bf16(const float *__restrict__ P, __nv_bfloat16 *__restrict__ wb) {
    const int i = blockIdx.x * blockDim.x + threadIdx.x;
    if (i >= WB_END) return;
    float v = 0.0f;
    if (i < WB2) {
        const int r = i / MLP_INP, c = i % MLP_INP;
        v = c < MLP_IN ? P[OFF_W1 + r * MLP_IN + c] : 0.0f;
    } else if (i < WB3) {
        v = P[OFF_W2 + (i - WB2)];
    } else if (i < WB4) {
        v = P[OFF_W3 + (i - WB3)];
    } else {
        const int r = (i - WB4) / MLP_H, c = (i - WB4) % MLP_H;
        v = r < MLP_OUT ? P[OFF_W4 + r * MLP_H + c] : 0.0f;
    }
    wb[i] = __float2bfloat16_rn(v);
}

// AdamW (Loshchilov & Hutter): moments, bias correction, decoupled decay of
// the weight matrices.
__device__ __forceinline__ float adamw_value(float p, float g, float &m, float &v, bool weight, float lr, float b1,
                                             float b2, float eps, float wd, float bc1, float bc2) {
    m = b1 * m + (1.0f - b1) * g;
    v = b2 * v + (1.0f - b2) * g * g;
    const float upd = (m / bc1) / (sqrtf(v / bc2) + eps) + (weight ? wd * p : 0.0f);
    return p - lr * upd;
}

__global__ void k_adamw(float *__restrict__ P, const float *__restrict__ G, float *__restrict__ Mm,
                        float *__restrict__ Vv, float lr, float b1, float b2, float eps, float wd, float bc1,
                        float bc2) {
    const int i = blockIdx.x * blockDim.x + threadIdx.x;
    if (i >= MLP_NPARAM) return;
    // written out, not adamw_value: the compiler's choice of fused multiply-adds, and
    // with it the last bit of a parameter, follows the form of the expressions
    const float g = G[i];
    const float m = b1 * Mm[i] + (1.0f - b1) * g;
    const float v = b2 * Vv[i] + (1.0f - b2) * g * g;
    Mm[i] = m;
    Vv[i] = v;
    const float p = P[i];
    const float upd = (m / bc1) / (sqrtf(v / bc2) + eps) + (is_weight(i) ? wd * p : 0.0f);
    P[i] = p - lr * upd;
}

// ---------------------------------------------------------------------------
// The BF16 network on 32 rows per block of 256 threads.  Every layer is a
// 32 x 128 x 128 product (67 MFLOP over a batch of 4096): what it costs is
// passes over memory and launches, not the products.  So a block keeps the
// whole network in shared memory (78 KB of BF16 weights), its rows' operands
// beside it and the pre-activations z in the registers of the threads that
// need them again for GELU'(z) (the backward product's accumulator tile is the
// forward one's), and a training step is three launches instead of 28: batch
// 4096 took 367 us per step with a launch per product, sum and pass, and
// 42 us with k_rows, k_wgrad and k_update.  32 rows: 128 blocks at batch 4096,
// one per SM.  Operands are rounded to BF16 where the
// products take them, sums run in the k order of a 16-wide mma chain and
// weight gradients over 256-row slices in order.
constexpr int RT_ROWS = 32, RT_THREADS = 256;
// outputs of many rows: ROWS / 16 x 4 warps per block (launch_rows)
constexpr int RT_WIDE = 128;
constexpr int LDK = MLP_H + 8, LDX = MLP_INP + 8, LDY = 24;  // row strides (BF16) free of bank conflicts for ldmatrix

template <int ROWS>
struct RowsSmem {
    __nv_bfloat16 w1[MLP_H][LDX], w2[MLP_H][LDK], w3[MLP_H][LDK], w4[MLP_OUTP][LDK];
    __nv_bfloat16 x[ROWS][LDX];
    __nv_bfloat16 a[2][ROWS][LDK];  // the operand of the current layer and the one being formed
    __nv_bfloat16 dy[RT_ROWS][LDY];
    double loss[RT_THREADS / 32];
};

// What a training pass leaves for k_wgrad: the operands of the weight
// gradients, activations rounded to BF16 as the products take them, and the
// layer gradients in FP32.
struct TrainOut {
    __nv_bfloat16 *x;     // [n][48] standardised inputs
    __nv_bfloat16 *a[3];  // [n][128]
    float *dz[3];         // [n][128]
    float *dy;            // [n][6]
    double *loss;         // per block: sum of squared errors
};

__device__ __forceinline__ uint32_t smem_u32(const void *p) { return (uint32_t)__cvta_generic_to_shared(p); }
__device__ __forceinline__ void ldsm4(uint32_t (&r)[4], const void *p) {
    asm volatile("ldmatrix.sync.aligned.m8n8.x4.shared.b16 {%0,%1,%2,%3}, [%4];"
                 : "=r"(r[0]), "=r"(r[1]), "=r"(r[2]), "=r"(r[3]) : "r"(smem_u32(p)) : "memory");
}
__device__ __forceinline__ void ldsm4t(uint32_t (&r)[4], const void *p) {
    asm volatile("ldmatrix.sync.aligned.m8n8.x4.trans.shared.b16 {%0,%1,%2,%3}, [%4];"
                 : "=r"(r[0]), "=r"(r[1]), "=r"(r[2]), "=r"(r[3]) : "r"(smem_u32(p)) : "memory");
}
__device__ __forceinline__ uint32_t pack_bf16(float lo, float hi) {
    const __nv_bfloat162 v = __floats2bfloat162_rn(lo, hi);
    return *reinterpret_cast<const uint32_t *>(&v);
}

// acc (16 rows at m0 x 32 columns at n0) = A [.][K] W^T with W [n][K], K in 16-wide steps
template <int LDA, int LDW>
__device__ __forceinline__ void rows_product(const __nv_bfloat16 (*A)[LDA], const __nv_bfloat16 (*W)[LDW], int K, int m0,
                                             int n0, float (&acc)[4][4]) {
    const int lane = threadIdx.x & 31;
#pragma unroll
    for (int j = 0; j < 4; ++j)
#pragma unroll
        for (int q = 0; q < 4; ++q) acc[j][q] = 0.0f;
#pragma unroll
    for (int k = 0; k < K; k += 16) {
        uint32_t a[4], b[2][4];
        ldsm4(a, &A[m0 + (lane & 15)][k + (lane >> 4) * 8]);
#pragma unroll
        for (int h = 0; h < 2; ++h) ldsm4(b[h], &W[n0 + 16 * h + (lane & 7) + (lane >> 4) * 8][k + ((lane >> 3) & 1) * 8]);
#pragma unroll
        for (int j = 0; j < 4; ++j) {
            const uint32_t bj[2] = {b[j >> 1][2 * (j & 1)], b[j >> 1][2 * (j & 1) + 1]};
            mma_bf16(acc[j], a, bj);
        }
    }
}

// acc = A [.][K] W with W [K][n]: the backward product, W read transposed
template <int LDA, int LDW>
__device__ __forceinline__ void rows_product_t(const __nv_bfloat16 (*A)[LDA], const __nv_bfloat16 (*W)[LDW], int K,
                                               int m0, int n0, float (&acc)[4][4]) {
    const int lane = threadIdx.x & 31;
#pragma unroll
    for (int j = 0; j < 4; ++j)
#pragma unroll
        for (int q = 0; q < 4; ++q) acc[j][q] = 0.0f;
#pragma unroll
    for (int k = 0; k < K; k += 16) {
        uint32_t a[4], b[2][4];
        ldsm4(a, &A[m0 + (lane & 15)][k + (lane >> 4) * 8]);
#pragma unroll
        for (int h = 0; h < 2; ++h) ldsm4t(b[h], &W[k + (lane & 7) + ((lane >> 3) & 1) * 8][n0 + 16 * h + (lane >> 4) * 8]);
#pragma unroll
        for (int j = 0; j < 4; ++j) {
            const uint32_t bj[2] = {b[j >> 1][2 * (j & 1)], b[j >> 1][2 * (j & 1) + 1]};
            mma_bf16(acc[j], a, bj);
        }
    }
}

// bias + GELU of an accumulator tile: z kept in acc, the activation to smem
__device__ __forceinline__ void rows_gelu(const float *__restrict__ bias, float (&acc)[4][4], __nv_bfloat16 (*out)[LDK],
                                          int m0, int n0) {
    const int lane = threadIdx.x & 31, grp = lane >> 2, tig = lane & 3;
#pragma unroll
    for (int j = 0; j < 4; ++j) {
        const int c = n0 + 8 * j + 2 * tig;
        const float b0 = __ldg(bias + c), b1 = __ldg(bias + c + 1);
#pragma unroll
        for (int h = 0; h < 2; ++h) {
            acc[j][2 * h] += b0;
            acc[j][2 * h + 1] += b1;
            *reinterpret_cast<uint32_t *>(&out[m0 + grp + 8 * h][c]) = pack_bf16(gelu_f(acc[j][2 * h]), gelu_f(acc[j][2 * h + 1]));
        }
    }
}

// gradient tile times GELU'(z): FP32 to global, BF16 operand to smem
__device__ __forceinline__ void rows_dgelu(const float (&z)[4][4], float (&acc)[4][4], __nv_bfloat16 (*out)[LDK],
                                           float *__restrict__ dz, int row0, int n, int m0, int n0) {
    const int lane = threadIdx.x & 31, grp = lane >> 2, tig = lane & 3;
#pragma unroll
    for (int j = 0; j < 4; ++j) {
        const int c = n0 + 8 * j + 2 * tig;
#pragma unroll
        for (int h = 0; h < 2; ++h) {
            const float v0 = acc[j][2 * h] * gelu_prime_f(z[j][2 * h]), v1 = acc[j][2 * h + 1] * gelu_prime_f(z[j][2 * h + 1]);
            const int r = m0 + grp + 8 * h;
            *reinterpret_cast<uint32_t *>(&out[r][c]) = pack_bf16(v0, v1);
            if (row0 + r < n) *reinterpret_cast<float2 *>(dz + (size_t)(row0 + r) * MLP_H + c) = make_float2(v0, v1);
        }
    }
}

// 16-byte copies of `rows` rows of `cols` BF16 values between global (row stride cols) and padded shared rows
template <int LD>
__device__ __forceinline__ void load_rows16(__nv_bfloat16 (*s)[LD], const __nv_bfloat16 *__restrict__ g, int rows, int cols) {
    const int per = cols / 8;
    for (int e = threadIdx.x; e < rows * per; e += blockDim.x)
        *reinterpret_cast<uint4 *>(&s[e / per][(e % per) * 8]) = __ldg(reinterpret_cast<const uint4 *>(g) + e);
}
template <int LD>
__device__ __forceinline__ void store_rows16(__nv_bfloat16 *__restrict__ g, const __nv_bfloat16 (*s)[LD], int rows, int cols) {
    const int per = cols / 8;
    for (int e = threadIdx.x; e < rows * per; e += blockDim.x)
        reinterpret_cast<uint4 *>(g)[e] = *reinterpret_cast<const uint4 *>(&s[e / per][(e % per) * 8]);
}

// TRAIN: forward, loss and backward of rows 32 b .. (b = blockIdx.x), raw
// inputs x and raw targets t.  Otherwise the outputs y, blocks striding over
// the row groups so that the weights are staged once per block.
template <bool TRAIN, int ROWS>
__global__ void __launch_bounds__(8 * ROWS) k_rows(MlpDev w, const float *__restrict__ x, const float *__restrict__ t,
                                                     int n, float *__restrict__ y, TrainOut o) {
    extern __shared__ __align__(16) unsigned char rows_raw[];
    static_assert(!TRAIN || ROWS == 32, "the loss is the sum of two warps");
    constexpr int NT = 8 * ROWS, MT = ROWS / 16;
    RowsSmem<ROWS> &S = *reinterpret_cast<RowsSmem<ROWS> *>(rows_raw);
    const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5, grp = lane >> 2, tig = lane & 3;
    const int m0 = 16 * (warp % MT), n0 = 32 * (warp / MT);
    load_rows16(S.w1, w.Wb + WB1, MLP_H, MLP_INP);
    load_rows16(S.w2, w.Wb + WB2, MLP_H, MLP_H);
    load_rows16(S.w3, w.Wb + WB3, MLP_H, MLP_H);
    load_rows16(S.w4, w.Wb + WB4, MLP_OUTP, MLP_H);
    for (int row0 = blockIdx.x * ROWS; row0 < n; row0 += gridDim.x * ROWS) {
        const int nrows = min(ROWS, n - row0);
        for (int e = tid; e < ROWS * MLP_INP; e += NT) {
            const int r = e / MLP_INP, c = e % MLP_INP;
            float v = 0.0f;
            if (r < nrows && c < MLP_IN) v = (x[(size_t)(row0 + r) * MLP_IN + c] - w.mean_x[c]) / w.std_x[c];
            S.x[r][c] = __float2bfloat16_rn(v);
        }
        if (TRAIN)
            for (int e = tid; e < ROWS * 16; e += NT) S.dy[e / 16][e % 16] = __float2bfloat16_rn(0.0f);
        __syncthreads();
        float z[3][4][4];
        rows_product(S.x, S.w1, MLP_INP, m0, n0, z[0]);
        rows_gelu(w.P + OFF_B1, z[0], S.a[0], m0, n0);
        __syncthreads();
        if (TRAIN) {
            store_rows16(o.x + (size_t)row0 * MLP_INP, S.x, nrows, MLP_INP);
            store_rows16(o.a[0] + (size_t)row0 * MLP_H, S.a[0], nrows, MLP_H);
        }
        rows_product(S.a[0], S.w2, MLP_H, m0, n0, z[1]);
        rows_gelu(w.P + OFF_B2, z[1], S.a[1], m0, n0);
        __syncthreads();
        if (TRAIN) store_rows16(o.a[1] + (size_t)row0 * MLP_H, S.a[1], nrows, MLP_H);
        rows_product(S.a[1], S.w3, MLP_H, m0, n0, z[2]);
        rows_gelu(w.P + OFF_B3, z[2], S.a[0], m0, n0);
        __syncthreads();
        if (TRAIN) store_rows16(o.a[2] + (size_t)row0 * MLP_H, S.a[0], nrows, MLP_H);
        double sq = 0.0;
        if (warp < MT) {  // the six outputs: one 16 x 8 tile per warp
            float acc[4] = {0.0f, 0.0f, 0.0f, 0.0f};
#pragma unroll
            for (int k = 0; k < MLP_H; k += 16) {
                uint32_t a[4], b[2];
                ldsm4(a, &S.a[0][m0 + (lane & 15)][k + (lane >> 4) * 8]);
                b[0] = ld_pair(&S.w4[grp][k + 2 * tig]);
                b[1] = ld_pair(&S.w4[grp][k + 8 + 2 * tig]);
                mma_bf16(acc, a, b);
            }
#pragma unroll
            for (int q = 0; q < 4; ++q) {
                const int r = m0 + grp + (q >= 2 ? 8 : 0), c = 2 * tig + (q & 1);
                if (c >= MLP_OUT || r >= nrows) continue;
                const float out = acc[q] + __ldg(w.P + OFF_B4 + c);
                const size_t at = (size_t)(row0 + r) * MLP_OUT + c;
                if (TRAIN) {
                    const float sc = 2.0f / (float)(n * MLP_OUT);  // dL/dy = 2 (y - t) / (6 n)
                    const float e = out - (t[at] - w.mean_y[c]) / w.std_y[c];
                    sq += (double)e * (double)e;
                    const float d = sc * e;
                    o.dy[at] = d;
                    S.dy[r][c] = __float2bfloat16_rn(d);
                } else {
                    y[at] = fmaf(out, w.std_y[c], w.mean_y[c]);
                }
            }
        }
        if constexpr (TRAIN) {
#pragma unroll
            for (int q = 16; q > 0; q >>= 1) sq += __shfl_xor_sync(0xffffffffu, sq, q);
            if (lane == 0) S.loss[warp] = sq;
            __syncthreads();
            if (tid == 0) o.loss[blockIdx.x] = S.loss[0] + S.loss[1];
            // backward: (dy W4), (dz W3), (dz W2), each times GELU' of the layer below
            float acc[4][4];
            {
                uint32_t a[4], b[4];
                ldsm4(a, &S.dy[m0 + (lane & 15)][(lane >> 4) * 8]);
                ldsm4t(b, &S.w4[lane & 7][n0 + (lane >> 3) * 8]);  // k 0..7; rows 8..15 are zero
#pragma unroll
                for (int j = 0; j < 4; ++j) {
                    const uint32_t bj[2] = {b[j], 0u};
#pragma unroll
                    for (int q = 0; q < 4; ++q) acc[j][q] = 0.0f;
                    mma_bf16(acc[j], a, bj);
                }
            }
            rows_dgelu(z[2], acc, S.a[1], o.dz[2], row0, n, m0, n0);
            __syncthreads();
            rows_product_t(S.a[1], S.w3, MLP_H, m0, n0, acc);
            rows_dgelu(z[1], acc, S.a[0], o.dz[1], row0, n, m0, n0);
            __syncthreads();
            rows_product_t(S.a[0], S.w2, MLP_H, m0, n0, acc);
            rows_dgelu(z[0], acc, S.a[1], o.dz[0], row0, n, m0, n0);
        }
        __syncthreads();  // the buffers are free for the next rows
    }
}

// Weight and bias gradients of the rows of slice blockIdx.y (KSLICE rows) into
// part[slice][MLP_NPARAM].  blockIdx.x < WG_TILES: one 64 x 64 tile of one
// layer's dz^T a, the whole slice of both operands staged once (ldmatrix
// transposes them), 16 k-steps in row order; otherwise 128 columns of the
// bias gradients, summed in row order.
constexpr int WG_THREADS = 128, WG_TILES = 12, WG_COLS = 4, WG_LD = 64 + 8;
struct WgradSmem {
    __nv_bfloat16 dz[KSLICE][WG_LD], a[KSLICE][WG_LD];
};

__global__ void __launch_bounds__(WG_THREADS) k_wgrad(TrainOut o, int n, float *__restrict__ part) {
    extern __shared__ __align__(16) unsigned char wg_raw[];
    WgradSmem &S = *reinterpret_cast<WgradSmem *>(wg_raw);
    const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5, grp = lane >> 2, tig = lane & 3;
    const int r0 = blockIdx.y * KSLICE, nr = min(KSLICE, n - r0);
    float *out = part + (size_t)blockIdx.y * MLP_NPARAM;
    if (blockIdx.x >= WG_TILES) {
        const int c = (blockIdx.x - WG_TILES) * WG_THREADS + tid;
        const int l = c / MLP_H;  // 0 .. 2: hidden layers, 3: the outputs
        if (l > 3 || (l == 3 && c - 3 * MLP_H >= MLP_OUT)) return;
        const int ld = l == 3 ? MLP_OUT : MLP_H, cc = c - l * MLP_H;
        const float *d = (l == 3 ? o.dy : l == 2 ? o.dz[2] : l == 1 ? o.dz[1] : o.dz[0]) + (size_t)r0 * ld + cc;
        float s = 0.0f;
#pragma unroll 32
        for (int r = 0; r < nr; ++r) s += __ldg(d + (size_t)r * ld);
        out[(l == 3 ? OFF_B4 : l == 2 ? OFF_B3 : l == 1 ? OFF_B2 : OFF_B1) + cc] = s;
        return;
    }
    // tiles: 0, 1 the first layer (128 x 34), 2..5 the second, 6..9 the third, 10, 11 the outputs (6 x 128)
    const int b = blockIdx.x, l = b < 2 ? 0 : b < 6 ? 1 : b < 10 ? 2 : 3;
    const int tm = l == 0 ? b : l == 3 ? 0 : ((b - 2) >> 1) & 1, tn = l == 0 ? 0 : b & 1;
    const int M = l == 3 ? MLP_OUT : MLP_H, N = l == 0 ? MLP_IN : MLP_H, lda = l == 0 ? MLP_INP : MLP_H;
    const float *dz = l == 3 ? o.dy : l == 2 ? o.dz[2] : l == 1 ? o.dz[1] : o.dz[0];
    const __nv_bfloat16 *act = l == 0 ? o.x : l == 1 ? o.a[0] : l == 2 ? o.a[1] : o.a[2];
    if (l == 3) {
        for (int e = tid; e < KSLICE * 8; e += WG_THREADS) {  // eight values per row of the 64: six outputs, then zeros
            const int r = e / 8, c = e % 8;
            const float v = r < nr && c < MLP_OUT ? __ldg(dz + (size_t)(r0 + r) * MLP_OUT + c) : 0.0f;
            S.dz[r][c] = __float2bfloat16_rn(v);
#pragma unroll
            for (int q = 1; q < 8; ++q) S.dz[r][8 * q + c] = __float2bfloat16_rn(0.0f);
        }
    } else {
#pragma unroll 8
        for (int e = tid; e < KSLICE * 16; e += WG_THREADS) {
            const int r = e / 16, c = (e % 16) * 4;
            float4 v = make_float4(0.0f, 0.0f, 0.0f, 0.0f);
            if (r < nr) v = __ldg(reinterpret_cast<const float4 *>(dz + (size_t)(r0 + r) * MLP_H + 64 * tm + c));
            *reinterpret_cast<uint2 *>(&S.dz[r][c]) = make_uint2(pack_bf16(v.x, v.y), pack_bf16(v.z, v.w));
        }
    }
    const int groups = l == 0 ? MLP_INP / 8 : 8;  // 16-byte groups of an activation row present in this tile
#pragma unroll 8
    for (int e = tid; e < KSLICE * 8; e += WG_THREADS) {
        const int r = e / 8, c = e % 8;
        uint4 v = make_uint4(0u, 0u, 0u, 0u);
        if (r < nr && c < groups) v = __ldg(reinterpret_cast<const uint4 *>(act + (size_t)(r0 + r) * lda + 64 * tn + 8 * c));
        *reinterpret_cast<uint4 *>(&S.a[r][8 * c]) = v;
    }
    __syncthreads();
    const int wm = 32 * (warp >> 1), wn = 32 * (warp & 1);
    float acc[2][4][4];
#pragma unroll
    for (int i = 0; i < 2; ++i)
#pragma unroll
        for (int j = 0; j < 4; ++j)
#pragma unroll
            for (int q = 0; q < 4; ++q) acc[i][j][q] = 0.0f;
    for (int k = 0; k < KSLICE; k += 16) {
        uint32_t a[2][4], bq[2][4];
#pragma unroll
        for (int i = 0; i < 2; ++i)
            ldsm4t(a[i], &S.dz[k + (lane & 7) + (lane >> 4) * 8][wm + 16 * i + ((lane >> 3) & 1) * 8]);
#pragma unroll
        for (int h = 0; h < 2; ++h)
            ldsm4t(bq[h], &S.a[k + (lane & 7) + ((lane >> 3) & 1) * 8][wn + 16 * h + (lane >> 4) * 8]);
#pragma unroll
        for (int i = 0; i < 2; ++i)
#pragma unroll
            for (int j = 0; j < 4; ++j) {
                const uint32_t bj[2] = {bq[j >> 1][2 * (j & 1)], bq[j >> 1][2 * (j & 1) + 1]};
                mma_bf16(acc[i][j], a[i], bj);
            }
    }
    out += l == 0 ? OFF_W1 : l == 1 ? OFF_W2 : l == 2 ? OFF_W3 : OFF_W4;
#pragma unroll
    for (int i = 0; i < 2; ++i)
#pragma unroll
        for (int j = 0; j < 4; ++j)
#pragma unroll
            for (int q = 0; q < 4; ++q) {
                const int m = 64 * tm + wm + 16 * i + grp + (q >= 2 ? 8 : 0), c = 64 * tn + wn + 8 * j + 2 * tig + (q & 1);
                if (m < M && c < N) out[(size_t)m * N + c] = acc[i][j][q];
            }
}

// The place of parameter i in the padded BF16 weights, or -1 for a bias.
__device__ __forceinline__ int wb_index(int i) {
    if (i < OFF_B1) return WB1 + (i / MLP_IN) * MLP_INP + i % MLP_IN;
    if (i >= OFF_W2 && i < OFF_B2) return WB2 + (i - OFF_W2);
    if (i >= OFF_W3 && i < OFF_B3) return WB3 + (i - OFF_W3);
    if (i >= OFF_W4 && i < OFF_B4) return WB4 + (i - OFF_W4);
    return -1;
}

// Gradient of every parameter as the slice sums in slice order, and (step)
// its AdamW update with the BF16 copy.  Block 0 also adds the blocks' losses (a
// lane every 32nd in order, then an xor tree): to *loss and, when given, to host-visible memory.
__global__ void __launch_bounds__(256) k_update(const float *__restrict__ part, int nsl, float *__restrict__ G, int step,
                                                float *__restrict__ P, float *__restrict__ Mm, float *__restrict__ Vv,
                                                __nv_bfloat16 *__restrict__ wb, float lr, float b1, float b2, float eps,
                                                float wd, float bc1, float bc2, const double *__restrict__ lpart,
                                                int nloss, int total, double *loss, double *host_loss) {
    const int i = blockIdx.x * blockDim.x + threadIdx.x;
    if (i < MLP_NPARAM) {
        float s = part[i];
#pragma unroll 16
        for (int z = 1; z < nsl; ++z) s += part[(size_t)z * MLP_NPARAM + i];
        G[i] = s;
        if (step) {
            float m = Mm[i], v = Vv[i];
            const float p = adamw_value(P[i], s, m, v, is_weight(i), lr, b1, b2, eps, wd, bc1, bc2);
            Mm[i] = m;
            Vv[i] = v;
            P[i] = p;
            const int at = wb_index(i);
            if (at >= 0) wb[at] = __float2bfloat16_rn(p);
        }
    }
    if (blockIdx.x == 0 && threadIdx.x < 32) {
        double s = 0.0;
        for (int k = threadIdx.x; k < nloss; k += 32) s += lpart[k];
#pragma unroll
        for (int q = 16; q > 0; q >>= 1) s += __shfl_xor_sync(0xffffffffu, s, q);
        if (threadIdx.x == 0) {
            s /= (double)total;
            *loss = s;
            if (host_loss) *host_loss = s;
        }
    }
}

// ---------------------------------------------------------------------------
// Inference of up to 16 samples per block (the predictor): features
// standardised, four layers with activations in shared memory, outputs
// de-standardised.  TC: BF16 tensor cores with the padded BF16 weights (the
// same operands and k order as k_rows, hence the same results); otherwise
// FP32 on the CUDA cores with the FP32 weights.
constexpr int INF_ROWS = 16, INF_THREADS = 128, ACT_LD = MLP_H + 8;

template <bool TC>
__device__ __forceinline__ void infer_layer(const MlpDev &w, int layer, const float (*actf)[ACT_LD],
                                            const __nv_bfloat16 (*actb)[ACT_LD], float (*outf)[ACT_LD],
                                            __nv_bfloat16 (*outb)[ACT_LD], int nrows) {
    const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
    const int K = layer == 0 ? MLP_IN : MLP_H;
    const int N = layer == 3 ? MLP_OUT : MLP_H;
    const float *bias = w.P + (layer == 0 ? OFF_B1 : layer == 1 ? OFF_B2 : layer == 2 ? OFF_B3 : OFF_B4);
    if constexpr (TC) {
        const __nv_bfloat16 *W = w.Wb + (layer == 0 ? WB1 : layer == 1 ? WB2 : layer == 2 ? WB3 : WB4);
        const int ldw = layer == 0 ? MLP_INP : MLP_H;
        const int Kp = layer == 0 ? MLP_INP : MLP_H;
        const int ntile = layer == 3 ? 1 : 4;  // n8 tiles per warp
        if (layer == 3 && warp > 0) return;
        const int grp = lane >> 2, tig = lane & 3;
        float acc[4][4];
#pragma unroll
        for (int j = 0; j < 4; ++j)
#pragma unroll
            for (int q = 0; q < 4; ++q) acc[j][q] = 0.0f;
        for (int kk = 0; kk < Kp; kk += 16) {
            uint32_t a[4];
            a[0] = ld_pair(&actb[grp][kk + 2 * tig]);
            a[1] = ld_pair(&actb[grp + 8][kk + 2 * tig]);
            a[2] = ld_pair(&actb[grp][kk + 8 + 2 * tig]);
            a[3] = ld_pair(&actb[grp + 8][kk + 8 + 2 * tig]);
#pragma unroll
            for (int j = 0; j < 4; ++j) {
                if (j >= ntile) break;
                const int c = 32 * warp + 8 * j + grp;
                uint32_t b[2];
                b[0] = ld_pair(W + (size_t)c * ldw + kk + 2 * tig);
                b[1] = ld_pair(W + (size_t)c * ldw + kk + 8 + 2 * tig);
                mma_bf16(acc[j], a, b);
            }
        }
#pragma unroll
        for (int j = 0; j < 4; ++j) {
            if (j >= ntile) break;
            const int c = 32 * warp + 8 * j + 2 * tig;
#pragma unroll
            for (int q = 0; q < 4; ++q) {
                const int r = grp + (q >= 2 ? 8 : 0), cc = c + (q & 1);
                if (cc < N) {
                    const float z = acc[j][q] + bias[cc];
                    const float v = layer == 3 ? z : gelu_f(z);
                    outf[r][cc] = v;
                    outb[r][cc] = __float2bfloat16_rn(v);
                }
            }
        }
    } else {
        const float *W = w.P + (layer == 0 ? OFF_W1 : layer == 1 ? OFF_W2 : layer == 2 ? OFF_W3 : OFF_W4);
        for (int e = tid; e < INF_ROWS * N; e += INF_THREADS) {
            const int r = e / N, c = e % N;
            float s = 0.0f;
            for (int k = 0; k < K; ++k) s = fmaf(actf[r][k], W[(size_t)c * K + k], s);
            const float z = s + bias[c];
            const float v = layer == 3 ? z : gelu_f(z);
            outf[r][c] = v;
            outb[r][c] = __float2bfloat16_rn(v);
        }
    }
    (void)nrows;
}

struct InferSmem {
    float af[2][INF_ROWS][ACT_LD];
    __align__(16) __nv_bfloat16 ab[2][INF_ROWS][ACT_LD];
};

template <bool TC>
__device__ __forceinline__ void mlp_infer_rows(const MlpDev &w, const float *__restrict__ x, int n, int row0,
                                               float *__restrict__ y, InferSmem &sm) {
    float (*af)[INF_ROWS][ACT_LD] = sm.af;
    __nv_bfloat16 (*ab)[INF_ROWS][ACT_LD] = sm.ab;
    const int tid = threadIdx.x;
    const int nrows = min(INF_ROWS, n - row0);
    for (int e = tid; e < INF_ROWS * ACT_LD; e += INF_THREADS) {
        const int r = e / ACT_LD, c = e % ACT_LD;
        float v = 0.0f;
        if (r < nrows && c < MLP_IN) v = (x[(size_t)(row0 + r) * MLP_IN + c] - w.mean_x[c]) / w.std_x[c];
        af[0][r][c] = v;
        ab[0][r][c] = __float2bfloat16_rn(v);
        af[1][r][c] = 0.0f;
        ab[1][r][c] = __float2bfloat16_rn(0.0f);
    }
    __syncthreads();
    for (int l = 0; l < 4; ++l) {
        const int s = l & 1;
        infer_layer<TC>(w, l, af[s], ab[s], af[s ^ 1], ab[s ^ 1], nrows);
        __syncthreads();
    }
    for (int e = tid; e < nrows * MLP_OUT; e += INF_THREADS) {
        const int r = e / MLP_OUT, c = e % MLP_OUT;
        y[(size_t)(row0 + r) * MLP_OUT + c] = fmaf(af[0][r][c], w.std_y[c], w.mean_y[c]);
    }
}

__global__ void __launch_bounds__(INF_THREADS) k_mlp_infer(MlpDev w, const float *__restrict__ x, int n,
                                                           float *__restrict__ y) {
    __shared__ InferSmem sm;
    mlp_infer_rows<false>(w, x, n, blockIdx.x * INF_ROWS, y, sm);
}

// ---------------------------------------------------------------------------
// Features of the predictor at time level t (all in the body frame of t,
// whose axes are the rows d_0, d_1, d_2 of the orientation matrix M):
//   [0:4]   unit quaternion (w, x, y, z), w >= 0, of M, by Shepperd's method
//           (S. W. Shepperd, J. Guidance and Control 1 (1978) 223): the
//           largest of 1 + tr M, 1 + 2 M_ii - tr M picks the stable formula
//   [4:7]   M v(t - 1/2)          [7:10]  M w(t - 1/2)
//   [10:34] M F(t - h) / sF, M T(t - h) / sT for h = 0, 1, 2, 3, with the
//           scales sF = max_h |F(t - h)|, sT = max_h |T(t - h)| (1 if zero)
// Targets: the departure of the next force and torque from their linear
// extrapolation, in the same frame and scale:
//   M (F(t+1) - 2 F(t) + F(t-1)) / sF,  M (T(t+1) - 2 T(t) + T(t-1)) / sT,
// so the prediction is F^ = 2 F(t) - F(t-1) + sF M^T y (and T^ alike): the
// network corrects linear extrapolation, independent of the force's size.
__device__ void quat_of(const double *M, double q[4]) {
    const double tr = M[0] + M[4] + M[8];
    const double c[4] = {1.0 + tr, 1.0 + 2.0 * M[0] - tr, 1.0 + 2.0 * M[4] - tr, 1.0 + 2.0 * M[8] - tr};
    int b = 0;
    for (int i = 1; i < 4; ++i)
        if (c[i] > c[b]) b = i;
    const double s = 2.0 * sqrt(c[b]);  // = 4 |q_b|
    const double r = 1.0 / s;
    if (b == 0) {
        q[0] = 0.25 * s; q[1] = (M[7] - M[5]) * r; q[2] = (M[2] - M[6]) * r; q[3] = (M[3] - M[1]) * r;
    } else if (b == 1) {
        q[0] = (M[7] - M[5]) * r; q[1] = 0.25 * s; q[2] = (M[1] + M[3]) * r; q[3] = (M[2] + M[6]) * r;
    } else if (b == 2) {
        q[0] = (M[2] - M[6]) * r; q[1] = (M[1] + M[3]) * r; q[2] = 0.25 * s; q[3] = (M[5] + M[7]) * r;
    } else {
        q[0] = (M[3] - M[1]) * r; q[1] = (M[2] + M[6]) * r; q[2] = (M[5] + M[7]) * r; q[3] = 0.25 * s;
    }
    if (q[0] < 0.0)
        for (int i = 0; i < 4; ++i) q[i] = -q[i];
}

__device__ __forceinline__ void to_body(const double *M, const double *a, double scale, float *out) {
    for (int i = 0; i < 3; ++i) out[i] = (float)((M[3 * i] * a[0] + M[3 * i + 1] * a[1] + M[3 * i + 2] * a[2]) / scale);
}

__device__ void scales_of(const double (*Fh)[3], const double (*Th)[3], double &sF, double &sT) {
    sF = 0.0;
    sT = 0.0;
    for (int h = 0; h < 4; ++h) {
        sF = fmax(sF, sqrt(Fh[h][0] * Fh[h][0] + Fh[h][1] * Fh[h][1] + Fh[h][2] * Fh[h][2]));
        sT = fmax(sT, sqrt(Th[h][0] * Th[h][0] + Th[h][1] * Th[h][1] + Th[h][2] * Th[h][2]));
    }
    if (!(sF > 0.0)) sF = 1.0;
    if (!(sT > 0.0)) sT = 1.0;
}

__device__ void features_of(const double *M, const double *v, const double *w, const double (*Fh)[3],
                            const double (*Th)[3], float *x) {
    double q[4], sF, sT;
    quat_of(M, q);
    scales_of(Fh, Th, sF, sT);
    for (int i = 0; i < 4; ++i) x[i] = (float)q[i];
    to_body(M, v, 1.0, x + 4);
    to_body(M, w, 1.0, x + 7);
    for (int h = 0; h < 4; ++h) {
        to_body(M, Fh[h], sF, x + 10 + 6 * h);
        to_body(M, Th[h], sT, x + 13 + 6 * h);
    }
}

// Prediction of F(t+1), T(t+1) at the start of the step t -> t+1 (slot =
// the window slot of t).  Linear extrapolation 2 F(t) - F(t-1) in mode 1, and
// in mode 2 while fewer than four history levels exist or while the
// network's own previous prediction missed by more than the threshold (the
// fallback); the network, in mode 2, runs whenever four levels exist, so its
// accuracy keeps being checked while it is not used.
__device__ void predict_block(const MlpDev &w, bool has_net, DevState *st, int slot, int mode, InferSmem &sm) {
    __shared__ int run_net;
    Predictor &P = st->pr;
    if (threadIdx.x == 0) {
        for (int q = 0; q < 3; ++q) {
            P.Fhat[q] = P.hist_n >= 2 ? 2.0 * P.Fh[0][q] - P.Fh[1][q] : P.Fh[0][q];
            P.That[q] = P.hist_n >= 2 ? 2.0 * P.Th[0][q] - P.Th[1][q] : P.Th[0][q];
        }
        P.predicted = 1;
        P.by_net = 0;
        P.steps += 1;
        run_net = mode == 2 && has_net && P.hist_n >= 4;
        if (run_net) {
            const BodySlot &S = st->s[slot];
            features_of(S.d, S.v, S.w, P.Fh, P.Th, P.feat);
        } else if (mode == 2) {
            P.fallbacks += 1;
        }
    }
    __syncthreads();
    if (!run_net) return;
    if (w.precision == 0) mlp_infer_rows<true>(w, P.feat, 1, 0, P.yb, sm);
    else mlp_infer_rows<false>(w, P.feat, 1, 0, P.yb, sm);
    __syncthreads();
    if (threadIdx.x == 0) {
        const double *M = st->s[slot].d;
        double sF, sT;
        scales_of(P.Fh, P.Th, sF, sT);
        for (int i = 0; i < 3; ++i) {  // linear extrapolation + scale * M^T y
            P.Fnet[i] = 2.0 * P.Fh[0][i] - P.Fh[1][i] + sF * (M[i] * P.yb[0] + M[3 + i] * P.yb[1] + M[6 + i] * P.yb[2]);
            P.Tnet[i] = 2.0 * P.Th[0][i] - P.Th[1][i] + sT * (M[i] * P.yb[3] + M[3 + i] * P.yb[4] + M[6 + i] * P.yb[5]);
        }
        P.net_ok = 1;
        if (!P.fallback) {
            for (int i = 0; i < 3; ++i) {
                P.Fhat[i] = P.Fnet[i];
                P.That[i] = P.Tnet[i];
            }
            P.by_net = 1;
            P.mlp_steps += 1;
        } else {
            P.fallbacks += 1;
        }
    }
}

__global__ void __launch_bounds__(INF_THREADS) k_predict(MlpDev w, int has_net, DevState *st, int slot, int mode) {
    __shared__ InferSmem sm;
    predict_block(w, has_net != 0, st, slot, mode, sm);
}

__global__ void __launch_bounds__(INF_THREADS) k_batch_predict(const RunDesc *__restrict__ runs, int slot) {
    __shared__ InferSmem sm;
    const RunDesc &R = runs[blockIdx.x];
    if (R.bc.predictor == 0) return;
    predict_block(R.mlp, R.mlp.P != nullptr, R.st, slot, R.bc.predictor, sm);
}

cudaError_t launch_predict(const MlpDev *w, DevState *st, int slot, int mode, cudaStream_t s) {
    MlpDev v;
    memset(&v, 0, sizeof v);
    if (w) v = *w;
    k_predict<<<1, INF_THREADS, 0, s>>>(v, w != nullptr, st, slot, mode);
    return cudaGetLastError();
}

cudaError_t launch_batch_predict(const RunDesc *runs, int nruns, int slot, cudaStream_t s) {
    k_batch_predict<<<nruns, INF_THREADS, 0, s>>>(runs, slot);
    return cudaGetLastError();
}

// Training pairs from a trajectory log of consecutive time levels (records
// as written by the force reduction): sample j uses records j .. j + 4
// (history t - 3 .. t with t = j + 3, target t + 1).  Records whose time
// levels are not consecutive give NaN features (and count in *bad).
__global__ void k_build_samples(const double *__restrict__ log, long long nsamp, float *__restrict__ x,
                                float *__restrict__ y, int *bad) {
    const long long j = (long long)blockIdx.x * blockDim.x + threadIdx.x;
    if (j >= nsamp) return;
    const double *r[5];
    for (int h = 0; h < 5; ++h) r[h] = log + (size_t)(j + h) * LOG_REC;  // r[3] = t, r[4] = t + 1
    bool ok = true;
    for (int h = 1; h < 5; ++h) ok = ok && r[h][21] == r[h - 1][21] + 1.0;
    double Fh[4][3], Th[4][3];
    for (int h = 0; h < 4; ++h)
        for (int q = 0; q < 3; ++q) {
            Fh[h][q] = r[3 - h][15 + q];
            Th[h][q] = r[3 - h][18 + q];
        }
    float *xo = x + (size_t)j * MLP_IN;
    features_of(r[3], r[3] + 9, r[3] + 12, Fh, Th, xo);
    double sF, sT, dF[3], dT[3];
    scales_of(Fh, Th, sF, sT);
    for (int q = 0; q < 3; ++q) {  // departure of t + 1 from the linear extrapolation
        dF[q] = r[4][15 + q] - 2.0 * Fh[0][q] + Fh[1][q];
        dT[q] = r[4][18 + q] - 2.0 * Th[0][q] + Th[1][q];
    }
    to_body(r[3], dF, sF, y + (size_t)j * MLP_OUT);
    to_body(r[3], dT, sT, y + (size_t)j * MLP_OUT + 3);
    if (!ok) {
        for (int i = 0; i < MLP_IN; ++i) xo[i] = NAN;
        atomicAdd(bad, 1);
    }
}

// BF16 outputs of n rows, blocks striding over the row groups: 32 rows per block
// and two blocks per SM, or 128 rows in a block of 1024 threads per SM, which holds
// twice the rows and does in one round what takes the narrow blocks two: us with
// narrow / wide blocks, 9728 rows (one round) 14.4 / 18.5, 12000 20.5 / 18.5, 15967
// 22.5 / 18.5, 29184 (three) 30.4 / 32.8, 38912 (four) 37.1 / 32.8, 48640 (five) 45.1 /
// 47.2, 58368 (six) 52.9 / 47.1, 68096 (seven) 60.1 / 61.5, 77824 (eight) 67.8 / 61.5,
// 87552 (nine) 75.5 / 75.3, 97280 (ten) 82.7 / 75.4.  Bound by latency and
// the GELU (384 erff a row), not by the products (1.2 GFLOP at 15967 rows).
static cudaError_t launch_rows(const MlpDev &w, const float *x, int n, float *y, cudaStream_t s) {
    const int rounds = (n + 304 * RT_ROWS - 1) / (304 * RT_ROWS);  // of narrow blocks
    if (rounds % 2 == 0 || rounds > 8) {
        const int groups = (n + RT_WIDE - 1) / RT_WIDE;
        k_rows<false, RT_WIDE><<<groups < 152 ? groups : 152, 8 * RT_WIDE, sizeof(RowsSmem<RT_WIDE>), s>>>(w, x, nullptr, n, y,
                                                                                                   TrainOut{});
        return cudaGetLastError();
    }
    const int groups = (n + RT_ROWS - 1) / RT_ROWS;
    k_rows<false, RT_ROWS><<<groups < 304 ? groups : 304, RT_THREADS, sizeof(RowsSmem<RT_ROWS>), s>>>(w, x, nullptr, n, y,
                                                                                                TrainOut{});
    return cudaGetLastError();
}

cudaError_t launch_mlp_infer(const MlpDev &w, const float *x, int n, float *y, cudaStream_t s) {
    if (n <= 0) return cudaSuccess;
    const int nb = (n + INF_ROWS - 1) / INF_ROWS;
    if (w.precision == 0) return launch_rows(w, x, n, y, s);
    k_mlp_infer<<<nb, INF_THREADS, 0, s>>>(w, x, n, y);
    return cudaGetLastError();
}

}  // namespace turret

// ===========================================================================
// Host object behind turret_mlp.
struct turret_mlp {
    int cap, precision;
    cudaStream_t stream;
    MlpDev dev;
    float *P, *G, *Mm, *Vv;
    __nv_bfloat16 *Wb;
    float *norm;  // mean_x [34], std_x [34], mean_y [6], std_y [6]
    float *X0, *T, *Y, *dY, *Z[3], *A[3], *D[2];
    float *part;  // split-K partial sums [MAX_SLICES][128][128]
    double *loss;
    double *host_loss;  // page-locked copy written by the update kernel, or null (the loss is then copied)
    long long adam_step;
    // the FP32 training step (standardise, forward, backward, AdamW, BF16 copy) as
    // one CUDA graph per batch size; between replays only the input pointers
    // and the optimiser's scalars change, in the three nodes that take them
    cudaGraph_t train_graph;  // kept: its nodes address the instantiated graph's nodes
    cudaGraphExec_t train_exec;
    int train_n;
    cudaGraphNode_t node_x, node_y, node_adam;
    std::string err;
};

namespace {
std::string g_mlp_err;

struct MCarver {
    char *base;
    size_t off;
    void *take(size_t bytes) {
        off = (off + 255) & ~(size_t)255;
        void *p = base ? base + off : nullptr;
        off += bytes;
        return p;
    }
};

void carve_mlp(MCarver &cv, int cap, turret_mlp *m) {
    turret_mlp t;
    turret_mlp &M = m ? *m : t;
    M.P = (float *)cv.take(MLP_NPARAM * 4);
    M.G = (float *)cv.take(MLP_NPARAM * 4);
    M.Mm = (float *)cv.take(MLP_NPARAM * 4);
    M.Vv = (float *)cv.take(MLP_NPARAM * 4);
    M.Wb = (__nv_bfloat16 *)cv.take(WB_END * 2);
    M.norm = (float *)cv.take(2 * (MLP_IN + MLP_OUT) * 4);
    const size_t c = (size_t)cap;
    M.X0 = (float *)cv.take(c * MLP_IN * 4);
    M.T = (float *)cv.take(c * MLP_OUT * 4);
    M.Y = (float *)cv.take(c * MLP_OUT * 4);
    M.dY = (float *)cv.take(c * MLP_OUT * 4);
    for (int l = 0; l < 3; ++l) {
        M.Z[l] = (float *)cv.take(c * MLP_H * 4);
        M.A[l] = (float *)cv.take(c * MLP_H * 4);
    }
    for (int l = 0; l < 2; ++l) M.D[l] = (float *)cv.take(c * MLP_H * 4);
    M.loss = (double *)cv.take(8);
    M.part = (float *)cv.take((size_t)MAX_SLICES * MLP_H * MLP_H * 4);
}
// a batch of more slices than part holds has them in D: 1 KB a row against 598 B a row and one slice
static_assert((size_t)MAX_SLICES * MLP_H * MLP_H / MLP_NPARAM * KSLICE * (2 * MLP_H * 4 - MLP_NPARAM * 4 / KSLICE - 1) >=
                  (size_t)MLP_NPARAM * 4, "D holds the partial gradients of large batches");

turret_status mfail(turret_mlp *m, turret_status s, const std::string &msg) {
    if (m) m->err = msg; else g_mlp_err = msg;
    if (s == TURRET_ECUDA) cudaGetLastError();  // a non-sticky error must not surface in later launches
    return s;
}

#define MK(call, where)                                                                                       \
    do {                                                                                                      \
        cudaError_t e_ = (call);                                                                              \
        if (e_ != cudaSuccess) return mfail(m, TURRET_ECUDA, std::string(where) + ": " + cudaGetErrorString(e_)); \
    } while (0)

cudaError_t gemm(const turret_mlp *m, const GemmArgs &g, int epi) {
    const dim3 grid((g.M + GBM - 1) / GBM, (g.N + GBN - 1) / GBN,
                    g.kslice > 0 ? (g.K + g.kslice - 1) / g.kslice : 1);
    k_gemm<<<grid, GTHREADS, 0, m->stream>>>(g, epi);
    return cudaGetLastError();
}

GemmArgs gargs(const float *A, int lda, int ta, const float *B, int ldb, int tb, float *C, int ldc, int M, int N,
               int K) {
    GemmArgs g;
    memset(&g, 0, sizeof g);
    g.A = A; g.lda = lda; g.ta = ta;
    g.B = B; g.ldb = ldb; g.tb = tb;
    g.C = C; g.ldc = ldc;
    g.M = M; g.N = N; g.K = K;
    return g;
}

// The FP32 check mode: forward pass of n standardised rows in X0 -> Y (keeps Z, A for backprop).
cudaError_t forward(turret_mlp *m, int n) {
    const float *W[4] = {m->P + OFF_W1, m->P + OFF_W2, m->P + OFF_W3, m->P + OFF_W4};
    const float *b[4] = {m->P + OFF_B1, m->P + OFF_B2, m->P + OFF_B3, m->P + OFF_B4};
    const float *in = m->X0;
    int K = MLP_IN;
    for (int l = 0; l < 3; ++l) {
        GemmArgs g = gargs(in, K, 0, W[l], K, 0, m->Z[l], MLP_H, n, MLP_H, K);
        g.bias = b[l];
        g.Aout = m->A[l];
        g.ldo = MLP_H;
        cudaError_t e = gemm(m, g, EPI_GELU);
        if (e != cudaSuccess) return e;
        in = m->A[l];
        K = MLP_H;
    }
    GemmArgs g = gargs(in, MLP_H, 0, W[3], MLP_H, 0, m->Y, MLP_OUT, n, MLP_OUT, MLP_H);
    g.bias = b[3];
    return gemm(m, g, EPI_STORE);
}

// Loss of the standardised targets in T and the gradient into G.
cudaError_t backward(turret_mlp *m, int n) {
    cudaError_t e;
    k_loss<<<1, LOSS_THREADS, 0, m->stream>>>(m->Y, m->T, n, m->dY, m->loss);
    if ((e = cudaGetLastError()) != cudaSuccess) return e;
    const int offW[4] = {OFF_W1, OFF_W2, OFF_W3, OFF_W4}, offB[4] = {OFF_B1, OFF_B2, OFF_B3, OFF_B4};
    const int kin[4] = {MLP_IN, MLP_H, MLP_H, MLP_H};
    const float *acts[4] = {m->X0, m->A[0], m->A[1], m->A[2]};
    const float *dz = m->dY;  // gradient of the current layer's output
    int nout = MLP_OUT;
    for (int l = 3; l >= 0; --l) {
        // dW_l = dz^T a_{l-1} ([nout][kin]), db_l = column sums of dz; both
        // reduce over the batch: KSLICE-row slices, partial sums added in order
        const int nsl = (n + KSLICE - 1) / KSLICE;
        GemmArgs g = gargs(dz, nout, 1, acts[l], kin[l], 1, m->G + offW[l], kin[l], nout, kin[l], n);
        g.kslice = KSLICE;
        g.part = m->part;
        if ((e = gemm(m, g, EPI_STORE)) != cudaSuccess) return e;
        k_sum_slices<<<(nout * kin[l] + 255) / 256, 256, 0, m->stream>>>(m->part, nsl, nout * kin[l], m->G + offW[l]);
        if ((e = cudaGetLastError()) != cudaSuccess) return e;
        k_colsum<<<dim3((nout + 127) / 128, nsl), 128, 0, m->stream>>>(dz, n, nout, nout, m->part);
        if ((e = cudaGetLastError()) != cudaSuccess) return e;
        k_sum_slices<<<(nout + 255) / 256, 256, 0, m->stream>>>(m->part, nsl, nout, m->G + offB[l]);
        if ((e = cudaGetLastError()) != cudaSuccess) return e;
        if (l == 0) break;
        // dz_{l-1} = (dz W_l) * gelu'(z_{l-1})
        float *dst = m->D[l & 1];
        GemmArgs h = gargs(dz, nout, 0, m->P + offW[l], kin[l], 1, dst, MLP_H, n, MLP_H, nout);
        h.Zg = m->Z[l - 1];
        h.ldz = MLP_H;
        if ((e = gemm(m, h, EPI_DGELU)) != cudaSuccess) return e;
        dz = dst;
        nout = MLP_H;
    }
    return cudaSuccess;
}

cudaError_t prepare(turret_mlp *m, const float *x, const float *y, int n) {
    k_standardise<<<(n * MLP_IN + 255) / 256, 256, 0, m->stream>>>(x, n, MLP_IN, m->norm, m->norm + MLP_IN, m->X0);
    cudaError_t e = cudaGetLastError();
    if (e != cudaSuccess || !y) return e;
    k_standardise<<<(n * MLP_OUT + 255) / 256, 256, 0, m->stream>>>(y, n, MLP_OUT, m->norm + 2 * MLP_IN,
                                                                    m->norm + 2 * MLP_IN + MLP_OUT, m->T);
    return cudaGetLastError();
}

// Gradients (and, with opt, one AdamW step) of raw rows x, targets y in BF16:
// forward and backward by rows, weight gradients by slices, update.  The
// buffers of the FP32 mode hold this mode's operands: X0, A the BF16 inputs
// and activations, Z the layer gradients, T the losses per block; the slices'
// partial gradients go to part, or to D where it is the larger (batches of
// more than 27 slices).
cudaError_t train_bf16(turret_mlp *m, const float *x, const float *y, int n, const turret_adamw *opt, float bc1,
                       float bc2) {
    const int groups = (n + RT_ROWS - 1) / RT_ROWS, nsl = (n + KSLICE - 1) / KSLICE;
    TrainOut o;
    o.x = (__nv_bfloat16 *)m->X0;
    for (int l = 0; l < 3; ++l) {
        o.a[l] = (__nv_bfloat16 *)m->A[l];
        o.dz[l] = m->Z[l];
    }
    o.dy = m->dY;
    o.loss = (double *)m->T;
    const size_t need = (size_t)nsl * MLP_NPARAM, have = (size_t)MAX_SLICES * MLP_H * MLP_H;
    float *part = need <= have ? m->part : m->D[0];
    k_rows<true, RT_ROWS><<<groups, RT_THREADS, sizeof(RowsSmem<RT_ROWS>), m->stream>>>(m->dev, x, y, n, nullptr, o);
    k_wgrad<<<dim3(WG_TILES + WG_COLS, nsl), WG_THREADS, sizeof(WgradSmem), m->stream>>>(o, n, part);
    const turret_adamw a = opt ? *opt : turret_adamw{0.0f, 0.0f, 0.0f, 1.0f, 0.0f};
    k_update<<<(MLP_NPARAM + 255) / 256, 256, 0, m->stream>>>(part, nsl, m->G, opt != nullptr, m->P, m->Mm, m->Vv, m->Wb,
                                                              a.lr, a.beta1, a.beta2, a.eps, a.weight_decay, bc1, bc2,
                                                              o.loss, groups, n * MLP_OUT, m->loss, m->host_loss);
    return cudaGetLastError();
}

// The loss of the last pass (waits for the stream).
cudaError_t read_loss(turret_mlp *m, float *loss) {
    double L = 0.0;
    cudaError_t e = cudaSuccess;
    const bool mapped = m->precision == 0 && m->host_loss;
    if (!mapped) e = cudaMemcpyAsync(&L, m->loss, 8, cudaMemcpyDeviceToHost, m->stream);
    if (e == cudaSuccess) e = cudaStreamSynchronize(m->stream);
    if (e == cudaSuccess) *loss = (float)(mapped ? *static_cast<volatile double *>(m->host_loss) : L);
    return e;
}

cudaError_t refresh(turret_mlp *m) {
    k_refresh_bf16<<<(WB_END + 255) / 256, 256, 0, m->stream>>>(m->P, m->Wb);
    return cudaGetLastError();
}

}  // namespace

extern "C" size_t mlp_workspace_bytes(int32_t batch_cap) {
    if (batch_cap < 1 || batch_cap > MAX_SLICES * KSLICE) return 0;
    MCarver cv{nullptr, 0};
    carve_mlp(cv, batch_cap, nullptr);
    return cv.off + 256;
}

extern "C" turret_status mlp_init(turret_mlp **out, int32_t batch_cap, int32_t precision, const float *params,
                                  void *ws, size_t ws_bytes, void *stream) {
    turret_mlp *m = nullptr;
    if (!out) return mfail(m, TURRET_EINVAL, "out is NULL");
    *out = nullptr;
    if (precision < 0 || precision > 1) return mfail(m, TURRET_EINVAL, "precision must be 0 (bf16) or 1 (fp32)");
    const size_t need = mlp_workspace_bytes(batch_cap);
    if (need == 0) return mfail(m, TURRET_EINVAL, "invalid batch capacity");
    if (!params) return mfail(m, TURRET_EINVAL, "NULL parameters");
    if (!ws || ws_bytes < need) return mfail(m, TURRET_ENOMEM, "mlp workspace too small");
    if (((uintptr_t)ws & 255) != 0) return mfail(m, TURRET_EINVAL, "workspace must be 256-byte aligned");
    m = new turret_mlp();
    m->cap = batch_cap;
    m->precision = precision;
    m->stream = (cudaStream_t)stream;
    m->adam_step = 0;
    m->train_exec = nullptr;
    m->train_graph = nullptr;
    m->train_n = 0;
    m->host_loss = nullptr;
    MCarver cv{(char *)ws, 0};
    carve_mlp(cv, batch_cap, m);
    std::vector<float> norm(2 * (MLP_IN + MLP_OUT));
    for (int i = 0; i < MLP_IN; ++i) norm[MLP_IN + i] = 1.0f;                 // std_x
    for (int i = 0; i < MLP_OUT; ++i) norm[2 * MLP_IN + MLP_OUT + i] = 1.0f;  // std_y
    cudaError_t e = cudaMemcpyAsync(m->P, params, MLP_NPARAM * 4, cudaMemcpyHostToDevice, m->stream);
    if (e == cudaSuccess) e = cudaMemsetAsync(m->Mm, 0, MLP_NPARAM * 4, m->stream);
    if (e == cudaSuccess) e = cudaMemsetAsync(m->Vv, 0, MLP_NPARAM * 4, m->stream);
    if (e == cudaSuccess) e = cudaMemcpyAsync(m->norm, norm.data(), norm.size() * 4, cudaMemcpyHostToDevice, m->stream);
    if (e == cudaSuccess) e = refresh(m);
    if (e == cudaSuccess && precision == 0) {
        const auto smem = cudaFuncAttributeMaxDynamicSharedMemorySize;
        e = cudaFuncSetAttribute(k_rows<true, RT_ROWS>, smem, (int)sizeof(RowsSmem<RT_ROWS>));
        if (e == cudaSuccess) e = cudaFuncSetAttribute(k_rows<false, RT_ROWS>, smem, (int)sizeof(RowsSmem<RT_ROWS>));
        if (e == cudaSuccess) e = cudaFuncSetAttribute(k_rows<false, RT_WIDE>, smem, (int)sizeof(RowsSmem<RT_WIDE>));
        if (e == cudaSuccess)
            e = cudaFuncSetAttribute(k_wgrad, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)sizeof(WgradSmem));
        if (cudaHostAlloc((void **)&m->host_loss, sizeof(double), cudaHostAllocDefault) != cudaSuccess) {
            m->host_loss = nullptr;  // the loss is then copied from the device
            cudaGetLastError();
        }
    }
    if (e == cudaSuccess) e = cudaStreamSynchronize(m->stream);
    if (e != cudaSuccess) {
        if (m->host_loss) cudaFreeHost(m->host_loss);
        delete m;
        return mfail(nullptr, TURRET_ECUDA, std::string("mlp_init: ") + cudaGetErrorString(e));
    }
    m->dev.P = m->P;
    m->dev.Wb = m->Wb;
    m->dev.mean_x = m->norm;
    m->dev.std_x = m->norm + MLP_IN;
    m->dev.mean_y = m->norm + 2 * MLP_IN;
    m->dev.std_y = m->norm + 2 * MLP_IN + MLP_OUT;
    m->dev.precision = precision;
    *out = m;
    return TURRET_OK;
}

extern "C" turret_status mlp_set_params(turret_mlp *m, const float *params) {
    if (!m || !params) return mfail(m, TURRET_EINVAL, "NULL argument");
    MK(cudaMemcpyAsync(m->P, params, MLP_NPARAM * 4, cudaMemcpyHostToDevice, m->stream), "set params");
    MK(refresh(m), "refresh bf16");
    MK(cudaStreamSynchronize(m->stream), "set params sync");
    return TURRET_OK;
}

extern "C" turret_status mlp_get_params(turret_mlp *m, float *params) {
    if (!m || !params) return mfail(m, TURRET_EINVAL, "NULL argument");
    MK(cudaMemcpyAsync(params, m->P, MLP_NPARAM * 4, cudaMemcpyDeviceToHost, m->stream), "get params");
    MK(cudaStreamSynchronize(m->stream), "get params sync");
    return TURRET_OK;
}

extern "C" turret_status mlp_set_norm(turret_mlp *m, const float *mean_x, const float *std_x, const float *mean_y,
                                      const float *std_y) {
    if (!m || !mean_x || !std_x || !mean_y || !std_y) return mfail(m, TURRET_EINVAL, "NULL argument");
    std::vector<float> h(2 * (MLP_IN + MLP_OUT));
    for (int i = 0; i < MLP_IN; ++i) {
        if (!(std_x[i] > 0.0f)) return mfail(m, TURRET_EINVAL, "non-positive std");
        h[i] = mean_x[i];
        h[MLP_IN + i] = std_x[i];
    }
    for (int i = 0; i < MLP_OUT; ++i) {
        if (!(std_y[i] > 0.0f)) return mfail(m, TURRET_EINVAL, "non-positive std");
        h[2 * MLP_IN + i] = mean_y[i];
        h[2 * MLP_IN + MLP_OUT + i] = std_y[i];
    }
    MK(cudaMemcpyAsync(m->norm, h.data(), h.size() * 4, cudaMemcpyHostToDevice, m->stream), "set norm");
    MK(cudaStreamSynchronize(m->stream), "set norm sync");
    return TURRET_OK;
}

extern "C" turret_status mlp_forward(turret_mlp *m, const float *x, int32_t n, float *y) {
    if (!m || !x || !y) return mfail(m, TURRET_EINVAL, "NULL argument");
    if (n < 1 || n > m->cap) return mfail(m, TURRET_EINVAL, "batch outside 1..capacity");
    if (m->precision == 0) {
        MK(launch_rows(m->dev, x, n, y, m->stream), "forward");
        return TURRET_OK;
    }
    MK(prepare(m, x, nullptr, n), "standardise");
    MK(forward(m, n), "forward");
    k_unstandardise<<<(n * MLP_OUT + 255) / 256, 256, 0, m->stream>>>(m->Y, n, m->dev.mean_y, m->dev.std_y, y);
    MK(cudaGetLastError(), "unstandardise");
    return TURRET_OK;
}

extern "C" turret_status mlp_infer(turret_mlp *m, const float *x, int32_t n, float *y) {
    if (!m || !x || !y) return mfail(m, TURRET_EINVAL, "NULL argument");
    if (n < 1) return mfail(m, TURRET_EINVAL, "empty batch");
    MK(launch_mlp_infer(m->dev, x, n, y, m->stream), "infer");
    return TURRET_OK;
}

extern "C" turret_status mlp_loss_grad(turret_mlp *m, const float *x, const float *y, int32_t n, float *loss,
                                       float *grad) {
    if (!m || !x || !y || !loss) return mfail(m, TURRET_EINVAL, "NULL argument");
    if (n < 1 || n > m->cap) return mfail(m, TURRET_EINVAL, "batch outside 1..capacity");
    if (m->precision == 0) {
        MK(train_bf16(m, x, y, n, nullptr, 1.0f, 1.0f), "loss and gradient");
    } else {
        MK(prepare(m, x, y, n), "standardise");
        MK(forward(m, n), "forward");
        MK(backward(m, n), "backward");
    }
    if (grad) MK(cudaMemcpyAsync(grad, m->G, MLP_NPARAM * 4, cudaMemcpyDeviceToDevice, m->stream), "grad");
    MK(read_loss(m, loss), "loss");
    return TURRET_OK;
}

namespace {
// One training step's kernels on the network's stream.
cudaError_t enqueue_train(turret_mlp *m, const float *x, const float *y, int n, const turret_adamw *opt, float bc1,
                          float bc2) {
    cudaError_t e = prepare(m, x, y, n);
    if (e == cudaSuccess) e = forward(m, n);
    if (e == cudaSuccess) e = backward(m, n);
    if (e != cudaSuccess) return e;
    k_adamw<<<(MLP_NPARAM + 255) / 256, 256, 0, m->stream>>>(m->P, m->G, m->Mm, m->Vv, opt->lr, opt->beta1,
                                                             opt->beta2, opt->eps, opt->weight_decay, bc1, bc2);
    if ((e = cudaGetLastError()) != cudaSuccess) return e;
    return refresh(m);
}

void drop_train_graph(turret_mlp *m) {
    if (m->train_exec) cudaGraphExecDestroy(m->train_exec);
    if (m->train_graph) cudaGraphDestroy(m->train_graph);
    m->train_exec = nullptr;
    m->train_graph = nullptr;
    m->train_n = 0;
}

// Capture the training step for batch size n and find the nodes whose
// arguments change between steps (the two standardisations, AdamW).
cudaError_t capture_train(turret_mlp *m, const float *x, const float *y, int n, const turret_adamw *opt) {
    drop_train_graph(m);
    cudaGraph_t gr;
    cudaError_t e = cudaStreamBeginCapture(m->stream, cudaStreamCaptureModeThreadLocal);
    if (e != cudaSuccess) return e;
    e = enqueue_train(m, x, y, n, opt, 1.0f, 1.0f);
    cudaError_t e2 = cudaStreamEndCapture(m->stream, &gr);
    if (e != cudaSuccess) {
        if (e2 == cudaSuccess) cudaGraphDestroy(gr);
        return e;
    }
    if (e2 != cudaSuccess) return e2;
    size_t nn = 0;
    m->node_x = m->node_y = m->node_adam = nullptr;
    e = cudaGraphGetNodes(gr, nullptr, &nn);
    std::vector<cudaGraphNode_t> nodes(nn);
    if (e == cudaSuccess) e = cudaGraphGetNodes(gr, nodes.data(), &nn);
    for (size_t k = 0; k < nn && e == cudaSuccess; ++k) {
        cudaGraphNodeType t;
        if (cudaGraphNodeGetType(nodes[k], &t) != cudaSuccess || t != cudaGraphNodeTypeKernel) continue;
        cudaKernelNodeParams kp;
        if ((e = cudaGraphKernelNodeGetParams(nodes[k], &kp)) != cudaSuccess) break;
        if (kp.func == (void *)k_adamw) m->node_adam = nodes[k];
        if (kp.func == (void *)k_standardise) {
            const int d = *static_cast<const int *>(kp.kernelParams[2]);
            (d == MLP_IN ? m->node_x : m->node_y) = nodes[k];
        }
    }
    if (e == cudaSuccess && (!m->node_x || !m->node_y || !m->node_adam)) e = cudaErrorInvalidValue;
    if (e == cudaSuccess) e = cudaGraphInstantiate(&m->train_exec, gr, 0);
    if (e != cudaSuccess) {
        cudaGraphDestroy(gr);
        m->train_exec = nullptr;
        return e;
    }
    m->train_graph = gr;
    m->train_n = n;
    return cudaSuccess;
}

// Replay the captured step with this step's inputs and optimiser scalars.
cudaError_t replay_train(turret_mlp *m, const float *x, const float *y, int n, const turret_adamw *opt, float bc1,
                         float bc2) {
    cudaKernelNodeParams kp;
    memset(&kp, 0, sizeof kp);
    int d = MLP_IN;
    const float *mean = m->norm, *stdv = m->norm + MLP_IN;
    float *outp = m->X0;
    void *args_x[6] = {&x, &n, &d, &mean, &stdv, &outp};
    kp.func = (void *)k_standardise;
    kp.gridDim = dim3((n * MLP_IN + 255) / 256);
    kp.blockDim = dim3(256);
    kp.kernelParams = args_x;
    cudaError_t e = cudaGraphExecKernelNodeSetParams(m->train_exec, m->node_x, &kp);
    if (e != cudaSuccess) return e;
    int dy = MLP_OUT;
    const float *meany = m->norm + 2 * MLP_IN, *stdy = m->norm + 2 * MLP_IN + MLP_OUT;
    float *outy = m->T;
    void *args_y[6] = {&y, &n, &dy, &meany, &stdy, &outy};
    kp.gridDim = dim3((n * MLP_OUT + 255) / 256);
    kp.kernelParams = args_y;
    if ((e = cudaGraphExecKernelNodeSetParams(m->train_exec, m->node_y, &kp)) != cudaSuccess) return e;
    float lr = opt->lr, b1 = opt->beta1, b2 = opt->beta2, eps = opt->eps, wd = opt->weight_decay;
    void *args_a[11] = {&m->P, &m->G, &m->Mm, &m->Vv, &lr, &b1, &b2, &eps, &wd, &bc1, &bc2};
    kp.func = (void *)k_adamw;
    kp.gridDim = dim3((MLP_NPARAM + 255) / 256);
    kp.kernelParams = args_a;
    if ((e = cudaGraphExecKernelNodeSetParams(m->train_exec, m->node_adam, &kp)) != cudaSuccess) return e;
    return cudaGraphLaunch(m->train_exec, m->stream);
}
}  // namespace

extern "C" turret_status mlp_train_step(turret_mlp *m, const float *x, const float *y, int32_t n,
                                        const turret_adamw *opt, float *loss) {
    if (!m || !x || !y || !opt) return mfail(m, TURRET_EINVAL, "NULL argument");
    if (n < 1 || n > m->cap) return mfail(m, TURRET_EINVAL, "batch outside 1..capacity");
    if (!(opt->lr >= 0.0f) || !(opt->beta1 >= 0.0f && opt->beta1 < 1.0f) || !(opt->beta2 >= 0.0f && opt->beta2 < 1.0f) ||
        !(opt->eps > 0.0f) || !(opt->weight_decay >= 0.0f))
        return mfail(m, TURRET_EINVAL, "invalid optimiser settings");
    if (m->stream) {  // the step count is part of the update: not for replay in a caller's graph
        cudaStreamCaptureStatus cs = cudaStreamCaptureStatusNone;
        MK(cudaStreamIsCapturing(m->stream, &cs), "training step");
        if (cs != cudaStreamCaptureStatusNone) return mfail(m, TURRET_ECUDA, "training step on a capturing stream");
    }
    m->adam_step += 1;
    const float bc1 = (float)(1.0 - pow((double)opt->beta1, (double)m->adam_step));
    const float bc2 = (float)(1.0 - pow((double)opt->beta2, (double)m->adam_step));
    if (m->precision == 0) {
        MK(train_bf16(m, x, y, n, opt, bc1, bc2), "training step");
    } else if (m->stream) {
        // FP32: a graph replay per step (the captured step has 28 kernels)
        if (m->train_n != n) MK(capture_train(m, x, y, n, opt), "training graph capture");
        MK(replay_train(m, x, y, n, opt, bc1, bc2), "training graph launch");
    } else {
        MK(enqueue_train(m, x, y, n, opt, bc1, bc2), "training step");
    }
    if (loss) MK(read_loss(m, loss), "loss");
    return TURRET_OK;
}

extern "C" turret_status mlp_destroy(turret_mlp *m) {
    if (!m) return TURRET_EINVAL;
    if (m->stream || m->host_loss) cudaStreamSynchronize(m->stream);
    drop_train_graph(m);
    if (m->host_loss) cudaFreeHost(m->host_loss);
    delete m;
    return TURRET_OK;
}

extern "C" const char *mlp_last_error(const turret_mlp *m) { return m ? m->err.c_str() : g_mlp_err.c_str(); }

extern "C" turret_status mlp_build_samples(const double *log, int64_t n_records, float *x, float *y, int32_t *bad,
                                           void *stream) {
    if (!log || !x || !y || !bad || n_records < 5) return TURRET_EINVAL;
    const long long ns = n_records - 4;
    cudaStream_t s = (cudaStream_t)stream;
    if (cudaMemsetAsync(bad, 0, sizeof(int32_t), s) != cudaSuccess) return TURRET_ECUDA;
    k_build_samples<<<(unsigned)((ns + 127) / 128), 128, 0, s>>>(log, ns, x, y, bad);
    return cudaGetLastError() == cudaSuccess ? TURRET_OK : TURRET_ECUDA;
}

// Device view of a network, for the step's predictor.
const MlpDev *mlp_device_view(const turret_mlp *m) { return m ? &m->dev : nullptr; }
