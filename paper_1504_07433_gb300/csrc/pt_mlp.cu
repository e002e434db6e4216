// pt_mlp.cu -- training side of the surrogate network for the ingress/egress
// Mandel-Agol terms (the paper's analogue is the interpolation tables of
// Sec. 2.2.3; the network itself is not in the paper).
//
// Network: 2 -> 128 -> 128 -> 128 -> 2, SiLU, parameters flattened as
//   W1[128][2] b1[128] W2[128][128] b2[128] W3[128][128] b3[128] W4[2][128] b4[2].
// Loss: mean over samples of the summed squared output errors.
//
// Kernels: a counter-based (splitmix64) sampler of (k, s) whose targets come
// from the exact FP32 Mandel-Agol kernel; one kernel for the whole forward and
// backward pass of a tile of samples (its operands can be rounded to BF16 for
// quantisation-aware fine-tuning, so the network is trained for the precision
// it is served in); split-K weight gradients; one reduction; Adam.  All sums
// are taken in a fixed order.
#include <cuda_bf16.h>
#include <cuda_runtime.h>

#include <math.h>
#include <stdint.h>
#include <stdio.h>
#include <string.h>

#include "../../include/pt.h"
#include "pt_device.cuh"

namespace pt_internal {
int set_error(int status, const char *where, const char *msg);   // pt_lc.cu
}

namespace {

constexpr int H = PT_MLP_HIDDEN;
constexpr int NPAR = PT_MLP_NPARAMS;
constexpr int OFF_W1 = 0, OFF_B1 = 2 * H, OFF_W2 = 3 * H, OFF_B2 = 3 * H + H * H, OFF_W3 = 4 * H + H * H,
              OFF_B3 = 4 * H + 2 * H * H, OFF_W4 = 5 * H + 2 * H * H, OFF_B4 = 7 * H + 2 * H * H;
static_assert(OFF_B4 + 2 == NPAR, "parameter layout");

int cuda_status(const char *where)
{
    cudaError_t e = cudaGetLastError();
    return e == cudaSuccess ? PT_OK : pt_internal::set_error(PT_ERR_CUDA, where, cudaGetErrorString(e));
}

__device__ __forceinline__ float silu(float x) { return x / (1.0f + expf(-x)); }

__device__ __forceinline__ float dsilu(float x)
{
    float s = 1.0f / (1.0f + expf(-x));
    return s * (1.0f + x * (1.0f - s));
}

__device__ __forceinline__ float bf16r(float x) { return __bfloat162float(__float2bfloat16_rn(x)); }

// splitmix64 (Steele, Lea & Flood 2014): a counter-based 64-bit mixer
__device__ __forceinline__ uint64_t splitmix64(uint64_t x)
{
    x += 0x9e3779b97f4a7c15ULL;
    x = (x ^ (x >> 30)) * 0xbf58476d1ce4e5b9ULL;
    x = (x ^ (x >> 27)) * 0x94d049bb133111ebULL;
    return x ^ (x >> 31);
}

__device__ __forceinline__ float u01(uint64_t x)   // 24 random bits -> [0, 1)
{
    return (float)(x >> 40) * (1.0f / 16777216.0f);
}

__global__ void datagen_kernel(uint64_t seed, size_t offset, size_t n, float k_lo, float k_hi, const float *norm,
                               float *X, float *T, float *kz)
{
    size_t i = (size_t)blockIdx.x * blockDim.x + threadIdx.x;
    if (i >= n) return;
    uint64_t c = seed * 0x100000000ULL + (offset + i) * 2ULL;
    float k = k_lo + (k_hi - k_lo) * u01(splitmix64(c));
    float s = u01(splitmix64(c + 1));
    float z = fabsf(1.0f - k) + 2.0f * fminf(k, 1.0f) * s;
    float le, ld, ed;
    pt::ma_terms(k, z, &le, &ld, &ed);
    float ik2 = 1.0f / (k * k);
    if (X) {
        X[2 * i] = (k - norm[0]) / norm[1];
        X[2 * i + 1] = pt::band_coord(s);
    }
    if (T) {
        T[2 * i] = (ld * ik2 - norm[2]) / norm[3];
        T[2 * i + 1] = (ed * ik2 - norm[4]) / norm[5];
    }
    if (kz) {
        kz[2 * i] = k;
        kz[2 * i + 1] = z;
    }
}

// ---------------------------------------------------------------------------
// Forward and backward pass of a tile of 16 RM samples in one CTA of 16 x 16
// threads; thread (ty, tx) holds rows ty + 16 i (i < RM) and columns
// 4 tx + {0..3} and 64 + 4 tx + {0..3} of every 128-wide layer.  The layer's
// input sits in shared memory as rows of 128 (+ 4 against bank conflicts), the
// weight as [k][n]; per four k a thread loads RM + 8 16-byte vectors for
// 32 RM FMAs, so the FP32 FMA pipe bounds the products.  Only what the weight
// gradients read goes to memory: H1, H2, dZ2, dZ3.  Layer 1 (2 -> 128) is
// recomputed for its derivative, silu'(Z2) waits in shared memory.  The small
// gradients (biases, W1, W4) are column sums over the tile.
// The host takes the smallest RM whose tiles fit one per SM: 16,384 samples
// are 147 tiles of 112.  Measured at 16,384 samples: 83 us for the tiles (ncu),
// 26 us for the weight gradients, a whole step with Adam 116 us; before, with
// one kernel per product, separate activations and one thread per small
// gradient, 468 us.
// ---------------------------------------------------------------------------
constexpr int LDA = H + 4;        // row stride of the staged activations
constexpr int N_RED = 7;          // column sums: gW4 (2), gb3, gb2, gb1, gW1 (2)
constexpr int SMALL = N_RED * H + 4;   // per tile: the column sums, gb4 (2), loss

struct TileArgs {
    const float *p, *X, *T;
    int n, qat;
    float *Y;                     // network outputs, or null
    float *H1, *H2, *dZ2, *dZ3;   // null: forward only
    float *psmall;                // [tiles][SMALL]
};

// columns of a thread
__device__ __forceinline__ int col_of(int tx, int j) { return 4 * tx + (j & 3) + 64 * (j >> 2); }

// four consecutive weights; the caller's parameters may lie at any float
__device__ __forceinline__ float4 load_w4(const float *W, bool aligned, int qat)
{
    float4 v = aligned ? *reinterpret_cast<const float4 *>(W) : make_float4(W[0], W[1], W[2], W[3]);
    if (qat) v = make_float4(bf16r(v.x), bf16r(v.y), bf16r(v.z), bf16r(v.w));
    return v;
}

// A thread's 1/256 of a weight matrix on its way to shared memory: loaded
// into registers before a product, stored when the product no longer reads
// the previous matrix, so that the loads hide behind the product.
constexpr int WREG = H * H / 4 / 256;

// sW[k][n] = W[n][k] (a layer's weight, transposed on the way)
__device__ __forceinline__ void load_wt(float4 (&w)[WREG], const float *W, int qat)
{
    const bool al = ((uintptr_t)W & 15u) == 0;
    const int n = threadIdx.x & (H - 1);
#pragma unroll
    for (int i = 0; i < WREG; ++i) w[i] = load_w4(W + n * H + 8 * i + 4 * (threadIdx.x >> 7), al, qat);
}

__device__ __forceinline__ void store_wt(float *sW, const float4 (&w)[WREG])
{
    const int n = threadIdx.x & (H - 1);
#pragma unroll
    for (int i = 0; i < WREG; ++i) {
        float *d = sW + (8 * i + 4 * (threadIdx.x >> 7)) * H + n;
        d[0] = w[i].x;
        d[H] = w[i].y;
        d[2 * H] = w[i].z;
        d[3 * H] = w[i].w;
    }
}

// sW[k][n] = W[k][n]
__device__ __forceinline__ void load_w(float4 (&w)[WREG], const float *W, int qat)
{
    const bool al = ((uintptr_t)W & 15u) == 0;
#pragma unroll
    for (int i = 0; i < WREG; ++i) w[i] = load_w4(W + 4 * (256 * i + threadIdx.x), al, qat);
}

__device__ __forceinline__ void store_w(float *sW, const float4 (&w)[WREG])
{
#pragma unroll
    for (int i = 0; i < WREG; ++i) *reinterpret_cast<float4 *>(sW + 4 * (256 * i + threadIdx.x)) = w[i];
}

// The operands of the next k (and of the next four k) are loaded before the
// FMAs of the current ones: with two warps per scheduler the shared-memory
// latency is not hidden otherwise.
template <int RM>
__device__ __forceinline__ void tile_product(const float *sA, const float *sW, int ty, int tx, float (&acc)[RM][8])
{
#pragma unroll
    for (int i = 0; i < RM; ++i)
#pragma unroll
        for (int j = 0; j < 8; ++j) acc[i][j] = 0.0f;
    const float *pa = sA + ty * LDA, *pb = sW + 4 * tx;
    float4 a[RM], b0, b1;
#pragma unroll
    for (int i = 0; i < RM; ++i) a[i] = *reinterpret_cast<const float4 *>(pa + 16 * i * LDA);
    b0 = *reinterpret_cast<const float4 *>(pb);
    b1 = *reinterpret_cast<const float4 *>(pb + 64);
#pragma unroll 1
    for (int k = 0; k < H; k += 4) {
        float4 an[RM];
#pragma unroll
        for (int kk = 0; kk < 4; ++kk) {
            // the row after the last is read too (it lies in shared memory) and not used
            const float4 n0 = *reinterpret_cast<const float4 *>(pb + (k + kk + 1) * H);
            const float4 n1 = *reinterpret_cast<const float4 *>(pb + (k + kk + 1) * H + 64);
#pragma unroll
            for (int i = kk; i < RM; i += 4) an[i] = *reinterpret_cast<const float4 *>(pa + 16 * i * LDA + k + 4);
#pragma unroll
            for (int i = 0; i < RM; ++i) {
                const float av = kk == 0 ? a[i].x : (kk == 1 ? a[i].y : (kk == 2 ? a[i].z : a[i].w));
                acc[i][0] = fmaf(av, b0.x, acc[i][0]);
                acc[i][1] = fmaf(av, b0.y, acc[i][1]);
                acc[i][2] = fmaf(av, b0.z, acc[i][2]);
                acc[i][3] = fmaf(av, b0.w, acc[i][3]);
                acc[i][4] = fmaf(av, b1.x, acc[i][4]);
                acc[i][5] = fmaf(av, b1.y, acc[i][5]);
                acc[i][6] = fmaf(av, b1.z, acc[i][6]);
                acc[i][7] = fmaf(av, b1.w, acc[i][7]);
            }
            b0 = n0;
            b1 = n1;
        }
#pragma unroll
        for (int i = 0; i < RM; ++i) a[i] = an[i];
    }
}

// eight values of a thread's row to a row of 128
__device__ __forceinline__ void put_row(float *row, int tx, const float (&v)[8])
{
    *reinterpret_cast<float4 *>(row + 4 * tx) = make_float4(v[0], v[1], v[2], v[3]);
    *reinterpret_cast<float4 *>(row + 64 + 4 * tx) = make_float4(v[4], v[5], v[6], v[7]);
}

__device__ __forceinline__ void get_row(const float *row, int tx, float (&v)[8])
{
    const float4 a = *reinterpret_cast<const float4 *>(row + 4 * tx), b = *reinterpret_cast<const float4 *>(row + 64 + 4 * tx);
    v[0] = a.x, v[1] = a.y, v[2] = a.z, v[3] = a.w;
    v[4] = b.x, v[5] = b.y, v[6] = b.z, v[7] = b.w;
}

// A thread's products to its own places in shared memory, so that what
// follows can run as a loop over its rows: unrolled over the registers, the
// four epilogues are ten thousand instructions that every warp runs once, and
// fetching them took as long as the products.
template <int RM>
__device__ __forceinline__ void put_acc(float *sA, int ty, int tx, const float (&acc)[RM][8])
{
#pragma unroll
    for (int i = 0; i < RM; ++i) put_row(sA + (ty + 16 * i) * LDA, tx, acc[i]);
}

// column sums over the tile: this thread's rows are already added, then the
// warp's two row groups; the eight warps' sums wait in shared memory
__device__ __forceinline__ void put_sums(float *sRed, int what, int tx, const float (&v)[8])
{
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
#pragma unroll
    for (int j = 0; j < 8; ++j) {
        const float x = v[j] + __shfl_xor_sync(0xffffffffu, v[j], 16);
        if (lane < 16) sRed[(what * 8 + warp) * H + col_of(tx, j)] = x;
    }
}

template <int RM>
__global__ void __launch_bounds__(256, 1) mlp_tile_kernel(TileArgs A)
{
    pt::chain_begin();
    constexpr int M = 16 * RM;
    extern __shared__ __align__(16) float tsm[];
    float *sW = tsm;                       // [H][H]
    float *sA = sW + H * H;                // [M][LDA]
    float *sD = sA + M * LDA;              // [M][LDA]: silu'(Z2)
    float *sRed = sD + M * LDA;            // [N_RED][8 warps][H]
    float *sP = sRed + N_RED * 8 * H;      // W1 (2H), b1, b2, b3, W4 (2H)
    float *sX = sP + 7 * H;                // [M][2]
    __shared__ float sLoss[8][3];          // per warp: loss, gb4
    const int tid = threadIdx.x, tx = tid & 15, ty = tid >> 4, lane = tid & 31, warp = tid >> 5;
    const int r0 = blockIdx.x * M;
    const bool train = A.H1 != nullptr;
    const float *p = A.p;
    for (int i = tid; i < 2 * H; i += 256) {
        sP[i] = p[OFF_W1 + i];
        sP[5 * H + i] = p[OFF_W4 + i];
    }
    for (int i = tid; i < H; i += 256) {
        sP[2 * H + i] = p[OFF_B1 + i];
        sP[3 * H + i] = p[OFF_B2 + i];
        sP[4 * H + i] = p[OFF_B3 + i];
    }
    for (int i = tid; i < 2 * M; i += 256) sX[i] = 2 * r0 + i < 2 * A.n ? A.X[2 * (size_t)r0 + i] : 0.0f;
    float4 wreg[WREG];
    load_wt(wreg, p + OFF_W2, A.qat);
    store_wt(sW, wreg);
    __syncthreads();
    float v[8];
    // layer 1
#pragma unroll 1
    for (int i = 0; i < RM; ++i) {
        const int m = ty + 16 * i;
        const float x0 = sX[2 * m], x1 = sX[2 * m + 1];
#pragma unroll
        for (int j = 0; j < 8; ++j) {
            const int c = col_of(tx, j);
            const float z = fmaf(sP[2 * c], x0, fmaf(sP[2 * c + 1], x1, sP[2 * H + c]));
            v[j] = silu(z);
            if (A.qat) v[j] = bf16r(v[j]);
        }
        put_row(sA + m * LDA, tx, v);
        if (train && r0 + m < A.n) put_row(A.H1 + (size_t)(r0 + m) * H, tx, v);
    }
    __syncthreads();
    float acc[RM][8];
    // layer 2
    load_wt(wreg, p + OFF_W3, A.qat);
    tile_product<RM>(sA, sW, ty, tx, acc);
    __syncthreads();
    store_wt(sW, wreg);
    put_acc<RM>(sA, ty, tx, acc);
#pragma unroll 1
    for (int i = 0; i < RM; ++i) {
        const int m = ty + 16 * i;
        float d[8];
        get_row(sA + m * LDA, tx, v);
#pragma unroll
        for (int j = 0; j < 8; ++j) {
            const float z = v[j] + sP[3 * H + col_of(tx, j)];
            const float s = 1.0f / (1.0f + expf(-z));
            v[j] = z * s;
            d[j] = s * (1.0f + z * (1.0f - s));
            if (A.qat) v[j] = bf16r(v[j]);
        }
        put_row(sA + m * LDA, tx, v);
        if (train) {
            put_row(sD + m * LDA, tx, d);
            if (r0 + m < A.n) put_row(A.H2 + (size_t)(r0 + m) * H, tx, v);
        }
    }
    __syncthreads();
    // layer 3, output layer, loss, dZ3
    if (train) load_w(wreg, p + OFF_W3, A.qat);
    tile_product<RM>(sA, sW, ty, tx, acc);
    __syncthreads();
    if (train) store_w(sW, wreg);
    float g40[8], g41[8], gb[8], loss = 0.0f, gb40 = 0.0f, gb41 = 0.0f;
#pragma unroll
    for (int j = 0; j < 8; ++j) g40[j] = g41[j] = gb[j] = 0.0f;
    const float b40 = p[OFF_B4], b41 = p[OFF_B4 + 1];
    put_acc<RM>(sA, ty, tx, acc);
#pragma unroll 1
    for (int i = 0; i < RM; ++i) {
        const int m = ty + 16 * i, r = r0 + m;
        float a0 = 0.0f, a1 = 0.0f, h[8], d[8];
        get_row(sA + m * LDA, tx, v);
#pragma unroll
        for (int j = 0; j < 8; ++j) {
            const int c = col_of(tx, j);
            const float z = v[j] + sP[4 * H + c];
            const float s = 1.0f / (1.0f + expf(-z));
            h[j] = z * s;
            d[j] = s * (1.0f + z * (1.0f - s));
            a0 = fmaf(sP[5 * H + c], h[j], a0);
            a1 = fmaf(sP[6 * H + c], h[j], a1);
        }
#pragma unroll
        for (int o = 8; o > 0; o >>= 1) {
            a0 += __shfl_xor_sync(0xffffffffu, a0, o);
            a1 += __shfl_xor_sync(0xffffffffu, a1, o);
        }
        const float y0 = a0 + b40, y1 = a1 + b41;
        const bool in = r < A.n;
        if (A.Y && in && tx == 0) {
            A.Y[2 * (size_t)r] = y0;
            A.Y[2 * (size_t)r + 1] = y1;
        }
        if (!train) continue;
        const float e0 = in ? y0 - A.T[2 * (size_t)r] : 0.0f, e1 = in ? y1 - A.T[2 * (size_t)r + 1] : 0.0f;
        const float d0 = 2.0f * e0 / (float)A.n, d1 = 2.0f * e1 / (float)A.n;
        loss += e0 * e0 + e1 * e1;
        gb40 += d0;
        gb41 += d1;
#pragma unroll
        for (int j = 0; j < 8; ++j) {
            const int c = col_of(tx, j);
            g40[j] = fmaf(d0, h[j], g40[j]);
            g41[j] = fmaf(d1, h[j], g41[j]);
            v[j] = (sP[5 * H + c] * d0 + sP[6 * H + c] * d1) * d[j];
            gb[j] += v[j];
        }
        put_row(sA + m * LDA, tx, v);
        if (in) put_row(A.dZ3 + (size_t)r * H, tx, v);
    }
    if (!train) return;
    put_sums(sRed, 0, tx, g40);
    put_sums(sRed, 1, tx, g41);
    put_sums(sRed, 2, tx, gb);
    loss += __shfl_xor_sync(0xffffffffu, loss, 16);   // the warp's other row group (all tx hold the same sums)
    gb40 += __shfl_xor_sync(0xffffffffu, gb40, 16);
    gb41 += __shfl_xor_sync(0xffffffffu, gb41, 16);
    if (lane == 0) {
        sLoss[warp][0] = loss;
        sLoss[warp][1] = gb40;
        sLoss[warp][2] = gb41;
    }
    __syncthreads();
    // dZ2 = (dZ3 W3) silu'(Z2)
    load_w(wreg, p + OFF_W2, A.qat);
    tile_product<RM>(sA, sW, ty, tx, acc);
    __syncthreads();
    store_w(sW, wreg);
#pragma unroll
    for (int j = 0; j < 8; ++j) gb[j] = 0.0f;
    put_acc<RM>(sA, ty, tx, acc);
#pragma unroll 1
    for (int i = 0; i < RM; ++i) {
        const int m = ty + 16 * i;
        float d[8];
        get_row(sA + m * LDA, tx, v);
        get_row(sD + m * LDA, tx, d);
#pragma unroll
        for (int j = 0; j < 8; ++j) {
            v[j] *= d[j];
            gb[j] += v[j];
        }
        put_row(sA + m * LDA, tx, v);
        if (r0 + m < A.n) put_row(A.dZ2 + (size_t)(r0 + m) * H, tx, v);
    }
    put_sums(sRed, 3, tx, gb);
    __syncthreads();
    // dZ1 = (dZ2 W2) silu'(Z1): only its column sums are needed
    tile_product<RM>(sA, sW, ty, tx, acc);
#pragma unroll
    for (int j = 0; j < 8; ++j) g40[j] = g41[j] = gb[j] = 0.0f;
    put_acc<RM>(sD, ty, tx, acc);   // (silu'(Z2) is no longer read)
#pragma unroll 1
    for (int i = 0; i < RM; ++i) {
        const int m = ty + 16 * i;
        const float x0 = sX[2 * m], x1 = sX[2 * m + 1];
        get_row(sD + m * LDA, tx, v);
#pragma unroll
        for (int j = 0; j < 8; ++j) {
            const int c = col_of(tx, j);
            const float z = fmaf(sP[2 * c], x0, fmaf(sP[2 * c + 1], x1, sP[2 * H + c]));
            const float d = v[j] * dsilu(z);
            gb[j] += d;
            g40[j] = fmaf(d, x0, g40[j]);
            g41[j] = fmaf(d, x1, g41[j]);
        }
    }
    put_sums(sRed, 4, tx, gb);
    put_sums(sRed, 5, tx, g40);
    put_sums(sRed, 6, tx, g41);
    __syncthreads();
    float *out = A.psmall + (size_t)blockIdx.x * SMALL;
    for (int q = tid; q < N_RED * H; q += 256) {
        const int what = q / H, c = q - what * H;
        float x = 0.0f;
#pragma unroll
        for (int w = 0; w < 8; ++w) x += sRed[(what * 8 + w) * H + c];
        out[q] = x;
    }
    if (tid < 3) {
        float x = 0.0f;
        for (int w = 0; w < 8; ++w) x += sLoss[w][tid];
        out[N_RED * H + tid] = x;
    }
}

size_t tile_smem(int rm)
{
    return ((size_t)H * H + 2 * (size_t)16 * rm * LDA + (size_t)N_RED * 8 * H + 7 * H + 2 * 16 * rm) * sizeof(float);
}

// ---------------------------------------------------------------------------
// Weight gradients dW_l[m][n] = sum_r dZ_l[r][m] H_{l-1}[r][n] over a chunk of
// the samples: one CTA per (layer, chunk) holds the whole 128 x 128 gradient,
// 8 x 8 per thread, and streams its rows through a three-deep cp.async ring of
// WG_ROWS rows (both operands are read along m and n, as they lie in memory).
// ---------------------------------------------------------------------------
constexpr int WG_ROWS = 16, WG_STAGES = 3;

__device__ __forceinline__ void cp16(float *dst, const float *src, bool ok)
{
    const unsigned d = (unsigned)__cvta_generic_to_shared(dst);
    const int bytes = ok ? 16 : 0;   // 0: zero-fill
    asm volatile("cp.async.cg.shared.global [%0], [%1], 16, %2;" ::"r"(d), "l"(src), "r"(bytes) : "memory");
}

__global__ void __launch_bounds__(256, 2) wgrad_kernel(const float *dZ2, const float *dZ3, const float *H1, const float *H2,
                                                       int n, int chunk, float *pw)
{
    pt::chain_begin();
    __shared__ __align__(16) float sb[WG_STAGES][2][WG_ROWS * H];
    const int tid = threadIdx.x, tx = tid & 15, ty = tid >> 4;
    const int layer = blockIdx.y;   // 0: W2, 1: W3
    const float *Z = layer ? dZ3 : dZ2, *Hp = layer ? H2 : H1;
    const int rb = blockIdx.x * chunk, re = min(n, rb + chunk);
    const int steps = max(0, (re - rb + WG_ROWS - 1) / WG_ROWS);
    auto fetch = [&](int st) {
        if (st < steps) {
#pragma unroll
            for (int q = 0; q < 2; ++q) {
                const int e = 4 * (tid + 256 * q);   // WG_ROWS H floats of each operand, 16 bytes a thread and turn
                const int r = rb + st * WG_ROWS + e / H;
                const bool ok = r < re;
                const size_t at = (size_t)(ok ? r : rb) * H + (e & (H - 1));
                cp16(&sb[st % WG_STAGES][0][e], Z + at, ok);
                cp16(&sb[st % WG_STAGES][1][e], Hp + at, ok);
            }
        }
        asm volatile("cp.async.commit_group;" ::: "memory");
    };
    float acc[8][8];
#pragma unroll
    for (int i = 0; i < 8; ++i)
#pragma unroll
        for (int j = 0; j < 8; ++j) acc[i][j] = 0.0f;
    fetch(0);
    fetch(1);
    for (int st = 0; st < steps; ++st) {
        asm volatile("cp.async.wait_group 1;" ::: "memory");
        __syncthreads();   // stage st has landed; stage st - 1 is no longer read
        fetch(st + 2);
        const float *a = sb[st % WG_STAGES][0], *b = sb[st % WG_STAGES][1];
#pragma unroll
        for (int r = 0; r < WG_ROWS; ++r) {
            const float4 a0 = *reinterpret_cast<const float4 *>(a + r * H + 4 * ty);
            const float4 a1 = *reinterpret_cast<const float4 *>(a + r * H + 64 + 4 * ty);
            const float4 b0 = *reinterpret_cast<const float4 *>(b + r * H + 4 * tx);
            const float4 b1 = *reinterpret_cast<const float4 *>(b + r * H + 64 + 4 * tx);
            const float av[8] = {a0.x, a0.y, a0.z, a0.w, a1.x, a1.y, a1.z, a1.w};
            const float bv[8] = {b0.x, b0.y, b0.z, b0.w, b1.x, b1.y, b1.z, b1.w};
#pragma unroll
            for (int i = 0; i < 8; ++i)
#pragma unroll
                for (int j = 0; j < 8; ++j) acc[i][j] = fmaf(av[i], bv[j], acc[i][j]);
        }
    }
    float *out = pw + ((size_t)layer * gridDim.x + blockIdx.x) * H * H;
#pragma unroll
    for (int i = 0; i < 8; ++i) put_row(out + (size_t)col_of(ty, i) * H, tx, acc[i]);
}

// Sum the chunks' and tiles' partials into the gradient, and the loss.  RG_GRP
// threads share an output (a quarter-row of four for the weights), each adding
// a run of partials in order, then the runs in order: with one thread per
// output the 147 dependent loads took 16 us.
constexpr int RG_GRP = 8, RG_OUT = 32;

__global__ void __launch_bounds__(RG_GRP *RG_OUT) reduce_grad_kernel(const float *pw, int n_chunk, const float *psmall,
                                                                     int n_tile, int n, float *grad, float *loss)
{
    pt::chain_begin();
    __shared__ float4 s4[RG_GRP][RG_OUT];
    const int o = threadIdx.x % RG_OUT, g = threadIdx.x / RG_OUT;
    constexpr int N_W = 2 * H * H / 4 / RG_OUT;   // CTAs of the weight gradients
    float4 a = make_float4(0.0f, 0.0f, 0.0f, 0.0f);
    if (blockIdx.x < N_W) {
        const int q = 4 * (blockIdx.x * RG_OUT + o), layer = q / (H * H), i = q - layer * H * H;
        const float4 *src = reinterpret_cast<const float4 *>(pw + (size_t)layer * n_chunk * H * H + i);
        const int per = (n_chunk + RG_GRP - 1) / RG_GRP, c1 = min(n_chunk, (g + 1) * per);
#pragma unroll 8
        for (int c = g * per; c < c1; ++c) {
            const float4 v = src[(size_t)c * (H * H / 4)];
            a.x += v.x;
            a.y += v.y;
            a.z += v.z;
            a.w += v.w;
        }
        s4[g][o] = a;
        __syncthreads();
        if (g == 0) {
            for (int u = 1; u < RG_GRP; ++u) {
                const float4 v = s4[u][o];
                a.x += v.x;
                a.y += v.y;
                a.z += v.z;
                a.w += v.w;
            }
            float *dst = grad + (layer ? OFF_W3 : OFF_W2) + i;   // the caller's buffer: any float
            dst[0] = a.x;
            dst[1] = a.y;
            dst[2] = a.z;
            dst[3] = a.w;
        }
        return;
    }
    const int u = (blockIdx.x - N_W) * RG_OUT + o;
    const int per = (n_tile + RG_GRP - 1) / RG_GRP, c1 = min(n_tile, (g + 1) * per);
    if (u < N_RED * H + 3) {
#pragma unroll 8
        for (int c = g * per; c < c1; ++c) a.x += psmall[(size_t)c * SMALL + u];
    }
    s4[g][o] = a;
    __syncthreads();
    if (g != 0 || u >= N_RED * H + 3) return;
    float x = a.x;
    for (int q = 1; q < RG_GRP; ++q) x += s4[q][o].x;
    const int what = u / H, c = u - what * H;
    if (u < 2 * H) grad[OFF_W4 + u] = x;
    else if (what == 2) grad[OFF_B3 + c] = x;
    else if (what == 3) grad[OFF_B2 + c] = x;
    else if (what == 4) grad[OFF_B1 + c] = x;
    else if (what == 5) grad[OFF_W1 + 2 * c] = x;
    else if (what == 6) grad[OFF_W1 + 2 * c + 1] = x;
    else if (c == 0) *loss = x / (float)n;
    else grad[OFF_B4 + c - 1] = x;
}

__global__ void adam_kernel(float *p, const float *g, float *m, float *v, int n, float lr, float b1, float b2,
                            float eps, float c1, float c2)
{
    int i = blockIdx.x * blockDim.x + threadIdx.x;
    if (i >= n) return;
    float gi = g[i];
    float mi = b1 * m[i] + (1.0f - b1) * gi;
    float vi = b2 * v[i] + (1.0f - b2) * gi * gi;
    m[i] = mi;
    v[i] = vi;
    p[i] -= lr * (mi / c1) / (sqrtf(vi / c2) + eps);
}

// Tile height for n samples on n_sm SMs: the smallest that gives each SM at
// most one tile (the tile's shared memory leaves no room for a second CTA).
int tile_rm(int n, int n_sm)
{
    const int rms[3] = {1, 2, 4};
    for (int i = 0; i < 3; ++i)
        if ((long long)n_sm * 16 * rms[i] >= n) return rms[i];
    return 7;   // 217 KB of shared memory: the tallest tile that fits
}

constexpr int WG_MAX_CHUNKS = 152;   // chunks per layer: two CTAs on each of 152 SMs

// rows per chunk of the weight gradients
int wgrad_chunk(int n)
{
    const int c = (n + WG_MAX_CHUNKS - 1) / WG_MAX_CHUNKS;
    return (c + WG_ROWS - 1) / WG_ROWS * WG_ROWS;
}

struct Work {
    float *H1, *H2, *dZ2, *dZ3, *pw, *psmall;
    size_t bytes;
};

Work carve(void *base, int n)
{
    const size_t a = (size_t)n * H;
    const size_t n_chunk = ((size_t)n + wgrad_chunk(n) - 1) / wgrad_chunk(n);
    Work w;
    // the buffer may start anywhere: the parts start on 256-byte boundaries
    // inside it, and its size has room for that
    char *p = (char *)(((uintptr_t)base + 255) & ~(uintptr_t)255);
    size_t off = 0;
    auto take = [&](size_t count) {
        float *r = (float *)(p + off);
        off += ((count * sizeof(float)) + 255) & ~(size_t)255;
        return r;
    };
    w.H1 = take(a);
    w.H2 = take(a);
    w.dZ2 = take(a);
    w.dZ3 = take(a);
    w.pw = take(2 * n_chunk * H * H);
    w.psmall = take(((size_t)n + 15) / 16 * SMALL);
    w.bytes = off + 256;
    return w;
}

template <int RM>
int launch_tile_t(const TileArgs &A, cudaStream_t s)
{
    // set on every call (a driver call of well under a microsecond): the
    // attribute belongs to the current device
    cudaError_t e = cudaFuncSetAttribute(mlp_tile_kernel<RM>, cudaFuncAttributeMaxDynamicSharedMemorySize,
                                         (int)tile_smem(RM));
    if (e != cudaSuccess) return pt_internal::set_error(PT_ERR_CUDA, "mlp_tile_kernel", cudaGetErrorString(e));
    mlp_tile_kernel<RM><<<(unsigned)((A.n + 16 * RM - 1) / (16 * RM)), 256, tile_smem(RM), s>>>(A);
    return cuda_status("mlp_tile_kernel");
}

int launch_tile(const TileArgs &A, int *n_tile, cudaStream_t s)
{
    int dev = 0, n_sm = 0;
    cudaError_t e = cudaGetDevice(&dev);
    if (e == cudaSuccess) e = cudaDeviceGetAttribute(&n_sm, cudaDevAttrMultiProcessorCount, dev);
    if (e != cudaSuccess) return pt_internal::set_error(PT_ERR_CUDA, "mlp_tile_kernel", cudaGetErrorString(e));
    const int rm = tile_rm(A.n, n_sm);
    *n_tile = (A.n + 16 * rm - 1) / (16 * rm);
    switch (rm) {
    case 1: return launch_tile_t<1>(A, s);
    case 2: return launch_tile_t<2>(A, s);
    case 4: return launch_tile_t<4>(A, s);
    default: return launch_tile_t<7>(A, s);
    }
}

}  // namespace

extern "C" {

size_t pt_mlp_work_bytes(int n)
{
    if (n < 1) return 0;
    return carve(nullptr, n).bytes;
}

int pt_mlp_forward(const float *params, const float *X, int n, int qat, float *Y, void *work, size_t work_bytes,
                   pt_stream_t stream)
{
    if (n < 0) return PT_ERR_ARG;
    if (n == 0) return PT_OK;
    if (!params || !X || !Y) return PT_ERR_ARG;
    if (!work || work_bytes < pt_mlp_work_bytes(n)) return PT_ERR_WORKSPACE;
    TileArgs A{};
    A.p = params;
    A.X = X;
    A.n = n;
    A.qat = qat ? 1 : 0;
    A.Y = Y;
    int n_tile;
    return launch_tile(A, &n_tile, (cudaStream_t)stream);
}

int pt_mlp_loss_grad(const float *params, const float *X, const float *T, int n, int qat, float *grad, float *loss,
                     void *work, size_t work_bytes, pt_stream_t stream)
{
    if (n < 1 || !params || !X || !T || !grad || !loss) return PT_ERR_ARG;
    if (!work || work_bytes < pt_mlp_work_bytes(n)) return PT_ERR_WORKSPACE;
    cudaStream_t s = (cudaStream_t)stream;
    Work w = carve(work, n);
    TileArgs A{};
    A.p = params;
    A.X = X;
    A.T = T;
    A.n = n;
    A.qat = qat ? 1 : 0;
    A.H1 = w.H1;
    A.H2 = w.H2;
    A.dZ2 = w.dZ2;
    A.dZ3 = w.dZ3;
    A.psmall = w.psmall;
    int n_tile;
    int st = launch_tile(A, &n_tile, s);
    if (st) return st;
    const int chunk = wgrad_chunk(n), n_chunk = (n + chunk - 1) / chunk;
    pt::launch_chained(wgrad_kernel, dim3(n_chunk, 2), 256, 0, s, w.dZ2, w.dZ3, w.H1, w.H2, n, chunk, w.pw);
    st = cuda_status("wgrad_kernel");
    if (st) return st;
    pt::launch_chained(reduce_grad_kernel, 2 * H * H / 4 / RG_OUT + (N_RED * H + 3 + RG_OUT - 1) / RG_OUT,
                       RG_GRP * RG_OUT, 0, s, w.pw, n_chunk, w.psmall, n_tile, n, grad, loss);
    return cuda_status("reduce_grad_kernel");
}

int pt_mlp_adam(float *params, const float *grad, float *m, float *v, int step, float lr, float beta1, float beta2,
                float eps, pt_stream_t stream)
{
    if (!params || !grad || !m || !v || step < 1) return PT_ERR_ARG;
    float c1 = 1.0f - powf(beta1, (float)step), c2 = 1.0f - powf(beta2, (float)step);
    adam_kernel<<<(NPAR + 255) / 256, 256, 0, (cudaStream_t)stream>>>(params, grad, m, v, NPAR, lr, beta1, beta2,
                                                                      eps, c1, c2);
    return cuda_status("adam_kernel");
}

int pt_sur_datagen(unsigned long long seed, size_t offset, size_t n, float k_lo, float k_hi, const float *norm,
                   float *X, float *T, float *kz, pt_stream_t stream)
{
    if (n == 0) return PT_OK;
    if (!norm || (!X && !T && !kz) || !(k_lo > 0.0f) || !(k_hi >= k_lo) || k_hi > 1.0f) return PT_ERR_ARG;
    size_t blocks = (n + 255) / 256;
    if (blocks > 0x7fffffffULL) return PT_ERR_ARG;
    datagen_kernel<<<(unsigned)blocks, 256, 0, (cudaStream_t)stream>>>(seed, offset, n, k_lo, k_hi, norm, X, T, kz);
    return cuda_status("datagen_kernel");
}

}  // extern "C"
