// pt_lc.cu -- light-curve kernels and their C ABI (include/pt.h).
//
// Kernels of the fused light-curve path (Secs. 2.1, 2.2, 3.2, 3.4):
//   row_prep_kernel     per geometry: conjunction anchor, double-float t0/P and
//                       a conservative transit window; per time: double-float
//                       split; per geometry and passband: the Mandel-Agol row
//                       of polynomials (pt_device.cuh), the caller's table at
//                       the geometry's k, or the Gimenez factors and weights.
//   product_kernel, product_tall_kernel
//                       Gimenez: the rows as FP32 products (pt_gim.cuh).
//   zi_rows_kernel      Gimenez interpolated in z (Sec. 3.3): the node values.
//   lc_rows_kernel      the light curves from the rows (pt_rows.cuh).
//   setup_kernel, ma_lc_kernel
//                       records and the tile kernel (256 times x 8 geometries
//                       per CTA, exact terms per point) of the Mandel-Agol calls
//                       with few geometries or points and without a work buffer.
//   ssr_part_kernel / ssr_reduce_kernel
//                       residual sums in a fixed order.
// Every sum is formed in a fixed order, so results are bitwise reproducible.
#include <cuda_runtime.h>

#include <math.h>
#include <stdint.h>
#include <stdio.h>
#include <string.h>

#include <algorithm>
#include <memory>
#include <mutex>
#include <new>

#include "../../include/pt.h"
#include "pt_device.cuh"
#include "pt_gim.cuh"
#include "pt_rows.cuh"

using pt::GeomRec;

namespace {

constexpr int TT = 256;      // times per CTA (= threads per CTA)
constexpr int VT_MA = 8;     // geometries per CTA, Mandel-Agol
constexpr int MAX_SS = 256;  // supersamples per exposure
constexpr int MAX_NEWTON = 64;  // cap on Newton steps
constexpr double PI_D = 3.14159265358979323846;

thread_local char g_last_error[512] = "";

int set_cuda_error(cudaError_t e, const char *where)
{
    snprintf(g_last_error, sizeof(g_last_error), "%s: %s", where, cudaGetErrorString(e));
    return PT_ERR_CUDA;
}

}  // namespace

// Shared by the other translation units of the library.
namespace pt_internal {
int set_error(int status, const char *where, const char *msg)
{
    snprintf(g_last_error, sizeof(g_last_error), "%s: %s", where, msg);
    return status;
}
}  // namespace pt_internal

namespace {

int check_launch(const char *where)
{
    cudaError_t e = cudaGetLastError();
    if (e != cudaSuccess) return set_cuda_error(e, where);
    return PT_OK;
}

size_t align256(size_t x) { return (x + 255) & ~(size_t)255; }

// ---------------------------------------------------------------------------
// Set-up kernel
// ---------------------------------------------------------------------------
struct SetupArgs {
    const double *t;
    int n_t;
    float2 *tsplit;
    const double *t0, *P;
    const float *a, *inc, *e, *w, *k;
    int n_v, n_b, k_per_band, n_geom;
    GeomRec *rec;
    float half_exp;
    int n_gblocks;
};

__device__ void make_geom(const SetupArgs &s, int g, GeomRec *out)
{
    int v = s.k_per_band ? g / s.n_b : g;
    pt::make_geom_rec(s.t0[v], s.P[v], s.a[v], s.inc[v], s.e != nullptr, s.e ? s.e[v] : 0.0f,
                      s.w ? s.w[v] : 0.0f, s.k[g], s.half_exp, out);
}

__global__ void setup_kernel(SetupArgs s)
{
    pt::chain_begin();
    if ((int)blockIdx.x < s.n_gblocks) {
        int g = blockIdx.x * blockDim.x + threadIdx.x;
        if (g < s.n_geom) make_geom(s, g, &s.rec[g]);
    } else {
        int i = (blockIdx.x - s.n_gblocks) * blockDim.x + threadIdx.x;
        if (i < s.n_t) {
            double t = s.t[i];
            float h = (float)t;
            s.tsplit[i] = make_float2(h, (float)(t - (double)h));
        }
    }
}

// ---------------------------------------------------------------------------
// Preparation of a light-curve call from row tables (pt_rows.cuh): the
// geometry records, the time split and the Mandel-Agol rows, in one launch
// (the records' FP64 latency and the tables' elliptic integrals run side by
// side).  Row CTAs take ROW_GEOM geometries: one node of a geometry's table
// per thread (the region inside the disk, in double-float arithmetic, on the
// first warps), then per row one coefficient per thread.
// ---------------------------------------------------------------------------
constexpr int ROW_GEOM = 2;
constexpr int ROW_THREADS = ROW_GEOM * pt::MT_NODES;

struct RowPrep {
    SetupArgs s;
    int n_tblocks;
    float *rows;      // [n_geom][nr][row_len]
    int row_len, nr, terms, n_bpg;
    const float *ld;
    float *wts;       // terms: the passbands' weights [n_geom n_bpg][3] (R_GIM: in gim)
    // R_INTERP: the caller's table
    const float4 *mtab;
    int mn_k, mn_z;
    float mk_lo, mk_hi, minv_dk;
    // R_GIM: the T_{n,j} and the passbands' weights (pt_gim.cuh)
    gim::Table gim;
};

// weights of row r of a geometry: a passband's depth, or one of the terms
__device__ __forceinline__ float3 row_weights(const RowPrep &P, int g, int r)
{
    if (P.terms) return make_float3(r == 0 ? 1.0f : 0.0f, r == 1 ? 1.0f : 0.0f, r == 2 ? 1.0f : 0.0f);
    float3 w;
    const float *ld = P.ld + 2 * ((size_t)g * P.n_bpg + r);
    pt::ma_weights(ld[0], ld[1], &w.x, &w.y, &w.z);
    return w;
}

template <int MODEL>
__global__ void __launch_bounds__(ROW_THREADS) row_prep_kernel(RowPrep P)
{
    pt::chain_begin();
    __shared__ float3 sF[ROW_GEOM][pt::MT_N * pt::MT_Q];
    const int tid = threadIdx.x;
    const SetupArgs &s = P.s;
    int blk = blockIdx.x;
    if (blk < s.n_gblocks) {
        // one warp per CTA: the records' FP64 operations share one slow pipe per SM
        const int g = blk * 32 + tid;
        if (tid < 32 && g < s.n_geom) make_geom(s, g, &s.rec[g]);
        if (P.wts && tid >= 32) {
            // beside them, the weights of the geometries' passbands
            const long long n = (long long)min(32, s.n_geom - blk * 32) * P.n_bpg;
            for (long long i = tid - 32; i < n; i += ROW_THREADS - 32) {
                const size_t row = (size_t)blk * 32 * P.n_bpg + i;
                float *w = P.wts + 3 * row;
                pt::ma_weights(P.ld[2 * row], P.ld[2 * row + 1], w, w + 1, w + 2);
            }
        }
        return;
    }
    blk -= s.n_gblocks;
    if (blk < P.n_tblocks) {
        const int i = blk * ROW_THREADS + tid;
        if (i < s.n_t) {
            const double t = s.t[i];
            const float h = (float)t;
            s.tsplit[i] = make_float2(h, (float)(t - (double)h));
        }
        return;
    }
    blk -= P.n_tblocks;
    if (MODEL == rows::R_INTERP) {
        // each row: the table's nodes at the geometry's k, combined
        const long long at = (long long)blk * ROW_THREADS + tid;
        const long long row = at / P.row_len;
        const int j = (int)(at - row * P.row_len);
        if (row >= (long long)s.n_geom * P.nr) return;
        const int g = (int)(row / P.nr), r = (int)(row - (long long)g * P.nr);
        float v = 0.0f;
        if (j < P.mn_z) {
            const float fk = (fminf(fmaxf(s.k[g], P.mk_lo), P.mk_hi) - P.mk_lo) * P.minv_dk;
            const int ik = min((int)fk, P.mn_k - 2);
            const float wk = fk - (float)ik;
            const float4 a = __ldg(P.mtab + (size_t)ik * P.mn_z + j), b = __ldg(P.mtab + (size_t)(ik + 1) * P.mn_z + j);
            const float3 w = row_weights(P, g, r);
            v = w.x * fmaf(wk, b.x - a.x, a.x) + w.y * fmaf(wk, b.y - a.y, a.y) + w.z * fmaf(wk, b.z - a.z, a.z);
        }
        P.rows[at] = v;
        return;
    }
    if (MODEL == rows::R_GIM) {
        gim::table_cta(P.gim, s.k, s.n_geom, P.n_bpg, P.ld, blk % P.gim.NP1, blk / P.gim.NP1);
        return;
    }
    const int first = blk * ROW_GEOM;
    constexpr int NODES_A = pt::MT_NA * pt::MT_Q, NODES_L = pt::MT_NODES - NODES_A;
    {
        const bool in_a = tid < ROW_GEOM * NODES_A;
        const int u = in_a ? tid : tid - ROW_GEOM * NODES_A;
        const int gl = in_a ? u / NODES_A : u / NODES_L;
        const int node = in_a ? u - gl * NODES_A : NODES_A + u - gl * NODES_L;
        if (first + gl < s.n_geom) {
            const float p = s.k[first + gl];
            if (pt::mt_valid(p)) {   // the others take the exact terms per point
                float3 f;
                pt::mt_node(p, node / pt::MT_Q, node % pt::MT_Q, &f.x, &f.y, &f.z);
                sF[gl][node] = f;
            }
        }
    }
    __syncthreads();
    {
        const int c = tid / (ROW_GEOM * pt::MT_N), u = tid - c * (ROW_GEOM * pt::MT_N);
        const int gl = u / pt::MT_N, i = u - gl * pt::MT_N, g = first + gl;
        if (g < s.n_geom && pt::mt_valid(s.k[g])) {
            for (int r = 0; r < P.nr; ++r) {
                const float3 w = row_weights(P, g, r);
                float f[pt::MT_Q];
#pragma unroll
                for (int q = 0; q < pt::MT_Q; ++q) {
                    const float3 v = sF[gl][i * pt::MT_Q + q];
                    f[q] = w.x * v.x + w.y * v.y + w.z * v.z;
                }
                P.rows[((size_t)g * P.nr + r) * P.row_len + 8 * i + c] = pt::mt_coef(i, c, f);
            }
        }
    }
}

// ---------------------------------------------------------------------------
// Shared pieces of the light-curve kernels
// ---------------------------------------------------------------------------
struct LcArgs {
    SetupArgs set;       // the geometries' inputs, for blocks that form their own records
    const float2 *tsplit;
    int n_t;
    const GeomRec *rec;
    int n_geom;
    const float *ld;     // [rows][2]
    int n_b, k_per_band, n_bpg;
    int band0;           // passband of the launch's first geometry, when k is per passband
    int n_ss;
    float t_exp;
    int max_iter;
    const float *y, *wt;
    float *flux;
    float *ssr_part;     // [rows][n_tiles]
    int n_tiles;
    int *n_bad;
    // interpolated Mandel-Agol terms (Sec. 2.2.3), when the kernel uses them
    const float4 *mtab;  // [n_k][n_z]: (lambda_e, lambda_d + 2/3 Theta, eta_d, 0)
    int mn_k, mn_z;
    float mk_lo, mk_hi, minv_dk, minv_dz;
};

__device__ __forceinline__ float block_sum(float v, float *sred)
{
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) v += __shfl_xor_sync(0xffffffffu, v, o);
    int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
    __syncthreads();
    if (lane == 0) sred[warp] = v;
    __syncthreads();
    float tot = 0.0f;
    if (threadIdx.x == 0) {
        for (int i = 0; i < (int)(blockDim.x >> 5); ++i) tot += sred[i];
    }
    return tot;
}

// Phase A: window test + compaction.  OWN: the block forms its geometries'
// records and splits its times itself, else they come from setup_kernel.
template <int VT, bool OWN>
__device__ __forceinline__ void phase_a(const LcArgs &A, GeomRec *srec, float (*sdt)[TT],
                                        unsigned char (*sflag)[TT], unsigned short *squeue, int *sqn)
{
    int tl = threadIdx.x;
    int t = blockIdx.x * TT + tl;
    bool tv = t < A.n_t;
    float2 ts = make_float2(0.0f, 0.0f);
    if constexpr (OWN) {
        if (tv) {
            const double x = A.set.t[t];
            ts.x = (float)x;
            ts.y = (float)(x - (double)ts.x);
        }
        if (tl < VT && (int)blockIdx.y * VT + tl < A.n_geom) make_geom(A.set, blockIdx.y * VT + tl, &srec[tl]);
    } else {
        if (tv) ts = A.tsplit[t];
        // stage the geometry records (6 float4 each)
        for (int i = tl; i < VT * 6; i += TT) {
            int vl = i / 6, c = i % 6;
            int g = blockIdx.y * VT + vl;
            if (g < A.n_geom)
                reinterpret_cast<float4 *>(&srec[vl])[c] = reinterpret_cast<const float4 *>(&A.rec[g])[c];
        }
    }
    if (tl == 0) *sqn = 0;
    __syncthreads();
#pragma unroll 1
    for (int vl = 0; vl < VT; ++vl) {
        int g = blockIdx.y * VT + vl;
        bool valid = tv && g < A.n_geom;
        float dt = 0.0f;
        bool inw = false;
        if (valid && pt::maybe_in_window(ts.x, srec[vl])) {
            dt = pt::reduce_time(ts.x, ts.y, srec[vl]);
            inw = (dt >= srec[vl].win_lo) && (dt <= srec[vl].win_hi);
        }
        sdt[vl][tl] = dt;
        sflag[vl][tl] = inw ? 1 : 0;
        if (__any_sync(0xffffffffu, inw)) {   // warp-uniform
            int slot = pt::warp_append(sqn, inw);
            if (inw) squeue[slot] = (unsigned short)(vl * TT + tl);
        }
    }
    __syncthreads();
}

__device__ __forceinline__ float ss_offset(float t_exp, int s, float inv_nss)
{
    return t_exp * (((float)s + 0.5f) * inv_nss - 0.5f);   // inv_nss = 1 / n_ss
}

// ---------------------------------------------------------------------------
// Mandel-Agol light curves
// ---------------------------------------------------------------------------
template <bool INTERP, bool OWN>
__global__ void __launch_bounds__(TT) ma_lc_kernel(LcArgs A)
{
    pt::chain_begin();
    __shared__ GeomRec srec[VT_MA];
    __shared__ float sdt[VT_MA][TT];
    __shared__ unsigned char sflag[VT_MA][TT];
    __shared__ unsigned short squeue[VT_MA * TT];
    __shared__ float sacc[3][VT_MA][TT];
    __shared__ float sub[3][TT];
    __shared__ float sred[TT / 32];
    __shared__ int sqn, sbad;

    if (threadIdx.x == 0) sbad = 0;
    phase_a<VT_MA, OWN>(A, srec, sdt, sflag, squeue, &sqn);
    const int tl = threadIdx.x;
    const int qn = sqn;
    const int nss = A.n_ss;
    const int G = TT / nss;
    const int units = G * nss;
    const float inv_nss = 1.0f / (float)nss;

    // Phase B: (pair, supersample) units
#pragma unroll 1
    for (int base = 0; base < qn; base += G) {
        int iu = tl / nss;
        int s = tl - iu * nss;
        int item = base + iu;
        float le = 0.0f, ld = 0.0f, ed = 0.0f;
        if (tl < units && item < qn) {
            int code = squeue[item];
            int vl = code / TT, ti = code % TT;
            const GeomRec &r = srec[vl];
            float dts = sdt[vl][ti] + ss_offset(A.t_exp, s, inv_nss);
            bool bad = false;
            float z = pt::orbit_z<true>(r, dts, A.max_iter, &bad);
            if (bad) atomicAdd(&sbad, 1);
            if constexpr (INTERP)
                pt::ma_interp(A.mtab, A.mn_k, A.mn_z, A.mk_lo, A.mk_hi, A.minv_dk, A.minv_dz, r.k, z, &le, &ld, &ed);
            else
                pt::ma_terms(r.k, z, &le, &ld, &ed);
        }
        sub[0][tl] = le;
        sub[1][tl] = ld;
        sub[2][tl] = ed;
        __syncthreads();
        if (tl < G && base + tl < qn) {
            float s0 = 0.0f, s1 = 0.0f, s2 = 0.0f;
            for (int j = 0; j < nss; ++j) {
                s0 += sub[0][tl * nss + j];
                s1 += sub[1][tl * nss + j];
                s2 += sub[2][tl * nss + j];
            }
            int code = squeue[base + tl];
            int vl = code / TT, ti = code % TT;
            sacc[0][vl][ti] = s0;
            sacc[1][vl][ti] = s1;
            sacc[2][vl][ti] = s2;
        }
        __syncthreads();
    }

    // Phase C: limb darkening per passband, stores and residuals
    const int t = blockIdx.x * TT + tl;
    const bool tv = t < A.n_t;
#pragma unroll 1
    for (int vl = 0; vl < VT_MA; ++vl) {
        int g = blockIdx.y * VT_MA + vl;
        if (g >= A.n_geom) break;
        bool inw = tv && sflag[vl][tl];
        float l0 = 0.0f, l1 = 0.0f, l2 = 0.0f;
        if (inw) {
            l0 = sacc[0][vl][tl] * inv_nss;
            l1 = sacc[1][vl][tl] * inv_nss;
            l2 = sacc[2][vl][tl] * inv_nss;
        }
#pragma unroll 1
        for (int bb = 0; bb < A.n_bpg; ++bb) {
            int row = g * A.n_bpg + bb;
            float we, wd, wn;
            pt::ma_weights(A.ld[row * 2], A.ld[row * 2 + 1], &we, &wd, &wn);
            float f = inw ? 1.0f - (we * l0 + wd * l1 + wn * l2) : 1.0f;
            if (A.flux && tv) A.flux[(size_t)row * A.n_t + t] = f;
            if (A.ssr_part) {
                int band = A.k_per_band ? (A.band0 + g) % A.n_b : bb;
                float val = 0.0f;
                if (tv) {
                    float r = A.y[(size_t)band * A.n_t + t] - f;
                    val = (A.wt ? A.wt[(size_t)band * A.n_t + t] : 1.0f) * r * r;
                }
                float tot = block_sum(val, sred);
                if (tl == 0) A.ssr_part[(size_t)row * A.n_tiles + blockIdx.x] = tot;
            }
        }
    }
    if (tl == 0 && sbad && A.n_bad) atomicAdd(A.n_bad, sbad);
}

// One warp per row.  The sum's rounding errors are carried along (two-sums), so
// that the partials' own rounding is all that is left; an infinite sum, whose
// errors are NaN, is itself.
__global__ void ssr_reduce_kernel(const float *part, int rows, int n_part, float *ssr)
{
    pt::chain_begin();
    int warp = (blockIdx.x * blockDim.x + threadIdx.x) >> 5;
    int lane = threadIdx.x & 31;
    if (warp >= rows) return;
    float h = 0.0f, l = 0.0f;
    auto add = [&](float v, float vl) {
        const float s = h + v, bb = s - h;
        l = (l + vl) + ((h - (s - bb)) + (v - bb));
        h = s;
    };
    for (int i = lane; i < n_part; i += 32) add(part[(size_t)warp * n_part + i], 0.0f);
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) add(__shfl_xor_sync(0xffffffffu, h, o), __shfl_xor_sync(0xffffffffu, l, o));
    const float s = h + l;
    if (lane == 0) ssr[warp] = s == s ? s : h;
}

// ssr[row] = sum_t wt (y - flux)^2 over one flux row, in a fixed order;
// row r observes passband r % n_b (rows are geometry-major, band-minor).
// ssr_part_kernel: one CTA per (row, chunk of SSR_CHUNK times); every thread
// loads its SSR_PER values before adding them, so a CTA keeps its whole chunk
// in flight (a loop that waits on each load in turn is latency-bound), then a
// fixed-order block sum.  ssr_reduce_kernel adds a row's chunk sums.
constexpr int SSR_PER = 16;
constexpr int SSR_CHUNK = 256 * SSR_PER;

int ssr_chunks(int n_t) { return (n_t + SSR_CHUNK - 1) / SSR_CHUNK; }

__global__ void __launch_bounds__(256) ssr_part_kernel(const float *flux, const float *y, const float *wt, int n_t,
                                                      int n_b, float *part)
{
    pt::chain_begin();
    __shared__ float sred[8];
    const size_t row = blockIdx.x;
    const int band = (int)(row % n_b);
    const float *f = flux + row * n_t;
    const float *yb = y + (size_t)band * n_t;
    const float *wb = wt ? wt + (size_t)band * n_t : nullptr;
    const int t0 = blockIdx.y * SSR_CHUNK + threadIdx.x;
    float fv[SSR_PER], yv[SSR_PER], wv[SSR_PER];
#pragma unroll
    for (int j = 0; j < SSR_PER; ++j) {
        const int t = t0 + j * 256;
        const bool ok = t < n_t;
        fv[j] = ok ? f[t] : 0.0f;
        yv[j] = ok ? yb[t] : 0.0f;
        wv[j] = ok ? (wb ? wb[t] : 1.0f) : 0.0f;
    }
    float acc = 0.0f;
#pragma unroll
    for (int j = 0; j < SSR_PER; ++j) {
        const float r = yv[j] - fv[j];
        acc = fmaf(wv[j], r * r, acc);
    }
    const float tot = block_sum(acc, sred);
    if (threadIdx.x == 0) part[row * gridDim.y + blockIdx.y] = tot;
}

int launch_ssr_rows(const float *flux, const float *y, const float *wt, int n_t, int n_b, size_t rows, float *part,
                    float *ssr, cudaStream_t s)
{
    const int nc = ssr_chunks(n_t);
    pt::launch_chained(ssr_part_kernel, dim3((unsigned)rows, (unsigned)nc), 256, 0, s, flux, y, wt, n_t, n_b, part);
    int st = check_launch("ssr_part_kernel");
    if (st) return st;
    pt::launch_chained(ssr_reduce_kernel, (unsigned)((rows * 32 + 255) / 256), 256, 0, s, part, (int)rows, nc, ssr);
    return check_launch("ssr_reduce_kernel");
}

// Interpolation-table nodes: the exact FP32 terms at (k_i, z_j), positions
// formed in FP64 and rounded once.
__global__ void ma_table_kernel(double k_lo, double k_hi, int n_k, int n_z, float4 *tab)
{
    size_t id = (size_t)blockIdx.x * blockDim.x + threadIdx.x;
    if (id >= (size_t)n_k * n_z) return;
    int i = (int)(id / n_z), j = (int)(id % n_z);
    float k = (float)(k_lo + i * (k_hi - k_lo) / (n_k - 1));
    float z = (float)(j * (1.0 + k_hi) / (n_z - 1));
    float le, ld, ed;
    pt::ma_terms(k, z, &le, &ld, &ed);
    tab[id] = make_float4(le, ld, ed, 0.0f);
}

__global__ void ma_terms_interp_kernel(const float4 *tab, int n_k, int n_z, float k_lo, float k_hi, float inv_dk,
                                       float inv_dz, const float *k, const float *z, size_t n, float *le, float *ld,
                                       float *ed)
{
    size_t i = (size_t)blockIdx.x * blockDim.x + threadIdx.x;
    if (i >= n) return;
    float a, b, c;
    pt::ma_interp(tab, n_k, n_z, k_lo, k_hi, inv_dk, inv_dz, k[i], z[i], &a, &b, &c);
    if (le) le[i] = a;
    if (ld) ld[i] = b;
    if (ed) ed[i] = c;
}

// ---------------------------------------------------------------------------
// Pointwise kernels
// ---------------------------------------------------------------------------
__global__ void ma_terms_kernel(const float *k, const float *z, size_t n, float *le, float *ld, float *ed)
{
    size_t i = (size_t)blockIdx.x * blockDim.x + threadIdx.x;
    if (i >= n) return;
    float a, b, c;
    pt::ma_terms(k[i], fabsf(z[i]), &a, &b, &c);
    if (le) le[i] = a;
    if (ld) ld[i] = b;
    if (ed) ed[i] = c;
}

__global__ void gim_alpha_kernel(const float *kk, const float *zz, size_t n, int NP1, int n_j,
                                 const float4 *coef, const double *A, const double *recb, float *alpha)
{
    size_t i = (size_t)blockIdx.x * blockDim.x + threadIdx.x;
    if (i >= n) return;
    float k = kk[i], z = fabsf(zz[i]);
    float *out = alpha + i * NP1;
    if (!(z < 1.0f + k) || !(k > 0.0f)) {
        for (int m = 0; m < NP1; ++m) out[m] = 0.0f;
        return;
    }
    float c = z / (1.0f + k);
    float x = c * c;
    float q = sqrtf((1.0f - c) * (1.0f + c));
    float bb = k / (1.0f + k);
    double xb = 1.0 - (double)k / (1.0 + (double)k);
    for (int n = 0; n < NP1; ++n) {
        const double *An = A + (size_t)n * n_j;
        const double *rb = recb + (size_t)n * n_j * 3;
        const float4 *cf = coef + (size_t)n * n_j;
        double hp = 0.0, hc = 1.0;
        float g = 1.0f, gp = 0.0f;
        float sum = (float)An[0];
        for (int j = 0; j + 1 < n_j; ++j) {
            double hn = (rb[3 * j] + rb[3 * j + 1] * xb) * hc + rb[3 * j + 2] * hp;
            hp = hc;
            hc = hn;
            float tj = (float)(An[j + 1] * hc * hc);
            float4 cc = cf[j];
            float gn = fmaf(fmaf(cc.y, x, cc.x), g, cc.z * gp);
            gp = g;
            g = gn;
            sum = fmaf(tj, gn, sum);
        }
        float q2 = q * q, pw = q2 * q2;
        for (int m = 0; m < n; ++m) pw *= q;
        out[n] = bb * bb * pw * sum;
    }
}

// ---------------------------------------------------------------------------
// z kernels (standalone)
// ---------------------------------------------------------------------------
__global__ void z_circ_kernel(const double *t, int n_t, const double *t0, const double *P, const float *a,
                              const float *inc, int n_ss, double t_exp, float *z)
{
    int v = blockIdx.y;
    int idx = blockIdx.x * blockDim.x + threadIdx.x;
    if (idx >= n_t * n_ss) return;
    int i = idx / n_ss, s = idx - i * n_ss;
    double tt = t[i] + t_exp * ((s + 0.5) / n_ss - 0.5);
    double x = (tt - t0[v]) * (1.0 / P[v]);
    x -= rint(x);
    float ph = (float)(2.0 * PI_D * x);
    float sp, cp;
    sincosf(ph, &sp, &cp);
    float out = PT_ZBEHIND;
    if (cp > 0.0f) {
        float ci = (float)cos((double)inc[v]) * cp;
        out = a[v] * sqrtf(fmaf(sp, sp, ci * ci));
    }
    z[(size_t)v * n_t * n_ss + idx] = out;
}

__global__ void z_ecc_kernel(const double *t, int n_t, const double *t0, const double *P, const float *a,
                             const float *inc, const float *e, const float *w, int n_ss, double t_exp,
                             int max_iter, double tol, float *z, int *n_bad)
{
    __shared__ double sMtr;
    int v = blockIdx.y;
    double ev = e[v], wv = w[v];
    if (threadIdx.x == 0) {
        double ftr = 0.5 * PI_D - wv;
        double Etr = 2.0 * atan2(sqrt(1.0 - ev) * sin(0.5 * ftr), sqrt(1.0 + ev) * cos(0.5 * ftr));
        sMtr = Etr - ev * sin(Etr);
    }
    __syncthreads();
    int idx = blockIdx.x * blockDim.x + threadIdx.x;
    if (idx >= n_t * n_ss) return;
    int i = idx / n_ss, s = idx - i * n_ss;
    double tt = t[i] + t_exp * ((s + 0.5) / n_ss - 0.5);
    double x = (tt - t0[v]) / P[v];
    x -= floor(x);
    double M = sMtr + 2.0 * PI_D * x;
    M -= 2.0 * PI_D * floor(M / (2.0 * PI_D));
    // FP64 Newton iteration on E - e sin E = M, start E = M (e < 0.8) or pi
    double E = (ev < 0.8) ? M : PI_D;
    bool conv = false;
    for (int it = 0; it < max_iter; ++it) {
        double sE, cE;
        sincos(E, &sE, &cE);
        double d = (E - ev * sE - M) / (1.0 - ev * cE);
        E -= d;
        if (fabs(d) < tol) {
            conv = true;
            break;
        }
    }
    if (!conv && n_bad) atomicAdd(n_bad, 1);
    double f = 2.0 * atan2(sqrt(1.0 + ev) * sin(0.5 * E), sqrt(1.0 - ev) * cos(0.5 * E));
    double r = a[v] * (1.0 - ev * cos(E));
    double sw, cw;
    sincos(wv + f, &sw, &cw);
    float out = PT_ZBEHIND;
    if (sw > 0.0) {
        double ci = cos((double)inc[v]);
        out = (float)(r * sqrt(cw * cw + sw * sw * ci * ci));
    }
    z[(size_t)v * n_t * n_ss + idx] = out;
}

// Exposure time: finite and non-negative (the supersamples of Sec. 3.2 span it).
bool exposure_ok(double t_exp) { return t_exp >= 0.0 && t_exp < 1.0e30; }

int check_orbit(const pt_orbit *orb, bool need_ecc)
{
    if (!orb || orb->n_v < 0) return PT_ERR_ARG;
    if (orb->n_v == 0) return PT_OK;
    if (!orb->t0 || !orb->P || !orb->a || !orb->inc) return PT_ERR_ARG;
    if ((orb->e == nullptr) != (orb->w == nullptr)) return PT_ERR_ARG;
    if (need_ecc && !orb->e) return PT_ERR_ARG;
    return PT_OK;
}

// The tile kernel: records, time split, per-tile residual partials.
struct WorkLayout {
    size_t rec, tsplit, part, total;
};

WorkLayout work_layout(int n_t, int n_v, int n_b, int k_per_band)
{
    int n_geom = k_per_band ? n_v * n_b : n_v;
    int n_tiles = (n_t + TT - 1) / TT;
    WorkLayout L;
    size_t off = 0;
    L.rec = off;
    off += align256((size_t)n_geom * sizeof(GeomRec));
    L.tsplit = off;
    off += align256((size_t)n_t * sizeof(float2));
    L.part = off;
    off += align256((size_t)n_v * n_b * n_tiles * sizeof(float));
    L.total = off;
    return L;
}

// Light curves from row tables: records, time split, rows, residual partials
// and, when many passbands share a geometry and only residuals are wanted, a
// flux scratch.
struct RowLayout {
    size_t rec, tsplit, rows, part, wts, fscr, total;
};

// rows of a geometry: one per passband, or the model's terms when more
// passbands share it
bool row_terms(int n_bpg) { return n_bpg > rows::MAX_BAND_ROWS; }
int rows_per_geom(int n_bpg, int n_terms) { return row_terms(n_bpg) ? n_terms : n_bpg; }

RowLayout row_layout(int n_t, int n_v, int n_b, int k_per_band, int n_terms, size_t row_len)
{
    const size_t n_geom = k_per_band ? (size_t)n_v * n_b : (size_t)n_v;
    const int n_bpg = k_per_band ? 1 : n_b;
    const size_t n_tiles = ((size_t)n_t + TT - 1) / TT;
    RowLayout L;
    size_t off = 0;
    L.rec = off;
    off += align256(n_geom * sizeof(GeomRec));
    L.tsplit = off;
    off += align256((size_t)n_t * sizeof(float2));
    L.rows = off;
    off += align256(n_geom * rows_per_geom(n_bpg, n_terms) * row_len * sizeof(float));
    L.part = off;   // per tile, or per chunk of a flux row
    off += align256((size_t)n_v * n_b * n_tiles * sizeof(float));
    L.wts = off;    // Mandel-Agol (the Gimenez weights follow the layout)
    if (row_terms(n_bpg)) off += align256((size_t)n_v * n_b * 3 * sizeof(float));
    L.fscr = off;
    if (row_terms(n_bpg)) off += align256((size_t)n_v * n_b * n_t * sizeof(float));
    L.total = off;
    return L;
}

// Tables pay from this many points (times x supersamples) per geometry: a
// Mandel-Agol row costs 144 evaluations of the terms, and only the in-window
// points read it.
constexpr long long ROWS_MIN_POINTS = 512;

// Dynamic shared memory: launches up to the default limit (48 KB, less room for a
// kernel's static arrays) need no opt-in.  The row kernel's and the preparation's
// size varies from call to call, so they opt in to one limit that covers all
// their calls (pt::allow_smem): the row kernel's 16 KB of lists, 96 KB of rows and 32 KB
// of residuals, the preparation's 2 x 16 chains of 512 steps (134 KB).
constexpr int DEFAULT_SMEM = 40 * 1024, VARIABLE_SMEM_MAX = 160 * 1024;

// Tile of the row kernel: geometries x blocks of 256 times.  As many
// geometries as 48 KB of rows hold (so that four CTAs fit an SM), the rest of
// the 32 bits in blocks of times (which spreads the staging of the rows over
// more pairs); then smaller tiles until there are four CTAs per SM.
int launch_rows(int model, rows::Args &A, int n_sm, cudaStream_t s)
{
    const size_t row_bytes = (size_t)A.nr * A.row_len * sizeof(float);
    const bool staged = row_bytes <= 96 * 1024;
    // residuals keep a value per pair and passband: fewer pairs per tile then
    const int bits = A.ssr_part ? (A.nr <= 2 ? 16 : A.nr <= 4 ? 8 : 4) : rows::MAX_BITS;
    int vt = 1, log_kt = 0;
    while (vt < bits && vt < A.n_geom && (!staged || 2 * vt * row_bytes <= 48 * 1024)) vt *= 2;
    while ((vt << log_kt) < bits && (rows::TB << log_kt) < A.n_t) ++log_kt;
    auto ctas = [&](int v, int lk) {
        return ((long long)A.n_t + (rows::TB << lk) - 1) / (rows::TB << lk) * ((A.n_geom + v - 1) / v);
    };
    while (log_kt > 0 && ctas(vt, log_kt) < 4LL * n_sm) --log_kt;
    while (vt > 1 && ctas(vt, log_kt) < 4LL * n_sm) vt /= 2;
    A.log_vt = 0;
    while ((1 << A.log_vt) < vt) ++A.log_vt;
    A.log_kt = log_kt;
    A.flux_vec = A.flux && A.n_t % 4 == 0 && ((uintptr_t)A.flux & 15u) == 0;
    A.n_tiles = (A.n_t + (rows::TB << log_kt) - 1) / (rows::TB << log_kt);
    A.n_blk = (A.n_t + rows::TB - 1) / rows::TB;
    const int smem = rows::smem_layout(vt, log_kt, A.nr, A.row_len, staged, A.ssr_part ? A.nr : 0).total;
    void (*fn)(rows::Args) = nullptr;
#define PT_ROWS_FN(M)                                                                                               \
    fn = A.nr == 1 ? rows::lc_rows_kernel<M, 1, true>                                                               \
         : A.nr <= 4 ? rows::lc_rows_kernel<M, 4, true> : rows::lc_rows_kernel<M, 9, true>
    switch (model) {
    case rows::R_MA: PT_ROWS_FN(rows::R_MA); break;
    case rows::R_GIM: PT_ROWS_FN(rows::R_GIM); break;
    case rows::R_ZI: PT_ROWS_FN(rows::R_ZI); break;
    default: PT_ROWS_FN(rows::R_INTERP); break;
    }
#undef PT_ROWS_FN
    // (the other models' rows are at most 64 KB)
    if (!staged) fn = model == rows::R_GIM ? rows::lc_rows_kernel<rows::R_GIM, 9, false> : rows::lc_rows_kernel<rows::R_ZI, 9, false>;
    if (smem > DEFAULT_SMEM) {
        if (smem > VARIABLE_SMEM_MAX) return pt_internal::set_error(PT_ERR_ARG, "lc_rows_kernel", "tile too large");
        cudaError_t e = pt::allow_smem(fn, VARIABLE_SMEM_MAX);
        if (e != cudaSuccess) return set_cuda_error(e, "lc_rows_kernel smem attribute");
    }
    // geometries along x, time tiles along y, in as many launches as y takes
    for (A.tile0 = 0; A.tile0 < A.n_tiles; A.tile0 += 65535) {
        const dim3 grid((unsigned)((A.n_geom + vt - 1) / vt), (unsigned)std::min(65535, A.n_tiles - A.tile0));
        pt::launch_chained(fn, grid, rows::TB, (size_t)smem, s, A);
        const int st = check_launch("lc_rows_kernel");
        if (st) return st;
    }
    return PT_OK;
}

int sm_count(int *n_sm)
{
    int dev = 0;
    cudaError_t e = cudaGetDevice(&dev);
    if (e == cudaSuccess) e = cudaDeviceGetAttribute(n_sm, cudaDevAttrMultiProcessorCount, dev);
    return e == cudaSuccess ? PT_OK : set_cuda_error(e, "SM count");
}

// pt_ma_quad and pt_ma_quad_interp run from row tables, except for a few
// geometries (there the tile kernel's one launch, without tables, is faster) and for too few points per geometry.  The tile kernel also serves the
// allocation-free variant, whose scratch must stay small.
constexpr int MA_TILE_MAX_GEOM = 4;

// Up to about four blocks per multiprocessor the tile kernel's blocks form
// their geometries' records themselves: the FP64 chain of a record takes as
// long in each block as once in a launch before them, and that launch is
// saved (one geometry x 1,000 times 10.0 -> 9.2 us of GPU time and 23 -> 19 us
// with the host; 500 blocks 26, either way, 1,250 blocks 42.3 -> 45.9).
constexpr long long MA_OWN_MAX_BLOCKS = 608;

bool ma_use_rows(int n_t, int n_v, int n_b, int k_per_band, int n_ss)
{
    const long long n_geom = k_per_band ? (long long)n_v * n_b : n_v;
    return n_geom > MA_TILE_MAX_GEOM && (long long)n_t * n_ss >= ROWS_MIN_POINTS;
}

// Rows of a caller's table: staged whole, so short ones only, and no longer
// than a light curve (a row is built node by node).
constexpr int INTERP_ROW_MAX = 2048;
size_t interp_row_len(int n_z) { return ((size_t)n_z + 3) & ~(size_t)3; }
size_t row_len_max(int n_t)
{
    const size_t m = interp_row_len(n_t < INTERP_ROW_MAX ? n_t : INTERP_ROW_MAX);
    return m > (size_t)pt::MT_ROW ? m : (size_t)pt::MT_ROW;
}

// Building a row and staging it costs its length.  Where many geometries fill the
// chip with it, a light curve has to read a long row often, from four points
// (times x supersamples) per node on (50,000 vectors x 3,000 times, half of them
// in transit, from 1,024 nodes: 1,572 us against 1,294 by the tile kernel; from 256
// nodes 1,061 against 1,265, and x 600 times 254 against 304).  Up to 8 M nodes in
// all, the rows' cost is hidden (5,000 vectors x 3,000 times from 1,024 nodes: 120
// us against 127).
bool interp_use_rows(int n_t, int n_v, int n_b, int k_per_band, int n_ss, size_t row_len)
{
    const size_t n_geom = k_per_band ? (size_t)n_v * n_b : (size_t)n_v;
    return row_len <= row_len_max(n_t) &&
           (row_len <= 512 || 4 * row_len <= (size_t)n_t * n_ss || n_geom * row_len <= (size_t)8 << 20);
}

}  // namespace

struct pt_ma_table_s {
    float k_lo, k_hi, inv_dk, inv_dz;
    int n_k, n_z;
    float4 *d_tab;   // [n_k][n_z]: (lambda_e, lambda_d + 2/3 Theta, eta_d, 0)
};

// The table's device view, for the batched path (pt_batch.cu).
namespace pt_internal {
bool ma_table_view(pt_ma_table t, const float4 **tab, int *n_k, int *n_z, float *k_lo, float *k_hi, float *inv_dk,
                   float *inv_dz)
{
    if (!t || !t->d_tab) return false;
    *tab = t->d_tab;
    *n_k = t->n_k;
    *n_z = t->n_z;
    *k_lo = t->k_lo;
    *k_hi = t->k_hi;
    *inv_dk = t->inv_dk;
    *inv_dz = t->inv_dz;
    return true;
}
}  // namespace pt_internal

struct pt_gim_plan_s {
    int N, n_j;
    void *d_mem;      // the one allocation that holds the tables below
    float4 *d_coef;   // [N+1][n_j]: recursion of G_j(nu+2, 1; x), FP32
    const double *d_A;      // [N+1][n_j]: A_{n,j}, FP64
    const double *d_recb;   // [N+1][n_j][3]: recursion of G_j(nu+2, nu+1; x), FP64
    float2 *d_dA;     // the same A_{n,j} and recursion as double-float pairs
    float2 *d_drb;
    float *d_B;       // [(N+1) n_j][8 n_int]: piecewise polynomials of the series' functions (pt_gim.cuh)
    int n_int;
    cudaEvent_t ev0, ev1;   // recorded around the evaluation kernel when set (profiling)
};

namespace {

// Three-term recursion of G_j(p,q;x) = 2F1(-j, p+j; q; x) in the form of
// Sec. 2.1.4, G_{j+1} = ((j1 + j2 x) G_j + j3 G_{j-1}) / j4, written as
// G_{j+1} = (r1 + r2 x) G_j + r3 G_{j-1}.  Entry 0 produces
// G_1 = 1 - (p+1) x / q from G_0 = 1.  For j >= 1, with s = 2j + p (from the
// standard recurrence of the Jacobi polynomial P_j^{(q-1, p-q)}(1 - 2x),
// rescaled by j!/(q)_j):
//   j1 = s [(s+1)(s-1) + (q-1)^2 - (p-q)^2],  j2 = -2 s (s+1)(s-1),
//   j3 = -2 j (j+p-q)(s+1),                    j4 = 2 (j+p)(s-1)(q+j).
void jacobi_rec(double p, double q, int j, double *r)
{
    if (j == 0) {
        r[0] = 1.0;
        r[1] = -(p + 1.0) / q;
        r[2] = 0.0;
        return;
    }
    double s = 2.0 * j + p;
    double j1 = s * ((s + 1.0) * (s - 1.0) + (q - 1.0) * (q - 1.0) - (p - q) * (p - q));
    double j2 = -2.0 * s * (s + 1.0) * (s - 1.0);
    double j3 = -2.0 * j * (j + p - q) * (s + 1.0);
    double j4 = 2.0 * (j + p) * (s - 1.0) * (q + j);
    r[0] = j1 / j4;
    r[1] = j2 / j4;
    r[2] = j3 / j4;
}

}  // namespace

namespace {

constexpr int ZI_MAX_VALUES = 16384;   // (n_in + n_edge)(N + 1) per geometry

// The row layout, then T, the passbands' weights and (interpolated in z) the
// node rows.
struct GimLayout {
    RowLayout row;
    size_t At, W, zi, total;
};

GimLayout gim_layout(const pt_gim_plan_s *p, int n_t, int n_v, int n_b, int k_per_band, int n_zi)
{
    GimLayout L;
    L.row = row_layout(n_t, n_v, n_b, k_per_band, p->N + 1, (size_t)gim::Q * p->n_int);
    const size_t n_geom = k_per_band ? (size_t)n_v * n_b : (size_t)n_v;
    const size_t R = n_geom * rows_per_geom(k_per_band ? 1 : n_b, p->N + 1);
    size_t off = L.row.total;
    L.At = off;
    off += align256((n_geom + 31) / 32 * 32 * (size_t)(p->N + 1) * p->n_j * sizeof(float));
    L.W = off;
    off += align256((size_t)n_v * n_b * (p->N + 1) * sizeof(float));
    L.zi = off;
    off += align256(R * (((size_t)n_zi + 3) & ~(size_t)3) * sizeof(float));
    L.total = off;
    return L;
}

}  // namespace

// ===========================================================================
// C ABI
// ===========================================================================
// Parameter domain (include/pt.h, pt_domain_check): counts the geometries
// (vector, or vector and passband when k is per passband) whose parameters
// lie outside it.  Reads its inputs only.
__global__ void domain_kernel(const double *t0, const double *P, const float *a, const float *inc, const float *e,
                              const float *w, const float *k, int n_v, int n_kv, int *n_out)
{
    int g = blockIdx.x * blockDim.x + threadIdx.x;
    bool bad = false;
    if (g < n_v * n_kv) {
        int v = g / n_kv;
        const float kk = k[g];
        bad = !(kk > 0.0f && kk <= 1.0e3f);
        if (g % n_kv == 0) {
            const double tv = t0[v], pv = P[v];
            const float av = a[v], iv = inc[v];
            bad |= !(fabs(tv) < 1.0e15) || !(pv > 0.0 && pv < 1.0e15) || !(av > 1.0f && av < 1.0e7f) ||
                   !(iv >= 0.0f && iv <= 3.14159274f);
            if (e) {
                const float ev = e[v], wv = w[v];
                bad |= !(ev >= 0.0f && ev <= 0.95f) || !(fabsf(wv) < 1.0e6f);
            }
        }
    }
    const unsigned m = __ballot_sync(0xffffffffu, bad);
    if ((threadIdx.x & 31) == 0 && m) atomicAdd(n_out, __popc(m));
}

extern "C" {

int pt_version(void) { return 100; }

const char *pt_status_string(int s)
{
    switch (s) {
    case PT_OK: return "ok";
    case PT_ERR_ARG: return "invalid argument";
    case PT_ERR_DOMAIN: return "parameter outside the supported domain";
    case PT_ERR_NOT_CONVERGED: return "iteration did not converge";
    case PT_ERR_CUDA: return "CUDA error";
    case PT_ERR_WORKSPACE: return "work buffer missing or too small";
    default: return "unknown status";
    }
}

const char *pt_last_error_string(void) { return g_last_error; }

int pt_z_circ(const double *t, int n_t, const pt_orbit *orb, int n_ss, double t_exp, float *z,
              pt_stream_t stream)
{
    int st = check_orbit(orb, false);
    if (st) return st;
    if (n_t < 0 || n_ss < 1 || (n_t > 0 && (!t || !z))) return PT_ERR_ARG;
    if (!exposure_ok(t_exp)) return pt_internal::set_error(PT_ERR_DOMAIN, "pt_z_circ", "exposure time must be finite and >= 0");
    if (n_t == 0 || orb->n_v == 0) return PT_OK;
    if ((long long)n_t * n_ss > 0x7fffffffLL || orb->n_v > 65535) return PT_ERR_ARG;
    dim3 grid((n_t * n_ss + 255) / 256, orb->n_v);
    z_circ_kernel<<<grid, 256, 0, (cudaStream_t)stream>>>(t, n_t, orb->t0, orb->P, orb->a, orb->inc, n_ss,
                                                           t_exp, z);
    return check_launch("pt_z_circ");
}

int pt_z_ecc(const double *t, int n_t, const pt_orbit *orb, int n_ss, double t_exp, int max_iter, double tol,
             float *z, int *n_bad, pt_stream_t stream)
{
    int st = check_orbit(orb, true);
    if (st) return st;
    if (n_t < 0 || n_ss < 1 || max_iter < 1 || max_iter > 1000 || !(tol > 0.0) || (n_t > 0 && (!t || !z)))
        return PT_ERR_ARG;
    if (!exposure_ok(t_exp)) return pt_internal::set_error(PT_ERR_DOMAIN, "pt_z_ecc", "exposure time must be finite and >= 0");
    if (n_t == 0 || orb->n_v == 0) return PT_OK;
    if ((long long)n_t * n_ss > 0x7fffffffLL || orb->n_v > 65535) return PT_ERR_ARG;
    dim3 grid((n_t * n_ss + 255) / 256, orb->n_v);
    z_ecc_kernel<<<grid, 256, 0, (cudaStream_t)stream>>>(t, n_t, orb->t0, orb->P, orb->a, orb->inc, orb->e,
                                                          orb->w, n_ss, t_exp, max_iter, tol, z, n_bad);
    return check_launch("pt_z_ecc");
}

int pt_ma_terms(const float *k, const float *z, size_t n, float *le, float *ld, float *ed, pt_stream_t stream)
{
    if (n == 0) return PT_OK;
    if (!k || !z) return PT_ERR_ARG;
    size_t blocks = (n + 255) / 256;
    if (blocks > 0x7fffffffULL) return PT_ERR_ARG;
    ma_terms_kernel<<<(unsigned)blocks, 256, 0, (cudaStream_t)stream>>>(k, z, n, le, ld, ed);
    return check_launch("pt_ma_terms");
}

int pt_domain_check(const pt_orbit *orb, const float *k, int n_k_per_v, int *n_out, pt_stream_t stream)
{
    int st = check_orbit(orb, false);
    if (st) return st;
    if (n_k_per_v < 1 || !n_out) return PT_ERR_ARG;
    if (orb->n_v == 0) return PT_OK;
    if (!k || (long long)orb->n_v * n_k_per_v > 0x7fffffffLL) return PT_ERR_ARG;
    const int n = orb->n_v * n_k_per_v;
    domain_kernel<<<(n + 255) / 256, 256, 0, (cudaStream_t)stream>>>(orb->t0, orb->P, orb->a, orb->inc, orb->e,
                                                                    orb->w, k, orb->n_v, n_k_per_v, n_out);
    return check_launch("pt_domain_check");
}

int pt_status_read(const int *n_bad, const int *n_domain, pt_stream_t stream)
{
    int h[2] = {0, 0};
    cudaStream_t s = (cudaStream_t)stream;
    const int *src[2] = {n_domain, n_bad};
    for (int i = 0; i < 2; ++i) {
        if (!src[i]) continue;
        cudaError_t e = cudaMemcpyAsync(&h[i], src[i], sizeof(int), cudaMemcpyDeviceToHost, s);
        if (e != cudaSuccess) return set_cuda_error(e, "pt_status_read");
    }
    cudaError_t e = cudaStreamSynchronize(s);
    if (e != cudaSuccess) return set_cuda_error(e, "pt_status_read");
    if (h[0] > 0) {
        snprintf(g_last_error, sizeof(g_last_error), "pt_status_read: %d geometries outside the parameter domain",
                 h[0]);
        return PT_ERR_DOMAIN;
    }
    if (h[1] > 0) {
        snprintf(g_last_error, sizeof(g_last_error),
                 "pt_status_read: %d Newton solves stopped at the step cap before converging", h[1]);
        return PT_ERR_NOT_CONVERGED;
    }
    return PT_OK;
}

static int lc_common_check(const double *t, int n_t, const pt_orbit *orb, const float *k, int k_per_band,
                           const float *ld, int n_b, int n_ss, double t_exp, int max_iter, const float *y,
                           float *flux, float *ssr, void *work)
{
    int st = check_orbit(orb, false);
    if (st) return st;
    if (n_t < 0 || n_b < 1 || n_ss < 1 || n_ss > MAX_SS || max_iter < 1 || max_iter > MAX_NEWTON)
        return PT_ERR_ARG;
    if (k_per_band != 0 && k_per_band != 1) return PT_ERR_ARG;
    if (!exposure_ok(t_exp))
        return pt_internal::set_error(PT_ERR_DOMAIN, "light curve", "exposure time must be finite and >= 0");
    if (n_t == 0 || orb->n_v == 0) return PT_OK;   // nothing to evaluate
    if (!flux && !ssr) return PT_ERR_ARG;
    if (!t || !k || !ld) return PT_ERR_ARG;
    if (ssr && !y) return PT_ERR_ARG;
    if (!work || ((uintptr_t)work & 15u)) return PT_ERR_WORKSPACE;
    return PT_OK;
}

size_t pt_ma_quad_work_bytes(int n_t, int n_v, int n_b, int k_per_band)
{
    if (n_t < 0 || n_v < 0 || n_b < 1) return 0;
    // the tile kernel, the exact rows, or a table's rows (of any length that takes them)
    size_t need = work_layout(n_t, n_v, n_b, k_per_band).total;
    const size_t r = row_layout(n_t, n_v, n_b, k_per_band, 3, row_len_max(n_t)).total;
    return r > need ? r : need;
}

static void fill_setup(SetupArgs *sa, const double *t, int n_t, const pt_orbit *orb, const float *k, int k_per_band,
                       int n_b, double t_exp, GeomRec *rec, float2 *tsplit)
{
    sa->t = t;
    sa->n_t = n_t;
    sa->tsplit = tsplit;
    sa->t0 = orb->t0;
    sa->P = orb->P;
    sa->a = orb->a;
    sa->inc = orb->inc;
    sa->e = orb->e;
    sa->w = orb->w;
    sa->k = k;
    sa->n_v = orb->n_v;
    sa->n_b = n_b;
    sa->k_per_band = k_per_band;
    sa->n_geom = k_per_band ? orb->n_v * n_b : orb->n_v;
    sa->rec = rec;
    sa->half_exp = (float)(0.5 * t_exp);
    sa->n_gblocks = 0;
}

static int launch_setup(const double *t, int n_t, const pt_orbit *orb, const float *k, int k_per_band, int n_b,
                        double t_exp, GeomRec *rec, float2 *tsplit, cudaStream_t s)
{
    SetupArgs sa;
    fill_setup(&sa, t, n_t, orb, k, k_per_band, n_b, t_exp, rec, tsplit);
    const int bs = 64;
    sa.n_gblocks = (sa.n_geom + bs - 1) / bs;
    int n_tblocks = (n_t + bs - 1) / bs;
    setup_kernel<<<sa.n_gblocks + n_tblocks, bs, 0, s>>>(sa);
    return check_launch("setup_kernel");
}

}  // extern "C"

// pt_ma_quad and pt_ma_quad_interp from row tables: preparation, row kernel
// (and the sum of the residual partials).
static int ma_quad_rows(const pt_ma_table_s *tab, const double *t, int n_t, const pt_orbit *orb, const float *k,
                        int k_per_band, const float *ld, int n_b, int n_ss, double t_exp, int max_iter,
                        const float *y, const float *wt, float *flux, float *ssr, void *work, size_t work_bytes,
                        int *n_bad, pt_stream_t stream)
{
    const size_t row_len = tab ? interp_row_len(tab->n_z) : (size_t)pt::MT_ROW;
    const RowLayout L = row_layout(n_t, orb->n_v, n_b, k_per_band, 3, row_len);
    if (work_bytes < L.total) return PT_ERR_WORKSPACE;
    const int n_geom = k_per_band ? orb->n_v * n_b : orb->n_v;
    const int n_bpg = k_per_band ? 1 : n_b;
    if ((n_geom + 31) / 32 > 65535) return PT_ERR_ARG;
    cudaStream_t s = (cudaStream_t)stream;
    char *wb = (char *)work;
    int n_sm = 0;
    int st = sm_count(&n_sm);
    if (st) return st;
    RowPrep P;
    memset(&P, 0, sizeof(P));
    fill_setup(&P.s, t, n_t, orb, k, k_per_band, n_b, t_exp, (GeomRec *)(wb + L.rec), (float2 *)(wb + L.tsplit));
    P.s.n_gblocks = (n_geom + 31) / 32;
    P.n_tblocks = (n_t + ROW_THREADS - 1) / ROW_THREADS;
    P.rows = (float *)(wb + L.rows);
    P.row_len = (int)row_len;
    P.nr = rows_per_geom(n_bpg, 3);
    P.terms = row_terms(n_bpg);
    P.n_bpg = n_bpg;
    P.ld = ld;
    P.wts = P.terms ? (float *)(wb + L.wts) : nullptr;
    if (tab) {
        P.mtab = tab->d_tab;
        P.mn_k = tab->n_k;
        P.mn_z = tab->n_z;
        P.mk_lo = tab->k_lo;
        P.mk_hi = tab->k_hi;
        P.minv_dk = tab->inv_dk;
    }
    const long long rblocks = tab ? ((long long)n_geom * P.nr * P.row_len + ROW_THREADS - 1) / ROW_THREADS
                                  : (n_geom + ROW_GEOM - 1) / ROW_GEOM;
    const long long blocks = (long long)P.s.n_gblocks + P.n_tblocks + rblocks;
    if (blocks > 0x7fffffffLL) return PT_ERR_ARG;
    if (tab) row_prep_kernel<rows::R_INTERP><<<(unsigned)blocks, ROW_THREADS, 0, s>>>(P);
    else row_prep_kernel<rows::R_MA><<<(unsigned)blocks, ROW_THREADS, 0, s>>>(P);
    st = check_launch("row_prep_kernel");
    if (st) return st;
    rows::Args A;
    memset(&A, 0, sizeof(A));
    A.tsplit = P.s.tsplit;
    A.n_t = n_t;
    A.rec = P.s.rec;
    A.n_geom = n_geom;
    A.rows = P.rows;
    A.row_len = P.row_len;
    A.nr = P.nr;
    A.terms = P.terms;
    A.n_bpg = n_bpg;
    A.n_b = n_b;
    A.k_per_band = k_per_band;
    A.ld = ld;
    A.wts = P.wts;
    A.n_ss = n_ss;
    A.t_exp = (float)t_exp;
    A.max_iter = max_iter;
    const bool fused_ssr = ssr && !P.terms;
    float *part = (float *)(wb + L.part);
    A.flux = flux ? flux : (P.terms ? (float *)(wb + L.fscr) : nullptr);
    A.ssr_part = fused_ssr ? part : nullptr;
    A.y = y;
    A.wt = wt;
    A.n_bad = n_bad;
    if (tab) {
        A.inv_dz = tab->inv_dz;
        A.n_z = tab->n_z;
    }
    st = launch_rows(tab ? rows::R_INTERP : rows::R_MA, A, n_sm, s);
    if (st || !ssr) return st;
    const int n_rows = orb->n_v * n_b;
    if (!fused_ssr) return launch_ssr_rows(A.flux, y, wt, n_t, n_b, (size_t)n_rows, part, ssr, s);
    pt::launch_chained(ssr_reduce_kernel, (unsigned)(((size_t)n_rows * 32 + 255) / 256), 256, 0, s, part, n_rows, A.n_blk,
                       ssr);
    return check_launch("ssr_reduce_kernel");
}

// pt_ma_quad and pt_ma_quad_interp: exact terms when tab is null, else the
// interpolated ones.
static int ma_quad_impl(const pt_ma_table_s *tab, const double *t, int n_t, const pt_orbit *orb, const float *k,
                        int k_per_band, const float *ld, int n_b, int n_ss, double t_exp, int max_iter,
                        const float *y, const float *wt, float *flux, float *ssr, void *work, size_t work_bytes,
                        int *n_bad, pt_stream_t stream, bool use_rows = true)
{
    int st = lc_common_check(t, n_t, orb, k, k_per_band, ld, n_b, n_ss, t_exp, max_iter, y, flux, ssr, work);
    if (st) return st;
    if (n_t == 0 || orb->n_v == 0) return PT_OK;
    if (use_rows && ma_use_rows(n_t, orb->n_v, n_b, k_per_band, n_ss) &&
        (!tab || interp_use_rows(n_t, orb->n_v, n_b, k_per_band, n_ss, interp_row_len(tab->n_z))))
        return ma_quad_rows(tab, t, n_t, orb, k, k_per_band, ld, n_b, n_ss, t_exp, max_iter, y, wt, flux, ssr, work,
                            work_bytes, n_bad, stream);
    WorkLayout L = work_layout(n_t, orb->n_v, n_b, k_per_band);
    if (work_bytes < L.total) return PT_ERR_WORKSPACE;
    cudaStream_t s = (cudaStream_t)stream;
    char *wb = (char *)work;
    GeomRec *rec = (GeomRec *)(wb + L.rec);
    float2 *tsplit = (float2 *)(wb + L.tsplit);
    float *part = (float *)(wb + L.part);
    const int n_geom = k_per_band ? orb->n_v * n_b : orb->n_v;
    const int n_tiles = (n_t + TT - 1) / TT, gy = (n_geom + VT_MA - 1) / VT_MA;
    if ((n_geom + 31) / 32 > 65535) return PT_ERR_ARG;   // as the row path
    const bool own = (long long)n_tiles * gy <= MA_OWN_MAX_BLOCKS;
    LcArgs A;
    memset(&A, 0, sizeof(A));
    if (own) {
        fill_setup(&A.set, t, n_t, orb, k, k_per_band, n_b, t_exp, rec, tsplit);
    } else {
        st = launch_setup(t, n_t, orb, k, k_per_band, n_b, t_exp, rec, tsplit, s);
        if (st) return st;
    }
    A.tsplit = tsplit;
    A.n_t = n_t;
    A.rec = rec;
    A.n_geom = k_per_band ? orb->n_v * n_b : orb->n_v;
    A.ld = ld;
    A.n_b = n_b;
    A.k_per_band = k_per_band;
    A.n_bpg = k_per_band ? 1 : n_b;
    A.n_ss = n_ss;
    A.t_exp = (float)t_exp;
    A.max_iter = max_iter;
    A.y = y;
    A.wt = wt;
    A.flux = flux;
    A.ssr_part = ssr ? part : nullptr;
    A.n_tiles = n_tiles;
    A.n_bad = n_bad;
    void (*fn)(LcArgs);
    if (tab) {
        A.mtab = tab->d_tab;
        A.mn_k = tab->n_k;
        A.mn_z = tab->n_z;
        A.mk_lo = tab->k_lo;
        A.mk_hi = tab->k_hi;
        A.minv_dk = tab->inv_dk;
        A.minv_dz = tab->inv_dz;
        fn = own ? ma_lc_kernel<true, true> : ma_lc_kernel<true, false>;
    } else {
        fn = own ? ma_lc_kernel<false, true> : ma_lc_kernel<false, false>;
    }
    // Time tiles along x, geometries along y, in as many launches as y takes.  (An
    // offset added to the geometry in the kernel costs 10 % where a block has few
    // times: 20,000 vectors x 20 times 32.9 -> 36.8 us.)
    const int chunk = 65535 * VT_MA;
    for (int first = 0; first < n_geom; first += chunk) {
        LcArgs C = A;
        const size_t row0 = (size_t)first * A.n_bpg;
        C.rec = A.rec + first;
        C.n_geom = std::min(chunk, n_geom - first);
        C.band0 = first % n_b;
        C.ld = A.ld + 2 * row0;
        C.flux = A.flux ? A.flux + row0 * n_t : nullptr;
        C.ssr_part = A.ssr_part ? A.ssr_part + row0 * n_tiles : nullptr;
        const dim3 grid(A.n_tiles, (C.n_geom + VT_MA - 1) / VT_MA);
        if (own)
            fn<<<grid, TT, 0, s>>>(C);
        else
            pt::launch_chained(fn, grid, TT, 0, s, C);
        st = check_launch("ma_lc_kernel");
        if (st) return st;
    }
    if (ssr) {
        int rows = orb->n_v * n_b;
        pt::launch_chained(ssr_reduce_kernel, (unsigned)(((size_t)rows * 32 + 255) / 256), 256, 0, s, part, rows, A.n_tiles,
                           ssr);
        st = check_launch("ssr_reduce_kernel");
    }
    return st;
}

extern "C" {

int pt_ma_quad(const double *t, int n_t, const pt_orbit *orb, const float *k, int k_per_band, const float *ld,
               int n_b, int n_ss, double t_exp, int max_iter, const float *y, const float *wt, float *flux,
               float *ssr, void *work, size_t work_bytes, int *n_bad, pt_stream_t stream)
{
    return ma_quad_impl(nullptr, t, n_t, orb, k, k_per_band, ld, n_b, n_ss, t_exp, max_iter, y, wt, flux, ssr,
                        work, work_bytes, n_bad, stream);
}

int pt_ma_quad_interp(pt_ma_table table, const double *t, int n_t, const pt_orbit *orb, const float *k,
                      int k_per_band, const float *ld, int n_b, int n_ss, double t_exp, int max_iter, const float *y,
                      const float *wt, float *flux, float *ssr, void *work, size_t work_bytes, int *n_bad,
                      pt_stream_t stream)
{
    if (!table) return PT_ERR_ARG;
    return ma_quad_impl(table, t, n_t, orb, k, k_per_band, ld, n_b, n_ss, t_exp, max_iter, y, wt, flux, ssr, work,
                        work_bytes, n_bad, stream);
}

int pt_ma_table_create(float k_lo, float k_hi, int n_k, int n_z, pt_ma_table *out)
{
    if (!out) return PT_ERR_ARG;
    *out = nullptr;
    if (!(k_lo > 0.0f) || !(k_hi > k_lo) || n_k < 2 || n_k > 4096 || n_z < 2 || n_z > 65536) return PT_ERR_ARG;
    pt_ma_table p = new pt_ma_table_s;
    p->k_lo = k_lo;
    p->k_hi = k_hi;
    p->n_k = n_k;
    p->n_z = n_z;
    p->inv_dk = (float)((n_k - 1) / ((double)k_hi - (double)k_lo));
    p->inv_dz = (float)((n_z - 1) / (1.0 + (double)k_hi));
    p->d_tab = nullptr;
    size_t cnt = (size_t)n_k * n_z;
    cudaError_t e = cudaMalloc(&p->d_tab, cnt * sizeof(float4));
    if (e == cudaSuccess) {
        ma_table_kernel<<<(unsigned)((cnt + 255) / 256), 256>>>(k_lo, k_hi, n_k, n_z, p->d_tab);
        e = cudaGetLastError();
    }
    if (e == cudaSuccess) e = cudaDeviceSynchronize();
    if (e != cudaSuccess) {
        cudaFree(p->d_tab);
        delete p;
        return set_cuda_error(e, "pt_ma_table_create");
    }
    *out = p;
    return PT_OK;
}

int pt_ma_table_destroy(pt_ma_table p)
{
    if (!p) return PT_OK;
    cudaFree(p->d_tab);
    delete p;
    return PT_OK;
}

int pt_ma_terms_interp(pt_ma_table p, const float *k, const float *z, size_t n, float *le, float *ld, float *ed,
                       pt_stream_t stream)
{
    if (!p) return PT_ERR_ARG;
    if (n == 0) return PT_OK;
    if (!k || !z) return PT_ERR_ARG;
    size_t blocks = (n + 255) / 256;
    if (blocks > 0x7fffffffULL) return PT_ERR_ARG;
    ma_terms_interp_kernel<<<(unsigned)blocks, 256, 0, (cudaStream_t)stream>>>(
        p->d_tab, p->n_k, p->n_z, p->k_lo, p->k_hi, p->inv_dk, p->inv_dz, k, z, n, le, ld, ed);
    return check_launch("pt_ma_terms_interp");
}

int pt_gim_plan_create(int N, int n_j, pt_gim_plan *out)
{
    if (!out || N < 1 || N > 16 || n_j < 2 || n_j > 512) return PT_ERR_ARG;
    *out = nullptr;
    const int NP1 = N + 1;
    const size_t cnt = (size_t)NP1 * n_j;
    const int n_int = gim::intervals(N, n_j);
    constexpr int Q = gim::Q;
    // one allocation: the uploaded tables, then those that the kernel derives
    size_t total = 0;
    auto part = [&](size_t bytes) {
        const size_t at = total;
        total += (bytes + 255) & ~(size_t)255;
        return at;
    };
    const size_t oA = part(cnt * sizeof(double)), orb = part(cnt * 3 * sizeof(double)),
                 orc = part(cnt * 3 * sizeof(float2)), upload = total, oc = part(cnt * sizeof(float4)),
                 odA = part(cnt * sizeof(float2)), odrb = part(cnt * 3 * sizeof(float2)),
                 oB = part(cnt * n_int * Q * sizeof(float));
    std::unique_ptr<double[]> host(new (std::nothrow) double[upload / sizeof(double)]);
    if (!host) return pt_internal::set_error(PT_ERR_CUDA, "pt_gim_plan_create", "out of host memory");
    double *hA = host.get() + oA / sizeof(double), *hrb = host.get() + orb / sizeof(double);
    float2 *hrc = (float2 *)(host.get() + orc / sizeof(double));
    for (int n = 0; n < NP1; ++n) {
        double nu = 0.5 * (n + 2);
        // A_{n,j} = (-1)^j (2j+nu+2)/nu * prod_{i=1..j} (nu+i)/(i+1)   (Eq. gimemez_a)
        double prod = 1.0;
        for (int j = 0; j < n_j; ++j) {
            const size_t at = (size_t)n * n_j + j;
            if (j > 0) prod *= (nu + j) / (j + 1.0);
            hA[at] = ((j & 1) ? -1.0 : 1.0) * (2.0 * j + nu + 2.0) / nu * prod;
            double rc[3];
            jacobi_rec(nu + 2.0, 1.0, j, rc);
            for (int c = 0; c < 3; ++c) {
                const float h = (float)rc[c];
                hrc[3 * at + c] = make_float2(h, (float)(rc[c] - (double)h));
            }
            jacobi_rec(nu + 2.0, nu + 1.0, j, hrb + 3 * at);
        }
    }
    gim::Basis P;
    // values at the points x_q -> Chebyshev coefficients -> powers of x, for
    // the sums (even powers) and differences (odd) of the pairs x_q, -x_q
    double T[Q][Q] = {};   // T_k by powers of x
    T[0][0] = T[1][1] = 1.0;
    for (int k = 2; k < Q; ++k)
        for (int c = 0; c < Q; ++c) T[k][c] = (c > 0 ? 2.0 * T[k - 1][c - 1] : 0.0) - T[k - 2][c];
    for (int q = 0; q < Q; ++q) P.xq[q] = cos((q + 0.5) * PI_D / Q);
    for (int c = 0; c < Q; ++c)
        for (int q = 0; q < Q / 2; ++q) {
            double v = 0.0;
            for (int k = 0; k < Q; ++k) v += (k == 0 ? 1.0 : 2.0) / Q * cos(k * (q + 0.5) * PI_D / Q) * T[k][c];
            const float h = (float)v;
            P.m[c & 1][c / 2][q] = make_float2(h, (float)(v - (double)h));
        }
    unsigned char *d = nullptr;
    cudaError_t e = cudaMalloc(&d, total);
    if (e != cudaSuccess) return set_cuda_error(e, "pt_gim_plan_create");
    e = cudaMemcpy(d, host.get(), upload, cudaMemcpyHostToDevice);
    if (e == cudaSuccess) {
        P.A = (const double *)(d + oA);
        P.recb = (const double *)(d + orb);
        P.rec = (const float2 *)(d + orc);
        P.coef = (float4 *)(d + oc);
        P.dA = (float2 *)(d + odA);
        P.drb = (float2 *)(d + odrb);
        P.B = (float *)(d + oB);
        P.NP1 = NP1;
        P.n_j = n_j;
        P.n_int = n_int;
        P.scale = (double)gim::row_scale(n_int);
        gim::basis_kernel<<<dim3((n_int + 3) / 4, NP1), gim::BASIS_TB, 3 * n_j * sizeof(float2)>>>(P);
        e = cudaGetLastError();
    }
    if (e == cudaSuccess) e = cudaStreamSynchronize(nullptr);
    if (e != cudaSuccess) {
        cudaFree(d);
        return set_cuda_error(e, "pt_gim_plan_create");
    }
    pt_gim_plan p = new (std::nothrow) pt_gim_plan_s;
    if (!p) {
        cudaFree(d);
        return pt_internal::set_error(PT_ERR_CUDA, "pt_gim_plan_create", "out of host memory");
    }
    p->N = N;
    p->n_j = n_j;
    p->n_int = n_int;
    p->d_mem = d;
    p->d_coef = P.coef;
    p->d_A = P.A;
    p->d_recb = P.recb;
    p->d_dA = P.dA;
    p->d_drb = P.drb;
    p->d_B = P.B;
    p->ev0 = p->ev1 = nullptr;
    *out = p;
    return PT_OK;
}

int pt_gim_plan_time_evaluation(pt_gim_plan p, void *ev_start, void *ev_end)
{
    if (!p || (ev_start == nullptr) != (ev_end == nullptr)) return PT_ERR_ARG;
    p->ev0 = (cudaEvent_t)ev_start;
    p->ev1 = (cudaEvent_t)ev_end;
    return PT_OK;
}

int pt_gim_plan_destroy(pt_gim_plan p)
{
    if (!p) return PT_OK;
    cudaFree(p->d_mem);
    delete p;
    return PT_OK;
}

int pt_gimenez_alpha(pt_gim_plan plan, const float *k, const float *z, size_t n, float *alpha,
                     pt_stream_t stream)
{
    if (!plan) return PT_ERR_ARG;
    if (n == 0) return PT_OK;
    if (!k || !z || !alpha) return PT_ERR_ARG;
    size_t blocks = (n + 127) / 128;
    if (blocks > 0x7fffffffULL) return PT_ERR_ARG;
    gim_alpha_kernel<<<(unsigned)blocks, 128, 0, (cudaStream_t)stream>>>(k, z, n, plan->N + 1, plan->n_j,
                                                                         plan->d_coef, plan->d_A,
                                                                         plan->d_recb, alpha);
    return check_launch("pt_gimenez_alpha");
}

size_t pt_gimenez_work_bytes(pt_gim_plan plan, int n_t, int n_v, int n_b, int k_per_band)
{
    if (!plan || n_t < 0 || n_v < 0 || n_b < 1) return 0;
    return gim_layout(plan, n_t, n_v, n_b, k_per_band, 0).total;
}

}  // extern "C"

// pt_gimenez (n_in == 0: the series' rows) and pt_gimenez_zi (the rows on z
// nodes): preparation with the T_{n,j}, the products that form the rows, (the
// nodes,) the row kernel.
static int gimenez_impl(pt_gim_plan plan, int n_in, int n_edge, const double *t, int n_t, const pt_orbit *orb,
                        const float *k, int k_per_band, const float *ld, int n_b, int n_ss, double t_exp,
                        int max_iter, const float *y, const float *wt, float *flux, float *ssr, void *work,
                        size_t work_bytes, int *n_bad, pt_stream_t stream)
{
    if (!plan) return PT_ERR_ARG;
    const bool zi = n_in > 0;
    if (zi && (n_in < 2 || n_edge < 1 || (size_t)(n_in + n_edge) * (plan->N + 1) > (size_t)ZI_MAX_VALUES))
        return PT_ERR_ARG;
    int st = lc_common_check(t, n_t, orb, k, k_per_band, ld, n_b, n_ss, t_exp, max_iter, y, flux, ssr, work);
    if (st) return st;
    if (n_t == 0 || orb->n_v == 0) return PT_OK;
    const int NP1 = plan->N + 1, Nc = gim::Q * plan->n_int;
    const GimLayout L = gim_layout(plan, n_t, orb->n_v, n_b, k_per_band, zi ? n_in + n_edge : 0);
    if (work_bytes < L.total) return PT_ERR_WORKSPACE;
    const int n_geom = k_per_band ? orb->n_v * n_b : orb->n_v;
    const int n_bpg = k_per_band ? 1 : n_b;
    if ((n_geom + 31) / 32 > 65535) return PT_ERR_ARG;
    cudaStream_t s = (cudaStream_t)stream;
    char *wb = (char *)work;
    int n_sm = 0;
    st = sm_count(&n_sm);
    if (st) return st;
    RowPrep P;
    memset(&P, 0, sizeof(P));
    fill_setup(&P.s, t, n_t, orb, k, k_per_band, n_b, t_exp, (GeomRec *)(wb + L.row.rec), (float2 *)(wb + L.row.tsplit));
    P.s.n_gblocks = (n_geom + 31) / 32;
    P.n_tblocks = (n_t + ROW_THREADS - 1) / ROW_THREADS;
    P.rows = (float *)(wb + L.row.rows);
    P.row_len = Nc;
    P.nr = rows_per_geom(n_bpg, NP1);
    P.terms = row_terms(n_bpg);
    P.n_bpg = n_bpg;
    P.ld = ld;
    const size_t R = (size_t)n_geom * P.nr;
    P.gim.dA = plan->d_dA;
    P.gim.drb = plan->d_drb;
    P.gim.NP1 = NP1;
    P.gim.n_j = plan->n_j;
    P.gim.At = (float *)(wb + L.At);
    P.gim.Gp = (n_geom + 31) / 32 * 32;
    P.gim.W = (float *)(wb + L.W);
    const long long blocks = (long long)P.s.n_gblocks + P.n_tblocks + (long long)NP1 * ((n_geom + gim::GPC - 1) / gim::GPC);
    if (blocks > 0x7fffffffLL || R > 0x7fffffffULL - 32) return PT_ERR_ARG;
    const size_t tsm = gim::table_smem(plan->n_j);
    cudaError_t e = cudaSuccess;
    if (tsm > VARIABLE_SMEM_MAX) return pt_internal::set_error(PT_ERR_ARG, "row_prep_kernel", "series too long");
    if (tsm > DEFAULT_SMEM) e = pt::allow_smem(row_prep_kernel<rows::R_GIM>, VARIABLE_SMEM_MAX);
    if (e != cudaSuccess) return set_cuda_error(e, "row_prep_kernel smem attribute");
    row_prep_kernel<rows::R_GIM><<<(unsigned)blocks, ROW_THREADS, tsm, s>>>(P);
    st = check_launch("row_prep_kernel");
    if (st) return st;
    gim::Product pr;
    memset(&pr, 0, sizeof(pr));
    pr.At = P.gim.At;
    pr.Gp = P.gim.Gp;
    pr.G = n_geom;
    pr.B = plan->d_B;
    pr.n_j = plan->n_j;
    pr.NP1 = NP1;
    pr.per = gim::chain_len(NP1, plan->n_j);
    pr.chains = gim::chains(NP1, plan->n_j);
    pr.Nc = Nc;
    pr.W = P.terms ? nullptr : P.gim.W;
    pr.nr = P.nr;
    pr.out = P.rows;
    const gim::Form form = gim::product_form((size_t)n_geom, Nc, gim::tall_fits(NP1, plan->n_j, P.terms || P.nr == 1), n_sm);
    pr.spread = form.spread;
    auto product = [&](auto fn, auto shape) -> int {
        using S = decltype(shape);
        const size_t n = ((size_t)n_geom + form.rt - 1) / form.rt * (((size_t)Nc + S::CT - 1) / S::CT);
        if (n > 0x7fffffffULL) return PT_ERR_ARG;
        const int warps = NP1 * (pr.spread ? pr.chains : 1);
        const size_t smem = ((size_t)warps * S::warp_floats(pr.spread || pr.chains == 1) +
                             (pr.W ? (size_t)form.rt * pr.nr * NP1 : 0)) * sizeof(float);
        if (smem > S::SMEM_MAX) return pt_internal::set_error(PT_ERR_ARG, "product_kernel", "too many orders");
        e = smem > DEFAULT_SMEM ? pt::allow_smem(fn, S::SMEM_MAX) : cudaSuccess;
        if (e != cudaSuccess) return set_cuda_error(e, "product_kernel smem attribute");
        pt::launch_chained(fn, (unsigned)n, 32 * warps, smem, s, pr);
        return PT_OK;
    };
#define PT_PRODUCT(RT, C) product(gim::product_kernel<RT, C>, gim::Shape<RT, C>())
    if (form.rt == gim::TALL) {
        const size_t n = ((size_t)n_geom + gim::TALL - 1) / gim::TALL * (((size_t)Nc + gim::TALL - 1) / gim::TALL);
        if (n > 0x7fffffffULL) return PT_ERR_ARG;
        e = pt::allow_smem(gim::product_tall_kernel, gim::TALL_SMEM);
        if (e != cudaSuccess) return set_cuda_error(e, "product_tall_kernel smem attribute");
        pt::launch_chained(gim::product_tall_kernel, (unsigned)n, 256, gim::TALL_SMEM, s, pr);
    } else if (form.rt == 32)
        st = form.c == 6 ? PT_PRODUCT(32, 6) : PT_PRODUCT(32, 4);
    else
        st = form.c == 2 ? PT_PRODUCT(8, 2) : PT_PRODUCT(8, 1);
#undef PT_PRODUCT
    if (st) return st;
    st = check_launch("product_kernel");
    if (st) return st;
    rows::Args A;
    memset(&A, 0, sizeof(A));
    A.tsplit = P.s.tsplit;
    A.n_t = n_t;
    A.rec = P.s.rec;
    A.n_geom = n_geom;
    A.rows = P.rows;
    A.row_len = P.row_len;
    A.nr = P.nr;
    A.terms = P.terms;
    A.n_bpg = n_bpg;
    A.n_b = n_b;
    A.k_per_band = k_per_band;
    A.n_ss = n_ss;
    A.t_exp = (float)t_exp;
    A.max_iter = max_iter;
    A.scale = gim::row_scale(plan->n_int);
    A.wts = P.gim.W;
    const bool fused_ssr = ssr && !P.terms;
    float *part = (float *)(wb + L.row.part);
    A.flux = flux ? flux : (P.terms ? (float *)(wb + L.row.fscr) : nullptr);
    A.ssr_part = fused_ssr ? part : nullptr;
    A.y = y;
    A.wt = wt;
    A.n_bad = n_bad;
    if (zi) {
        A.n_in = n_in;
        A.n_edge = n_edge;
        const int zi_len = (n_in + n_edge + 3) & ~3;
        float *zrows = (float *)(wb + L.zi);
        const long long n = (long long)R * zi_len;
        if ((n + 127) / 128 > 0x7fffffffLL) return PT_ERR_ARG;
        pt::launch_chained(gim::zi_rows_kernel, (unsigned)((n + 127) / 128), 128, 0, s, A, k, (int)R, zi_len, zrows);
        st = check_launch("zi_rows_kernel");
        if (st) return st;
        A.rows = zrows;
        A.row_len = zi_len;
    }
    if (plan->ev0 && (e = cudaEventRecord(plan->ev0, s)) != cudaSuccess) return set_cuda_error(e, "pt_gimenez timing event");
    st = launch_rows(zi ? rows::R_ZI : rows::R_GIM, A, n_sm, s);
    if (st) return st;
    if (plan->ev1 && (e = cudaEventRecord(plan->ev1, s)) != cudaSuccess) return set_cuda_error(e, "pt_gimenez timing event");
    if (!ssr) return PT_OK;
    const int n_rows = orb->n_v * n_b;
    if (!fused_ssr) return launch_ssr_rows(A.flux, y, wt, n_t, n_b, (size_t)n_rows, part, ssr, s);
    pt::launch_chained(ssr_reduce_kernel, (unsigned)(((size_t)n_rows * 32 + 255) / 256), 256, 0, s, part, n_rows, A.n_blk,
                       ssr);
    return check_launch("ssr_reduce_kernel");
}

extern "C" {

int pt_gimenez(pt_gim_plan plan, const double *t, int n_t, const pt_orbit *orb, const float *k, int k_per_band,
               const float *ld, int n_b, int n_ss, double t_exp, int max_iter, const float *y, const float *wt,
               float *flux, float *ssr, void *work, size_t work_bytes, int *n_bad, pt_stream_t stream)
{
    return gimenez_impl(plan, 0, 0, t, n_t, orb, k, k_per_band, ld, n_b, n_ss, t_exp, max_iter, y, wt, flux, ssr,
                        work, work_bytes, n_bad, stream);
}

size_t pt_gimenez_zi_work_bytes(pt_gim_plan plan, int n_in, int n_edge, int n_t, int n_v, int n_b, int k_per_band)
{
    if (!plan || n_t < 0 || n_v < 0 || n_b < 1 || n_in < 2 || n_edge < 1) return 0;
    return gim_layout(plan, n_t, n_v, n_b, k_per_band, n_in + n_edge).total;
}

int pt_gimenez_zi(pt_gim_plan plan, int n_in, int n_edge, const double *t, int n_t, const pt_orbit *orb,
                  const float *k, int k_per_band, const float *ld, int n_b, int n_ss, double t_exp, int max_iter,
                  const float *y, const float *wt, float *flux, float *ssr, void *work, size_t work_bytes,
                  int *n_bad, pt_stream_t stream)
{
    if (n_in < 2) return PT_ERR_ARG;
    return gimenez_impl(plan, n_in, n_edge, t, n_t, orb, k, k_per_band, ld, n_b, n_ss, t_exp, max_iter, y, wt, flux,
                        ssr, work, work_bytes, n_bad, stream);
}

}  // extern "C"

// ===========================================================================
// Allocation-free variant of pt_ma_quad.
//
// Some callers cannot call cudaMalloc: a host program that hands all device
// memory to its own fixed pool and forbids outside allocations, or a tight
// sampling loop where an allocation (and the stall it can cause) is not
// acceptable.  For them pt_ma_quad_noalloc takes its scratch from a
// statically sized __device__ array instead of a caller-provided work
// buffer.  The array is part of the module image: every GPU that loads the
// library holds PT_MA_NOALLOC_SCRATCH_BYTES of it until the process exits.
// ===========================================================================
namespace {

static __device__ __align__(256) unsigned char g_ma_noalloc_scratch[PT_MA_NOALLOC_SCRATCH_BYTES];

constexpr int NOALLOC_MAX_DEVICES = 64;
void *g_noalloc_ptr[NOALLOC_MAX_DEVICES] = {nullptr};
std::mutex g_noalloc_mutex;

// Device address of the scratch array for the current device.  In host code
// the symbol name is only a host-side stand-in, so the address is fetched
// with cudaGetSymbolAddress once per device (with that device current) and
// cached.
int noalloc_scratch(void **out)
{
    int dev = -1;
    cudaError_t e = cudaGetDevice(&dev);
    if (e != cudaSuccess) return set_cuda_error(e, "pt_ma_quad_noalloc: cudaGetDevice");
    if (dev < 0 || dev >= NOALLOC_MAX_DEVICES) {
        snprintf(g_last_error, sizeof(g_last_error), "pt_ma_quad_noalloc: device %d beyond the %d supported", dev,
                 NOALLOC_MAX_DEVICES);
        return PT_ERR_ARG;
    }
    std::lock_guard<std::mutex> lock(g_noalloc_mutex);
    if (!g_noalloc_ptr[dev]) {
        void *p = nullptr;
        e = cudaGetSymbolAddress(&p, g_ma_noalloc_scratch);
        if (e != cudaSuccess) return set_cuda_error(e, "pt_ma_quad_noalloc: cudaGetSymbolAddress");
        g_noalloc_ptr[dev] = p;
    }
    *out = g_noalloc_ptr[dev];
    return PT_OK;
}

}  // namespace

extern "C" int pt_ma_quad_noalloc(const double *t, int n_t, const pt_orbit *orb, const float *k, int k_per_band,
                                  const float *ld, int n_b, int n_ss, double t_exp, int max_iter,
                                  const float *y, const float *wt, float *flux, float *ssr, int *n_bad,
                                  pt_stream_t stream)
{
    if (!orb || n_t < 0 || orb->n_v < 0 || n_b < 1) return PT_ERR_ARG;
    // the tile kernel: its scratch is small (records, time split, partials)
    size_t need = work_layout(n_t, orb->n_v, n_b, k_per_band).total;
    if (need > (size_t)PT_MA_NOALLOC_SCRATCH_BYTES) {
        snprintf(g_last_error, sizeof(g_last_error),
                 "pt_ma_quad_noalloc: this problem needs %zu bytes of scratch, the static scratch holds %zu; "
                 "use pt_ma_quad with a work buffer", need, (size_t)PT_MA_NOALLOC_SCRATCH_BYTES);
        return PT_ERR_WORKSPACE;
    }
    void *scratch = nullptr;
    int st = noalloc_scratch(&scratch);
    if (st) return st;
    // Every scratch byte the kernels read is written earlier in the same call
    // (geometry records, time split, residual partials), so nothing is cleared.
    return ma_quad_impl(nullptr, t, n_t, orb, k, k_per_band, ld, n_b, n_ss, t_exp, max_iter, y, wt, flux, ssr,
                        scratch, (size_t)PT_MA_NOALLOC_SCRATCH_BYTES, n_bad, stream, false);
}
