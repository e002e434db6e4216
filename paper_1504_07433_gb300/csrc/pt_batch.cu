// pt_batch.cu -- one persistent, graph-captured launch over many MCMC walkers,
// passbands and light curves of uneven length (spectrophotometry: the paper's
// motivation in Sec. 1; per-passband radius ratios and limb darkening,
// Secs. 2.2.2 and 3.5; the device-side likelihood of Sec. 3.4).
//
// batch_prep_kernel, per call:
//   - the walkers' geometry records, the double-float split of the times;
//   - per tile of BT consecutive times (as stored; they need not be sorted)
//     the tile's time range and, per passband, its residual sum with the flux
//     at 1;
//   - per (walker, passband) the row table of its transit depth as a function
//     of z (pt_device.cuh: 144 evaluations of the exact terms).  Every row is
//     then read at tens of thousands of separations (all in-window times of
//     all light curves), so the elliptic integrals have left the per-point
//     work: at 1,024 walkers x 64 passbands x 81,058 times a call went from
//     17.5 ms (the terms evaluated per point) to 2.80 ms.
// batch_kernel: persistent CTAs take (walker, group of BG passbands, slice of
// the times) items from an atomic counter, ordered so that consecutive items
// share their observations in L2.  Per item the group's rows are staged in
// shared memory; tiles that cannot meet the walker's transit window add their
// prepared residual sums (and flux 1); the others are evaluated one time per
// thread: z once, then the group's depths, fluxes and residuals, the sums in
// registers.  Per point and passband that is about 22 instructions for the
// depth and 4 for the residual; the issue rate bounds it, the observations
// come from L2.
// The plan autotunes the CTA size and the number of slices by timing the
// candidates on the caller's buffers, then captures counter reset +
// preparation + persistent kernel + reduction into one CUDA graph.
#include <cuda_runtime.h>

#include <math.h>
#include <stdint.h>
#include <stdio.h>
#include <string.h>

#include <algorithm>
#include <vector>

#include "../../include/pt.h"
#include "pt_device.cuh"

using pt::GeomRec;

namespace pt_internal {
int set_error(int status, const char *where, const char *msg);   // pt_lc.cu
bool ma_table_view(pt_ma_table t, const float4 **tab, int *n_k, int *n_z, float *k_lo, float *k_hi, float *inv_dk,
                   float *inv_dz);                                   // pt_lc.cu
}

namespace {

constexpr int BT = 64;                   // times per tile
constexpr int BG = 16;                   // passbands per group (residual sums of a group in registers)
constexpr int PREP_ROWS = 2;             // row tables per CTA of the preparation
constexpr int PREP = PREP_ROWS * pt::MT_NODES;   // its threads: one node of a row each
constexpr int PREP_TILES = PREP / BT;    // tiles of times per CTA
constexpr size_t INTERP_SMEM = 64 * 1024;   // largest staged group of interpolated rows

// What a depth is formed from.
enum Mode {
    M_ROWS = 0,     // k_mode 0: row tables of the exact depth
    M_KHAT = 1,     // k_mode 1: the exact terms once per time with k_hat, scaled per passband (Sec. 3.5)
    M_INTERP = 2,   // k_mode 2: rows of the caller's table, interpolated in k, staged in shared memory
    M_GATHER = 3,   // k_mode 2 with rows too long to stage: bilinear reads of the table per point
    M_EXACT = 4     // k_mode 0, too few points for row tables: the exact terms per point
};

// What is asked for: the two usual calls have no run-time choice per point.
enum Out { O_FLUX = 0, O_SSR = 1 /* unit weights */, O_ANY = 2 };

struct BatchArgs {
    const float2 *tsplit;
    int n_t;
    const GeomRec *rec;
    const float *k;      // [n_v][n_b]
    const float *ld;     // [n_v][n_b][2]
    const float *rows;   // [n_v][n_b][MT_ROW], M_ROWS
    const int2 *tiles;       // [n_tiles] (first time, length): tiles never straddle a light curve
    const float2 *tile_mm;   // [n_tiles] smallest and largest time
    const float *base;   // [n_b][n_tiles] residual sums with the flux at 1
    int n_tiles;
    int n_v, n_b, n_ss;
    float t_exp;
    int max_iter;
    const float *y, *wt; // [n_b][n_t]
    float *flux;         // [n_v][n_b][n_t]
    float *ssr_part;     // [n_v][n_b][n_slices]
    int bg;              // passbands per group, at most BG
    int n_groups, n_slices, tiles_per_slice;
    int n_items;
    int *counter;
    int *n_bad;
    // k_mode 2: the Mandel-Agol terms interpolated from this table (Sec. 2.2.3)
    const float4 *mtab;
    int mn_k, mn_z;
    float mk_lo, mk_hi, minv_dk, minv_dz;
};

struct PrepArgs {
    const double *t;
    int n_t;
    float2 *tsplit;
    pt_orbit orb;
    const float *k, *ld;
    int n_b;
    float half_exp;
    GeomRec *rec;
    int khat;
    const int2 *tiles;
    float2 *tile_mm;
    float *base;         // null: no residual sums wanted
    const float *y, *wt;
    int n_tiles;
    float *rows;         // null: no row tables
    int n_gblocks, n_tblocks, n_bblocks;
};

// transit depth weights of one passband: depth = we le + wd ld + wn ed
__device__ __forceinline__ float3 band_weights(const float *ld, size_t row)
{
    float3 w;
    pt::ma_weights(ld[row * 2], ld[row * 2 + 1], &w.x, &w.y, &w.z);
    return w;
}

constexpr int PREP_BASE = 8;   // (passband, tile) residual sums per warp of the preparation

__global__ void __launch_bounds__(PREP) batch_prep_kernel(PrepArgs s)
{
    __shared__ float sF[PREP_ROWS][pt::MT_N * (pt::MT_Q + 1)];
    __shared__ double smin[PREP / 32], smax[PREP / 32];
    const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
    int blk = blockIdx.x;
    if (blk < s.n_gblocks) {
        // one warp per CTA: the records' FP64 operations share one slow pipe per SM
        const int v = blk * 32 + tid;
        if (tid >= 32 || v >= s.orb.n_v) return;
        // the geometry's k: the largest passband k (its window covers every
        // passband), or in k_hat mode the mean, the only k evaluated
        float kmax = 0.0f, ksum = 0.0f;
        for (int b = 0; b < s.n_b; ++b) {
            float kb = s.k[(size_t)v * s.n_b + b];
            kmax = fmaxf(kmax, kb);
            ksum += kb;
        }
        if (s.khat) kmax = ksum / (float)s.n_b;
        bool ecc = s.orb.e != nullptr;
        pt::make_geom_rec(s.orb.t0[v], s.orb.P[v], s.orb.a[v], s.orb.inc[v], ecc, ecc ? s.orb.e[v] : 0.0f,
                          ecc ? s.orb.w[v] : 0.0f, kmax, s.half_exp, &s.rec[v]);
        return;
    }
    blk -= s.n_gblocks;
    if (blk < s.n_tblocks) {
        // PREP_TILES tiles: time split, smallest and largest time (rounded outward)
        const int tile = blk * PREP_TILES + tid / BT;
        const int2 tl = tid < PREP_TILES * BT && tile < s.n_tiles ? s.tiles[tile] : make_int2(0, 0);
        const int i = tl.x + (tid & (BT - 1));
        double lo = INFINITY, hi = -INFINITY;
        if ((tid & (BT - 1)) < tl.y) {
            const double x = s.t[i];
            const float h = (float)x;
            s.tsplit[i] = make_float2(h, (float)(x - (double)h));
            lo = hi = x;
        }
#pragma unroll
        for (int o = 16; o > 0; o >>= 1) {
            lo = fmin(lo, __shfl_xor_sync(0xffffffffu, lo, o));
            hi = fmax(hi, __shfl_xor_sync(0xffffffffu, hi, o));
        }
        if (lane == 0) {
            smin[warp] = lo;
            smax[warp] = hi;
        }
        __syncthreads();
        const int out = blk * PREP_TILES + tid;
        if (tid < PREP_TILES && out < s.n_tiles) {
            lo = fmin(smin[2 * tid], smin[2 * tid + 1]);
            hi = fmax(smax[2 * tid], smax[2 * tid + 1]);
            float flo = (float)lo, fhi = (float)hi;
            if ((double)flo > lo) flo = nextafterf(flo, -INFINITY);
            if ((double)fhi < hi) fhi = nextafterf(fhi, INFINITY);
            s.tile_mm[out] = make_float2(flo, fhi);
        }
        return;
    }
    blk -= s.n_tblocks;
    if (blk < s.n_bblocks) {
        // residual sums of (passband, tile) with the flux at 1, one warp each
        const long long n_task = (long long)s.n_b * s.n_tiles;
        const long long q0 = ((long long)blk * (PREP / 32) + warp) * PREP_BASE;
        for (long long q = q0; q < q0 + PREP_BASE && q < n_task; ++q) {
            const int b = (int)(q / s.n_tiles), tile = (int)(q - (long long)b * s.n_tiles);
            const int2 tl = s.tiles[tile];
            float acc = 0.0f;
#pragma unroll
            for (int h = 0; h < BT / 32; ++h) {
                const int i = tl.x + 32 * h + lane;
                if (32 * h + lane < tl.y) {
                    const float r = s.y[(size_t)b * s.n_t + i] - 1.0f;
                    acc = fmaf((s.wt ? s.wt[(size_t)b * s.n_t + i] : 1.0f) * r, r, acc);
                }
            }
#pragma unroll
            for (int o = 16; o > 0; o >>= 1) acc += __shfl_xor_sync(0xffffffffu, acc, o);
            if (lane == 0) s.base[q] = acc;
        }
        return;
    }
    blk -= s.n_bblocks;
    // PREP_ROWS row tables: a node per thread (region A's, in double-float
    // arithmetic, on the first warps), then a coefficient per thread
    const size_t n_rows = (size_t)s.orb.n_v * s.n_b, first = (size_t)blk * PREP_ROWS;
    constexpr int NODES_A = pt::MT_NA * pt::MT_Q, NODES_L = pt::MT_NODES - NODES_A;
    {
        const bool in_a = tid < PREP_ROWS * NODES_A;
        const int u = in_a ? tid : tid - PREP_ROWS * NODES_A;
        const int r = in_a ? u / NODES_A : u / NODES_L;
        const int node = in_a ? u - r * NODES_A : NODES_A + u - r * NODES_L;
        const size_t row = first + r;
        if (row < n_rows) {
            const float p = s.k[row];
            if (pt::mt_valid(p)) {   // the others take the exact terms per point
                const float3 w = band_weights(s.ld, row);
                const int i = node / pt::MT_Q, q = node - i * pt::MT_Q;
                float le, ld, ed;
                pt::mt_node(p, i, q, &le, &ld, &ed);
                sF[r][i * (pt::MT_Q + 1) + q] = w.x * le + w.y * ld + w.z * ed;
            }
        }
    }
    __syncthreads();
    {
        const int c = tid / (PREP_ROWS * pt::MT_N), u = tid - c * (PREP_ROWS * pt::MT_N);
        const int r = u / pt::MT_N, i = u - r * pt::MT_N;
        const size_t row = first + r;
        if (row < n_rows && pt::mt_valid(s.k[row]))
            s.rows[row * pt::MT_ROW + 8 * i + c] = pt::mt_coef(i, c, sF[r] + i * (pt::MT_Q + 1));
    }
}
static_assert(PREP % 32 == 0 && PREP_ROWS * pt::MT_NA * pt::MT_Q % 32 == 0, "whole warps in region A");

// Can a time in [tmin, tmax] lie in the transit window of some epoch?  The
// interval is widened by m, 1e-6 of the magnitudes involved, above the FP32
// rounding of these expressions, so the test never misses an epoch.
__device__ __forceinline__ bool tile_meets_window(const GeomRec &g, float tmin, float tmax)
{
    if (g.win_lo > g.win_hi) return false;                // never in transit
    if (g.win_hi - g.win_lo >= 0.5f * g.Ph) return true;  // a wide window: no test
    const float m = 1e-6f * (fabsf(tmin) + fabsf(tmax) + fabsf(g.t0h) + g.Ph) + 1e-9f;
    const float n_lo = ceilf((tmin - g.t0h - g.win_hi - m) * g.invP);
    const float n_hi = floorf((tmax - g.t0h - g.win_lo + m) * g.invP);
    return !(n_lo > n_hi);
}

// A 16-byte shared-memory load at this place: the passbands' constants are
// loop-invariant, and left to itself the compiler keeps all of a group's 64
// of them in registers and spills.
__device__ __forceinline__ float4 lds_here(const float4 *p)
{
    float4 v;
    asm volatile("ld.shared.v4.f32 {%0, %1, %2, %3}, [%4];"
                 : "=f"(v.x), "=f"(v.y), "=f"(v.z), "=f"(v.w)
                 : "r"((unsigned)__cvta_generic_to_shared(p)));
    return v;
}

// The passbands `mask` of an item's group that have no row table (the radius ratio
// outside mt_valid, or all of them in a plan with too few points for tables): the
// exact terms per point.  A chunk of TT times at a time: the in-window ones are listed in
// order with their separations, and the warps take (passband, part of the list)
// tasks, a lane per unit, so that lanes stay full and one orbit solution serves
// all passbands (with supersamples each unit solves its own).  Sums are formed
// per task, in order.  (A passband at a time over all the threads' times, as
// before, 1,000 walkers x 16 passbands x 300 times took 174 us, 57 now; x 9,000
// times at k = 0.7 1,723, 966 now.)
template <int TT>
struct ExactSmem {
    int at[2][TT];             // times of the chunk: in the window, outside it in a tile that meets it
    float dt[TT], z[TT];       // of the in-window ones
    int cnt[2][TT / 32];
    int band[BG];
    float sum[BG];             // one per task
};

template <int TT>
__device__ __forceinline__ int exact_item(const BatchArgs &A, const GeomRec &g, int v, int b0, unsigned mask, int slice,
                                          ExactSmem<TT> &S)
{
    constexpr int NW = TT / 32, TPP = TT / BT;
    const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
    const int nb = __popc(mask), n_seg = max(1, NW / nb), n_task = nb * n_seg;   // (n_task <= BG: nb, or up to NW <= 8)
    const float inv_ss = 1.0f / (float)A.n_ss;
    const int t_end = min(A.n_tiles, (slice + 1) * A.tiles_per_slice);
    if (tid < BG) {
        S.sum[tid] = 0.0f;
        if ((mask >> tid) & 1u) S.band[__popc(mask & ((1u << tid) - 1u))] = b0 + tid;
    }
    int nbad = 0;
#pragma unroll 1
    for (int c0 = slice * A.tiles_per_slice; c0 < t_end; c0 += TPP) {
        const int tj = c0 + tid / BT;
        int i = -1;            // this thread's time
        bool meets = false, in = false;
        float dt = 0.0f, z = 0.0f;
        if (tj < t_end) {
            const float2 mm = A.tile_mm[tj];
            const int2 tl = A.tiles[tj];
            if ((tid & (BT - 1)) < tl.y) i = tl.x + (tid & (BT - 1));
            meets = tile_meets_window(g, mm.x, mm.y);
            if (meets && i >= 0) {
                const float2 ts = A.tsplit[i];
                dt = pt::reduce_time(ts.x, ts.y, g);
                in = dt >= g.win_lo && dt <= g.win_hi;
            }
        }
        if (in && A.n_ss == 1) {
            bool bad = false;
            z = pt::orbit_z<true>(g, dt, A.max_iter, &bad);
            if (bad) ++nbad;
        }
        if (A.flux && i >= 0 && !in)
            for (unsigned m = mask; m; m &= m - 1u) A.flux[((size_t)v * A.n_b + b0 + __ffs(m) - 1) * A.n_t + i] = 1.0f;
        // tiles that do not meet the window: their residuals are in the base (a lane each)
        const unsigned skipped = __ballot_sync(0xffffffffu, tj < t_end && !meets && (tid & (BT - 1)) == 0);
        const unsigned bin = __ballot_sync(0xffffffffu, in), bout = __ballot_sync(0xffffffffu, meets && i >= 0 && !in);
        __syncthreads();   // the previous chunk is no longer read
        if (lane == 0) {
            S.cnt[0][warp] = __popc(bin) | (skipped ? 1 << 16 : 0);
            S.cnt[1][warp] = __popc(bout);
        }
        __syncthreads();
        int at0 = 0, at1 = 0, n_in = 0, n_out = 0;
        unsigned skip = 0u;    // bit w: warp w's first tile is skipped (BT / 32 warps per tile)
#pragma unroll
        for (int w = 0; w < NW; ++w) {
            const int c = S.cnt[0][w] & 0xffff;
            skip |= S.cnt[0][w] >> 16 ? 1u << w : 0u;
            at0 += w < warp ? c : 0;
            at1 += w < warp ? S.cnt[1][w] : 0;
            n_in += c;
            n_out += S.cnt[1][w];
        }
        const unsigned below = (1u << lane) - 1u;
        if (in) {
            at0 += __popc(bin & below);
            S.at[0][at0] = i;
            S.dt[at0] = dt;
            S.z[at0] = z;
        } else if (meets && i >= 0) {
            S.at[1][at1 + __popc(bout & below)] = i;
        }
        __syncthreads();
#pragma unroll 1
        for (int task = warp; task < n_task; task += NW) {
            const int jj = task / n_seg, seg = task - jj * n_seg, b = S.band[jj];
            const size_t row = (size_t)v * A.n_b + b;
            float acc = 0.0f;
            if (A.ssr_part) {
                if (seg == 0 && lane < NW && (skip >> lane) & 1u) acc = A.base[(size_t)b * A.n_tiles + c0 + lane / (BT / 32)];
                const float *y = A.y + (size_t)b * A.n_t, *wt = A.wt + (size_t)b * A.n_t;
                for (int q = seg * 32 + lane; q < n_out; q += 32 * n_seg) {
                    const int at = S.at[1][q];
                    const float r = y[at] - 1.0f;
                    acc = fmaf((A.wt ? wt[at] : 1.0f) * r, r, acc);
                }
            }
            const float k = A.k[row];
            const float3 w = band_weights(A.ld, row);
#pragma unroll 1
            for (int q = seg * 32 + lane; q < n_in; q += 32 * n_seg) {
                float dep = 0.0f;
                float warm[4] = {__int_as_float(0x7fffffff), 0.0f, 0.0f, 0.0f};   // Kepler warm start (none yet)
#pragma unroll 1
                for (int s = 0; s < A.n_ss; ++s) {
                    float zs = S.z[q];
                    if (A.n_ss > 1) {
                        bool bad = false;
                        zs = pt::orbit_z<true>(g, S.dt[q] + A.t_exp * (((float)s + 0.5f) * inv_ss - 0.5f), A.max_iter, &bad, warm);
                        if (bad && jj == 0) ++nbad;   // every passband solves the same orbit
                    }
                    float le, ld, ed;
                    pt::ma_terms(k, zs, &le, &ld, &ed);
                    dep += w.x * le + w.y * ld + w.z * ed;
                }
                dep = __fmul_rn(dep, inv_ss);
                const int at = S.at[0][q];
                if (A.flux) A.flux[row * A.n_t + at] = 1.0f - dep;
                if (A.ssr_part) {
                    const float r = (A.y[(size_t)b * A.n_t + at] - 1.0f) + dep;
                    acc = fmaf((A.wt ? A.wt[(size_t)b * A.n_t + at] : 1.0f) * r, r, acc);
                }
            }
            if (A.ssr_part) {
#pragma unroll
                for (int o = 16; o > 0; o >>= 1) acc += __shfl_xor_sync(0xffffffffu, acc, o);
                if (lane == 0) S.sum[task] += acc;
            }
        }
    }
    if (A.ssr_part) {
        __syncthreads();
        if (tid < nb) {
            float x = 0.0f;
            for (int s = 0; s < n_seg; ++s) x += S.sum[tid * n_seg + s];
            A.ssr_part[((size_t)v * A.n_b + S.band[tid]) * A.n_slices + slice] = x;
        }
    }
    __syncthreads();
    return nbad;
}

// The warp's sums of 16 values per lane, value j on lanes 2 j and 2 j + 1: at each
// level of the tree half the lanes keep half of the values (16 shuffles for 80).
__device__ __forceinline__ float warp_sums(const float (&v)[BG])
{
    static_assert(BG == 16, "a value per pair of lanes");
    const int lane = threadIdx.x & 31;
    float a[8], b[4], c[2];
#pragma unroll
    for (int i = 0; i < 8; ++i)
        a[i] = (lane & 16 ? v[8 + i] : v[i]) + __shfl_xor_sync(0xffffffffu, lane & 16 ? v[i] : v[8 + i], 16);
#pragma unroll
    for (int i = 0; i < 4; ++i)
        b[i] = (lane & 8 ? a[4 + i] : a[i]) + __shfl_xor_sync(0xffffffffu, lane & 8 ? a[i] : a[4 + i], 8);
#pragma unroll
    for (int i = 0; i < 2; ++i)
        c[i] = (lane & 4 ? b[2 + i] : b[i]) + __shfl_xor_sync(0xffffffffu, lane & 4 ? b[i] : b[2 + i], 4);
    const float x = (lane & 2 ? c[1] : c[0]) + __shfl_xor_sync(0xffffffffu, lane & 2 ? c[0] : c[1], 2);
    return x + __shfl_xor_sync(0xffffffffu, x, 1);
}

// ... out of the way of the row tables' kernel
template <int TT>
__device__ __noinline__ int exact_item_call(const BatchArgs *A, const GeomRec *g, int v, int b0, unsigned mask, int slice,
                                            ExactSmem<TT> *S)
{
    return exact_item<TT>(*A, *g, v, b0, mask, slice, *S);
}

// A plan without tables: exact_item on every item.  The terms are a long dependent
// chain, so as many warps as there are registers without spills.
template <int TT>
__global__ void __launch_bounds__(TT, 1024 / TT) batch_exact_kernel(const __grid_constant__ BatchArgs A)
{
    __shared__ GeomRec srec;
    __shared__ ExactSmem<TT> S;
    __shared__ int s_item;
    const int tid = threadIdx.x;
    int nbad = 0;
    for (;;) {
        if (tid == 0) s_item = atomicAdd(A.counter, 1);
        __syncthreads();
        const int it = s_item;
        if (it >= A.n_items) break;
        const int v = it % A.n_v, sg = it / A.n_v;
        const int grp = sg % A.n_groups, slice = sg / A.n_groups;
        const int b0 = grp * A.bg, nb = min(A.bg, A.n_b - b0);
        if (tid < 6) reinterpret_cast<float4 *>(&srec)[tid] = reinterpret_cast<const float4 *>(&A.rec[v])[tid];
        __syncthreads();
        const int bad = exact_item<TT>(A, srec, v, b0, 0xffffffffu >> (32 - nb), slice, S);
        if (grp == 0) nbad += bad;
    }
    if (nbad && A.n_bad) atomicAdd(A.n_bad, nbad);
}

template <int TT, int MODE, bool SS, int OUT>
__global__ void __launch_bounds__(TT, 768 / TT) batch_kernel(const __grid_constant__ BatchArgs A)
{
    extern __shared__ __align__(16) float dyn[];   // M_ROWS: [BG][MT_ROW]; M_INTERP: [BG][mn_z]
    __shared__ GeomRec srec;
    __shared__ float4 sband[BG];   // M_ROWS: k, the scales, valid; M_KHAT: depth weights; others: we, wd, wn, k
    __shared__ ExactSmem<TT> sex;   // M_ROWS
    __shared__ float sred[TT / 32][BG];
    __shared__ int slist[TT], swcnt[TT / 32];
    __shared__ int s_item;
    const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
    constexpr int NW = TT / 32, TPP = TT / BT;   // tiles per pass
    const bool want_ssr = OUT == O_SSR || (OUT == O_ANY && A.ssr_part), want_flux = OUT == O_FLUX || (OUT == O_ANY && A.flux);
    const float inv_ss = 1.0f / (float)A.n_ss;
    const unsigned row_base = pt::mt_base(dyn);   // M_ROWS
    int nbad = 0;
    for (;;) {
        if (tid == 0) s_item = atomicAdd(A.counter, 1);
        __syncthreads();
        const int it = s_item;
        if (it >= A.n_items) break;
        const int v = it % A.n_v;
        const int sg = it / A.n_v;
        const int grp = sg % A.n_groups, slice = sg / A.n_groups;
        const int b0 = grp * A.bg, nb = min(A.bg, A.n_b - b0);
        const size_t row0 = (size_t)v * A.n_b + b0;
        if (tid < 6) reinterpret_cast<float4 *>(&srec)[tid] = reinterpret_cast<const float4 *>(&A.rec[v])[tid];
        // groups of 4 passbands are evaluated together; the last group's
        // padding repeats the item's last passband and is dropped at the stores
        const int nb4 = (nb + 3) & ~3;
        bool row_ok = true;
        if (tid < nb4) {
            const size_t row = row0 + min(tid, nb - 1);
            const float kb = A.k[row];
            const float3 w = band_weights(A.ld, row);
            if (MODE == M_ROWS) {
                float sA = 0.0f, sL = 0.0f;
                row_ok = pt::mt_valid(kb);
                if (row_ok) pt::mt_scales(kb, &sA, &sL);
                sband[tid] = make_float4(kb, sA, sL, row_ok ? 1.0f : 0.0f);
            } else if (MODE == M_KHAT) {
                const float r = kb / A.rec[v].k;
                const float r2 = r * r;
                sband[tid] = make_float4(r2 * w.x, r2 * w.y, r2 * w.z, 0.0f);
            } else {
                sband[tid] = make_float4(w.x, w.y, w.z, kb);
            }
        }
        const int n_without = __syncthreads_count(!row_ok);
        const bool all_ok = n_without == 0, any_ok = n_without < nb4;
        if (MODE == M_ROWS && any_ok) {
            // a row without a table (its radius ratio outside mt_valid) is staged as zeros
            for (int i = tid; i < nb4 * (pt::MT_ROW / 4); i += TT) {
                const int j = i / (pt::MT_ROW / 4);
                float4 c = make_float4(0.0f, 0.0f, 0.0f, 0.0f);
                if (sband[j].w != 0.0f)
                    c = reinterpret_cast<const float4 *>(A.rows + (row0 + min(j, nb - 1)) * pt::MT_ROW)[i - j * (pt::MT_ROW / 4)];
                reinterpret_cast<float4 *>(dyn)[i] = c;
            }
            __syncthreads();
        }
        if (MODE == M_INTERP) {
            // each passband's row of the table: nodes interpolated in k, combined with its weights
            for (int i = tid; i < nb4 * A.mn_z; i += TT) {
                const int b = i / A.mn_z, j = i - b * A.mn_z;
                const float4 w = sband[b];
                const float fk = (fminf(fmaxf(w.w, A.mk_lo), A.mk_hi) - A.mk_lo) * A.minv_dk;
                const int ik = min((int)fk, A.mn_k - 2);
                const float wk = fk - (float)ik;
                const float4 p0 = __ldg(A.mtab + (size_t)ik * A.mn_z + j), p1 = __ldg(A.mtab + (size_t)(ik + 1) * A.mn_z + j);
                dyn[i] = w.x * fmaf(wk, p1.x - p0.x, p0.x) + w.y * fmaf(wk, p1.y - p0.y, p0.y) +
                         w.z * fmaf(wk, p1.z - p0.z, p0.z);
            }
            __syncthreads();
        }
        bool first = true;
        const int t_end = MODE == M_ROWS && !any_ok ? 0 : min(A.n_tiles, (slice + 1) * A.tiles_per_slice);
        for (int c0 = slice * A.tiles_per_slice; c0 < t_end; c0 += TT) {
            float acc[BG];   // residual sums of this chunk: at most BT + 1 terms each
#pragma unroll
            for (int j = 0; j < BG; ++j) acc[j] = 0.0f;
            // one window test per thread; the tiles to evaluate listed in order
            const int jt = c0 + tid;
            bool ev = false;
            if (jt < t_end) {
                const float2 mm = A.tile_mm[jt];
                ev = tile_meets_window(srec, mm.x, mm.y);
                if (!ev && want_ssr) {
                    const float *bp = A.base + (size_t)b0 * A.n_tiles + jt;
#pragma unroll
                    for (int j = 0; j < BG; ++j) {
                        if (j >= nb) break;
                        acc[j] += *bp;
                        bp += A.n_tiles;
                    }
                }
            }
            const unsigned bal = __ballot_sync(0xffffffffu, ev);
            __syncthreads();   // the previous chunk's list is no longer read
            if (lane == 0) swcnt[warp] = __popc(bal);
            __syncthreads();
            int base = 0, n_ev = 0;
#pragma unroll
            for (int w = 0; w < NW; ++w) {
                base += (w < warp) ? swcnt[w] : 0;
                n_ev += swcnt[w];
            }
            if (ev) slist[base + __popc(bal & ((1u << lane) - 1u))] = jt;
            if (want_flux) {
                // flux 1 on the skipped tiles
                const int c1 = min(t_end, c0 + TT);
                for (int tj = c0 + tid / BT; tj < c1; tj += TPP) {
                    const float2 mm = A.tile_mm[tj];
                    const int2 tl = A.tiles[tj];
                    if ((tid & (BT - 1)) < tl.y && !tile_meets_window(srec, mm.x, mm.y)) {
                        float *fp = A.flux + row0 * A.n_t + tl.x + (tid & (BT - 1));
                        for (int j = 0; j < nb; ++j, fp += A.n_t) *fp = 1.0f;
                    }
                }
            }
            __syncthreads();
            for (int q = tid / BT; q < n_ev; q += TPP) {
                const int2 tl = A.tiles[slist[q]];
                if ((tid & (BT - 1)) >= tl.y) continue;
                const int i = tl.x + (tid & (BT - 1));
                const float2 ts = A.tsplit[i];
                float dt = 0.0f;
                bool inw = false;
                if (pt::maybe_in_window(ts.x, srec)) {
                    dt = pt::reduce_time(ts.x, ts.y, srec);
                    inw = dt >= srec.win_lo && dt <= srec.win_hi;
                }
                // observations of the first passbands, on their way during the orbit;
                // element offsets from passband b0's row are 32-bit (the host keeps
                // a group's rows within 2^32 elements)
                const float *yp = A.y + (size_t)b0 * A.n_t, *wp = A.wt + (size_t)b0 * A.n_t;
                float *fp = A.flux + row0 * A.n_t;
                unsigned at_y = (unsigned)i, at = (unsigned)i;
                float yn[4] = {0.0f, 0.0f, 0.0f, 0.0f}, wn[4] = {0.0f, 0.0f, 0.0f, 0.0f};
                auto load4 = [&](int j0) {
                    if (OUT == O_FLUX || !want_ssr) return;
                    if (j0 + 4 <= nb) {
#pragma unroll
                        for (int u = 0; u < 4; ++u) {
                            yn[u] = yp[at_y];
                            if (OUT == O_ANY) wn[u] = A.wt ? wp[at_y] : 1.0f;
                            at_y += (unsigned)A.n_t;
                        }
                    } else {   // a padding passband's sum is dropped
#pragma unroll
                        for (int u = 0; u < 4; ++u) {
                            if (j0 + u < nb) {
                                yn[u] = yp[at_y];
                                if (OUT == O_ANY) wn[u] = A.wt ? wp[at_y] : 1.0f;
                            }
                            at_y += (unsigned)A.n_t;
                        }
                    }
                };
                load4(0);
                // transit depth of passband j at one separation
                float zm1 = 0.0f, off_limb = 0.0f, zz = 0.0f, wz = 0.0f;
                int iz = 0;
                auto at_z = [&](float z) {
                    zz = z;
                    if (MODE == M_ROWS) {
                        zm1 = z - 1.0f;
                        off_limb = pt::mt_off_limb(zm1);
                    } else if (MODE == M_INTERP) {   // cell and weight in z
                        const float fz = fminf(fmaxf(z, 0.0f) * A.minv_dz, (float)(A.mn_z - 1));
                        iz = min((int)fz, A.mn_z - 2);
                        wz = fz - (float)iz;
                    }
                };
                auto depth = [&](int j) {
                    const float4 w = lds_here(sband + j);
                    if (MODE == M_ROWS) {
                        float t;
                        const unsigned bits = pt::mt_find(w.x, w.y, w.z, zm1, off_limb, &t);
                        return pt::mt_eval(row_base + (unsigned)(j * pt::MT_ROW * 4), bits, t);
                    }
                    if (MODE == M_INTERP) {
                        const float *row = dyn + j * A.mn_z + iz;
                        return zz < 1.0f + w.w ? fmaf(wz, row[1] - row[0], row[0]) : 0.0f;
                    }
                    float le, ld, ed;
                    pt::ma_interp(A.mtab, A.mn_k, A.mn_z, A.mk_lo, A.mk_hi, A.minv_dk, A.minv_dz, w.w, zz, &le, &ld, &ed);
                    return w.x * le + w.y * ld + w.z * ed;
                };
                float D[SS && MODE != M_KHAT ? BG : 1];
                float te0 = 0.0f, te1 = 0.0f, te2 = 0.0f;   // M_KHAT: the mean terms with k_hat
                if (!SS) {
                    bool bad = false;
                    const float z = inw ? pt::orbit_z<true>(srec, dt, A.max_iter, &bad) : PT_ZBEHIND;
                    if (bad && grp == 0) ++nbad;   // every group solves the same orbit
                    at_z(z);
                } else {
                    if (MODE != M_KHAT) {
#pragma unroll
                        for (int j = 0; j < BG; ++j) D[MODE != M_KHAT ? j : 0] = 0.0f;
                    }
                    float warm[4] = {__int_as_float(0x7fffffff), 0.0f, 0.0f, 0.0f};   // Kepler warm start (none yet)
#pragma unroll 1
                    for (int s = 0; s < (inw ? A.n_ss : 0); ++s) {
                        bool bad = false;
                        const float z = pt::orbit_z<true>(srec, dt + A.t_exp * (((float)s + 0.5f) * inv_ss - 0.5f),
                                                          A.max_iter, &bad, warm);
                        if (bad && grp == 0) ++nbad;
                        if (MODE == M_KHAT) {
                            float a0, a1, a2;
                            pt::ma_terms(srec.k, z, &a0, &a1, &a2);
                            te0 += a0;
                            te1 += a1;
                            te2 += a2;
                        } else {
                            at_z(z);
#pragma unroll
                            for (int j0 = 0; j0 < BG; j0 += 4) {
                                if (j0 >= nb) break;
#pragma unroll
                                for (int j = j0; j < j0 + 4; ++j) D[MODE != M_KHAT ? j : 0] += depth(j);
                            }
                        }
                    }
                    te0 *= inv_ss;
                    te1 *= inv_ss;
                    te2 *= inv_ss;
                }
#pragma unroll
                for (int j0 = 0; j0 < BG; j0 += 4) {
                    if (j0 >= nb) break;
                    float yc[4], wc[4];
#pragma unroll
                    for (int u = 0; u < 4; ++u) {
                        yc[u] = yn[u];
                        wc[u] = wn[u];
                    }
                    if (j0 + 4 < nb) load4(j0 + 4);
#pragma unroll
                    for (int u = 0; u < 4; ++u) {
                        const int j = j0 + u;
                        float dep;
                        if (MODE == M_KHAT) {
                            const float4 w = lds_here(sband + j);
                            dep = w.x * te0 + w.y * te1 + w.z * te2;
                        }
                        else if (SS) dep = __fmul_rn(D[SS && MODE != M_KHAT ? j : 0], inv_ss);   // rounded the same in every variant
                        else dep = depth(j);
                        if (want_flux && j < nb) fp[at] = 1.0f - dep;
                        at += (unsigned)A.n_t;
                        if (want_ssr) {
                            // y - f with f = 1 - depth not rounded in between
                            const float r = (yc[u] - 1.0f) + dep;
                            acc[j] = fmaf(OUT == O_ANY ? wc[u] * r : r, r, acc[j]);
                        }
                    }
                }
            }
            if (want_ssr) {
                // The chunk's sums go to the warp's: carried on in the registers, a
                // thread's sum would be one chain over the whole slice (4,000 terms
                // at 1e6 times).
                const float x = warp_sums(acc);
                if ((lane & 1) == 0) sred[warp][lane >> 1] = first ? x : sred[warp][lane >> 1] + x;
                first = false;
            }
        }
        if (want_ssr) {
            __syncthreads();
            if (tid < nb) {
                float x = 0.0f;
                if (!first)
                    for (int w = 0; w < NW; ++w) x += sred[w][tid];
                if (MODE != M_ROWS || sband[tid].w != 0.0f) A.ssr_part[(row0 + tid) * A.n_slices + slice] = x;
            }
        }
        if (MODE == M_ROWS && !all_ok) {
            __syncthreads();   // the zero rows' flux is in place
            unsigned mask = 0u;
            for (int j = 0; j < nb; ++j) mask |= sband[j].w == 0.0f ? 1u << j : 0u;
            const int bad = exact_item_call<TT>(&A, &srec, v, b0, mask, slice, &sex);
            if (!any_ok && grp == 0) nbad += bad;   // (else counted by the pass over the rows)
        }
        __syncthreads();   // shared memory is free for the next item
    }
    if (nbad && A.n_bad) atomicAdd(A.n_bad, nbad);
}

__global__ void batch_reduce_kernel(const float *part, int rows, int n_slices, float *ssr)
{
    const int row = blockIdx.x * blockDim.x + threadIdx.x;
    if (row >= rows) return;
    float s = 0.0f;
    for (int i = 0; i < n_slices; ++i) s += part[(size_t)row * n_slices + i];
    ssr[row] = s;
}

}  // namespace

struct pt_batch_plan_s {
    pt_batch_desc d;
    int tt, ctas_per_sm, grid, n_sm;
    int mode;
    int n_tiles, bg, n_groups, n_slices, n_items, max_slices;
    int v_chunk;           // walkers whose row tables exist at a time
    int2 *d_tiles;
    float2 *d_mm;
    float *d_base;
    float *d_rows;
    int *d_counter;
    GeomRec *d_rec;
    float2 *d_tsplit;
    float *d_part;
    cudaGraph_t graph;
    cudaGraphExec_t exec;
    float tuned_ms;
};

namespace {

int berr(cudaError_t e, const char *where)
{
    return pt_internal::set_error(PT_ERR_CUDA, where, cudaGetErrorString(e));
}

using BatchFn = void (*)(BatchArgs);

template <int TT, int MODE, bool SS>
BatchFn batch_fn_o(int out)
{
    return out == O_FLUX ? batch_kernel<TT, MODE, SS, O_FLUX>
           : out == O_SSR ? batch_kernel<TT, MODE, SS, O_SSR>
                          : batch_kernel<TT, MODE, SS, O_ANY>;
}

template <int TT>
BatchFn batch_fn_t(int mode, bool ss, int out)
{
    switch (mode) {
    case M_ROWS: return ss ? batch_fn_o<TT, M_ROWS, true>(out) : batch_fn_o<TT, M_ROWS, false>(out);
    case M_KHAT: return batch_kernel<TT, M_KHAT, true, O_ANY>;
    case M_INTERP: return batch_kernel<TT, M_INTERP, true, O_ANY>;
    case M_EXACT: return batch_exact_kernel<TT>;
    default: return batch_kernel<TT, M_GATHER, true, O_ANY>;
    }
}

BatchFn batch_fn(const pt_batch_plan_s &p, int tt)
{
    const int out = !p.d.ssr ? O_FLUX : (!p.d.flux && !p.d.wt) ? O_SSR : O_ANY;
    const bool ss = p.d.n_ss > 1;
    return tt == 128 ? batch_fn_t<128>(p.mode, ss, out) : batch_fn_t<256>(p.mode, ss, out);
}

static_assert((size_t)BG * pt::MT_ROW * sizeof(float) <= INTERP_SMEM, "one shared-memory limit for all modes");

size_t dyn_smem(const pt_batch_plan_s &p, int n_z)
{
    if (p.mode == M_ROWS) return (size_t)BG * pt::MT_ROW * sizeof(float);
    if (p.mode == M_INTERP) return (size_t)BG * n_z * sizeof(float);
    return 0;
}

int table_args(const pt_batch_desc &d, BatchArgs *A)
{
    A->mtab = nullptr;
    A->mn_k = A->mn_z = 0;
    A->mk_lo = A->mk_hi = A->minv_dk = A->minv_dz = 0.0f;
    if (d.k_mode == 2 && !pt_internal::ma_table_view(d.table, &A->mtab, &A->mn_k, &A->mn_z, &A->mk_lo, &A->mk_hi,
                                                     &A->minv_dk, &A->minv_dz))
        return pt_internal::set_error(PT_ERR_ARG, "pt_batch_run", "k_mode 2 needs an interpolation table");
    return PT_OK;
}

// Enqueue one full evaluation (counter reset, preparation, persistent kernel,
// residual reduction) for the plan's current configuration.
int enqueue(pt_batch_plan_s &p, cudaStream_t s)
{
    const pt_batch_desc &d = p.d;
    cudaError_t e = cudaMemsetAsync(p.d_counter, 0, sizeof(int), s);
    if (e != cudaSuccess) return berr(e, "cudaMemsetAsync");
    // walkers [v0, v0 + n): as many as the row tables hold
    for (int v0 = 0; v0 < d.orb.n_v; v0 += p.v_chunk) {
        const int n = std::min(p.v_chunk, d.orb.n_v - v0);
        const size_t r0 = (size_t)v0 * d.n_b;
        if (v0 > 0) {
            e = cudaMemsetAsync(p.d_counter, 0, sizeof(int), s);
            if (e != cudaSuccess) return berr(e, "cudaMemsetAsync");
        }
        PrepArgs sa;
        sa.t = d.t;
        sa.n_t = d.n_t;
        sa.tsplit = p.d_tsplit;
        sa.orb = d.orb;
        sa.orb.t0 += v0;
        sa.orb.P += v0;
        sa.orb.a += v0;
        sa.orb.inc += v0;
        if (sa.orb.e) sa.orb.e += v0;
        if (sa.orb.w) sa.orb.w += v0;
        sa.orb.n_v = n;
        sa.k = d.k + r0;
        sa.ld = d.ld + 2 * r0;
        sa.khat = d.k_mode == 1;
        sa.n_b = d.n_b;
        sa.half_exp = (float)(0.5 * d.t_exp);
        sa.rec = p.d_rec + v0;
        sa.tiles = p.d_tiles;
        sa.tile_mm = p.d_mm;
        sa.base = p.d_base;
        sa.y = d.y;
        sa.wt = d.wt;
        sa.n_tiles = p.n_tiles;
        sa.rows = p.d_rows;
        sa.n_gblocks = (n + 31) / 32;
        // (the times' share does not depend on the walkers: once)
        sa.n_tblocks = v0 > 0 ? 0 : (p.n_tiles + PREP_TILES - 1) / PREP_TILES;
        const long long per = (long long)(PREP / 32) * PREP_BASE;
        sa.n_bblocks = d.ssr && v0 == 0 ? (int)(((long long)d.n_b * p.n_tiles + per - 1) / per) : 0;
        const long long blocks = (long long)sa.n_gblocks + sa.n_tblocks + sa.n_bblocks +
                                 (p.d_rows ? ((long long)n * d.n_b + PREP_ROWS - 1) / PREP_ROWS : 0);
        batch_prep_kernel<<<(unsigned)blocks, PREP, 0, s>>>(sa);
        e = cudaGetLastError();
        if (e != cudaSuccess) return berr(e, "batch_prep_kernel");
        BatchArgs A;
        int st = table_args(d, &A);
        if (st) return st;
        A.tsplit = p.d_tsplit;
        A.n_t = d.n_t;
        A.rec = p.d_rec + v0;
        A.k = d.k + r0;
        A.ld = d.ld + 2 * r0;
        A.rows = p.d_rows;
        A.tiles = p.d_tiles;
        A.tile_mm = p.d_mm;
        A.base = p.d_base;
        A.n_tiles = p.n_tiles;
        A.n_v = n;
        A.n_b = d.n_b;
        A.n_ss = d.n_ss;
        A.t_exp = (float)d.t_exp;
        A.max_iter = d.max_iter;
        A.y = d.y;
        A.wt = d.wt;
        A.flux = d.flux ? d.flux + r0 * d.n_t : nullptr;
        A.ssr_part = d.ssr ? p.d_part + r0 * p.n_slices : nullptr;
        A.bg = p.bg;
        A.n_groups = p.n_groups;
        A.n_slices = p.n_slices;
        A.tiles_per_slice = (p.n_tiles + p.n_slices - 1) / p.n_slices;
        A.n_items = n * p.n_groups * p.n_slices;
        A.counter = p.d_counter;
        A.n_bad = d.n_bad;
        batch_fn(p, p.tt)<<<std::min(p.grid, A.n_items), p.tt, dyn_smem(p, A.mn_z), s>>>(A);
        e = cudaGetLastError();
        if (e != cudaSuccess) return berr(e, "batch_kernel");
    }
    if (d.ssr) {
        int rows = d.orb.n_v * d.n_b;
        batch_reduce_kernel<<<(rows + 127) / 128, 128, 0, s>>>(p.d_part, rows, p.n_slices, d.ssr);
        e = cudaGetLastError();
        if (e != cudaSuccess) return berr(e, "batch_reduce_kernel");
    }
    return PT_OK;
}

// Slices of the times (an item each per walker and passband group); the
// partial sums are sized for the largest number at creation.
constexpr int MAX_SLICES = 64;

// Row tables from this many points (times x supersamples) per row: a table
// costs 144 evaluations of the exact terms, a row reads it at the in-window
// points, about a third of them in the light curves of transits.  5,000 walkers
// x 16 passbands: 600 times 351 us by the exact terms and 414 from rows, 800 times
// 455 and 435, 1,000 times 563 and 459; 200 times x 3 supersamples 287 and 395.
constexpr int ROWS_MIN_POINTS = 768;

// A plan's row tables are made for this many bytes of walkers at a time (768 bytes
// per walker and passband: 100,000 walkers x 256 passbands would be 20 GB).  A chunk
// still has millions of rows, so the launches between chunks do not show.
constexpr size_t ROWS_MAX_BYTES = (size_t)2 << 30;

int configure(pt_batch_plan_s &p, int tt, int n_slices, int n_z)
{
    const BatchFn fn = batch_fn(p, tt);
    const size_t smem = dyn_smem(p, n_z);
    // (INTERP_SMEM covers every mode's size, and is the same for every plan)
    cudaError_t e = pt::allow_smem(fn, INTERP_SMEM);
    int per_sm = 0;
    if (e == cudaSuccess) e = cudaOccupancyMaxActiveBlocksPerMultiprocessor(&per_sm, fn, tt, smem);
    if (e != cudaSuccess) return berr(e, "batch_kernel occupancy");
    if (per_sm < 1) return pt_internal::set_error(PT_ERR_ARG, "batch_kernel", "does not fit on an SM");
    p.tt = tt;
    p.ctas_per_sm = per_sm;
    p.n_slices = n_slices;
    p.n_items = p.d.orb.n_v * p.n_groups * n_slices;
    p.grid = std::min(per_sm * p.n_sm, p.n_items);
    return PT_OK;
}

void free_plan(pt_batch_plan_s *p)
{
    if (!p) return;
    if (p->exec) cudaGraphExecDestroy(p->exec);
    if (p->graph) cudaGraphDestroy(p->graph);
    cudaFree(p->d_tiles);
    cudaFree(p->d_mm);
    cudaFree(p->d_base);
    cudaFree(p->d_rows);
    cudaFree(p->d_counter);
    cudaFree(p->d_rec);
    cudaFree(p->d_tsplit);
    cudaFree(p->d_part);
    delete p;
}

}  // namespace

extern "C" {

int pt_batch_plan_create(const pt_batch_desc *d, int autotune, pt_batch_plan *out)
{
    if (!d || !out) return PT_ERR_ARG;
    *out = nullptr;
    const pt_orbit &o = d->orb;
    if (o.n_v < 1 || d->n_t < 1 || d->n_lc < 1 || d->n_b < 1 || d->n_b > 256 || d->n_ss < 1 || d->n_ss > 256 ||
        d->max_iter < 1 || d->max_iter > 64)
        return PT_ERR_ARG;
    if (!d->t || !d->lc_offsets || !o.t0 || !o.P || !o.a || !o.inc || !d->k || !d->ld) return PT_ERR_ARG;
    if ((o.e == nullptr) != (o.w == nullptr)) return PT_ERR_ARG;
    if (!d->flux && !d->ssr) return PT_ERR_ARG;
    if (d->k_mode < 0 || d->k_mode > 2) return PT_ERR_ARG;
    if ((d->k_mode == 2) != (d->table != nullptr)) return PT_ERR_ARG;
    if (d->ssr && !d->y) return PT_ERR_ARG;
    if (!(d->t_exp >= 0.0 && d->t_exp < 1.0e30))
        return pt_internal::set_error(PT_ERR_DOMAIN, "pt_batch_plan_create", "exposure time must be finite and >= 0");
    if (d->lc_offsets[0] != 0 || d->lc_offsets[d->n_lc] != d->n_t) return PT_ERR_ARG;
    for (int j = 0; j < d->n_lc; ++j)
        if (d->lc_offsets[j + 1] < d->lc_offsets[j]) return PT_ERR_ARG;
    const long long n_rows = (long long)o.n_v * d->n_b;
    pt_batch_plan_s *p = new pt_batch_plan_s();
    p->d = *d;
    p->d.lc_offsets = nullptr;
    int dev = 0;
    cudaGetDevice(&dev);
    cudaDeviceGetAttribute(&p->n_sm, cudaDevAttrMultiProcessorCount, dev);
    BatchArgs tab;
    int st = table_args(*d, &tab);
    if (st) {
        free_plan(p);
        return st;
    }
    // rows of the caller's table are staged in shared memory while a group fits
    p->mode = d->k_mode == 0 ? ((long long)d->n_t * d->n_ss >= ROWS_MIN_POINTS ? M_ROWS : M_EXACT)
              : d->k_mode == 1 ? M_KHAT
              : (size_t)BG * tab.mn_z * sizeof(float) <= INTERP_SMEM ? M_INTERP : M_GATHER;
    // tiles of BT times within each light curve
    std::vector<int2> tiles;
    for (int j = 0; j < d->n_lc; ++j)
        for (int s = d->lc_offsets[j]; s < d->lc_offsets[j + 1]; s += BT)
            tiles.push_back(make_int2(s, std::min(BT, d->lc_offsets[j + 1] - s)));
    p->n_tiles = (int)tiles.size();
    const bool tables = p->mode == M_ROWS;
    p->bg = d->n_t <= (1 << 28) ? BG : 1;   // a group's observations within 32-bit offsets
    p->n_groups = (d->n_b + p->bg - 1) / p->bg;
    // many rows need no slices: bounds the partial sums
    p->max_slices = (int)std::max(1LL, std::min((long long)MAX_SLICES, (1LL << 26) / n_rows));
    cudaError_t e = cudaMalloc(&p->d_counter, sizeof(int));
    if (e == cudaSuccess) e = cudaMalloc(&p->d_rec, (size_t)o.n_v * sizeof(GeomRec));
    if (e == cudaSuccess) e = cudaMalloc(&p->d_tsplit, (size_t)d->n_t * sizeof(float2));
    if (e == cudaSuccess) e = cudaMalloc(&p->d_tiles, tiles.size() * sizeof(int2));
    if (e == cudaSuccess) e = cudaMalloc(&p->d_mm, tiles.size() * sizeof(float2));
    if (e == cudaSuccess && d->ssr) e = cudaMalloc(&p->d_base, (size_t)d->n_b * tiles.size() * sizeof(float));
    if (e == cudaSuccess && d->ssr) e = cudaMalloc(&p->d_part, (size_t)n_rows * p->max_slices * sizeof(float));
    // row tables of as many walkers as ROWS_MAX_BYTES hold, in equal chunks
    p->v_chunk = o.n_v;
    if (tables) {
        const long long cap = std::max(1LL, (long long)(ROWS_MAX_BYTES / ((size_t)d->n_b * pt::MT_ROW * sizeof(float))));
        const long long n_chunk = (o.n_v + cap - 1) / cap;
        p->v_chunk = (int)((o.n_v + n_chunk - 1) / n_chunk);
        const size_t bytes = (size_t)p->v_chunk * d->n_b * pt::MT_ROW * sizeof(float);
        if (e == cudaSuccess) e = cudaMalloc(&p->d_rows, bytes);
        // (the two unused floats per interval are staged with the others)
        if (e == cudaSuccess) e = cudaMemset(p->d_rows, 0, bytes);
    }
    if (e == cudaSuccess) e = cudaMemcpy(p->d_tiles, tiles.data(), tiles.size() * sizeof(int2), cudaMemcpyHostToDevice);
    if (e != cudaSuccess) {
        st = berr(e, "pt_batch_plan_create");
        free_plan(p);
        return st;
    }
    cudaStream_t cs;
    e = cudaStreamCreateWithFlags(&cs, cudaStreamNonBlocking);
    if (e != cudaSuccess) {
        st = berr(e, "cudaStreamCreate");
        free_plan(p);
        return st;
    }
    // autotuner: CTA size x slices of the times, timed on the caller's
    // buffers.  The fewest slices tried give every resident CTA about an
    // item (or a chunk of tiles per slice, if there are too few tiles).
    const int tts[2] = {256, 128};
    const long long base_items = (long long)o.n_v * p->n_groups;
    int best_tt = 0, best_sl = 1;
    float best = 1e30f;
    cudaEvent_t e0, e1;
    cudaEventCreate(&e0);
    cudaEventCreate(&e1);
    for (int ti = 0; ti < 2 && st == PT_OK; ++ti) {
        const int tt = tts[ti];
        if (!autotune && ti > 0) break;
        st = configure(*p, tt, 1, tab.mn_z);
        if (st) break;
        const int sl_max = std::max(1, std::min(p->max_slices, p->n_tiles / (tt / BT)));
        int sl0 = 1;
        while (sl0 < sl_max && base_items * sl0 < (long long)p->n_sm * p->ctas_per_sm) sl0 *= 2;
        for (int f = 1; f <= (autotune ? 8 : 1) && st == PT_OK; f *= 2) {
            const int sl = std::min(sl0 * f, sl_max);
            if (f > 1 && (sl0 * (f / 2) >= sl_max)) break;
            st = configure(*p, tt, sl, tab.mn_z);
            if (st) break;
            st = enqueue(*p, cs);   // warm-up
            if (st) break;
            float ms_tot = 0.0f;
            const int reps = autotune ? 2 : 1;
            for (int r = 0; r < reps && st == PT_OK; ++r) {
                cudaEventRecord(e0, cs);
                st = enqueue(*p, cs);
                cudaEventRecord(e1, cs);
                cudaEventSynchronize(e1);
                float ms = 0.0f;
                cudaEventElapsedTime(&ms, e0, e1);
                ms_tot += ms;
            }
            float ms = ms_tot / reps;
            if (st == PT_OK && ms < best) {
                best = ms;
                best_tt = tt;
                best_sl = sl;
            }
        }
    }
    cudaEventDestroy(e0);
    cudaEventDestroy(e1);
    if (st == PT_OK && best_tt == 0) st = PT_ERR_ARG;
    if (st == PT_OK) st = configure(*p, best_tt, best_sl, tab.mn_z);
    if (st == PT_OK) {
        e = cudaStreamSynchronize(cs);
        if (e != cudaSuccess) st = berr(e, "autotune");
    }
    p->tuned_ms = best;
    // capture the evaluation into a graph
    if (st == PT_OK) {
        e = cudaStreamBeginCapture(cs, cudaStreamCaptureModeThreadLocal);
        if (e != cudaSuccess) st = berr(e, "cudaStreamBeginCapture");
        if (st == PT_OK) {
            int st2 = enqueue(*p, cs);
            e = cudaStreamEndCapture(cs, &p->graph);
            if (st2) st = st2;
            else if (e != cudaSuccess) st = berr(e, "cudaStreamEndCapture");
        }
        if (st == PT_OK) {
            e = cudaGraphInstantiate(&p->exec, p->graph, 0);
            if (e != cudaSuccess) st = berr(e, "cudaGraphInstantiate");
        }
    }
    cudaStreamDestroy(cs);
    if (st) {
        free_plan(p);
        return st;
    }
    *out = p;
    return PT_OK;
}

int pt_batch_run(pt_batch_plan p, pt_stream_t stream)
{
    if (!p || !p->exec) return PT_ERR_ARG;
    cudaError_t e = cudaGraphLaunch(p->exec, (cudaStream_t)stream);
    return e == cudaSuccess ? PT_OK : berr(e, "cudaGraphLaunch");
}

int pt_batch_plan_info(pt_batch_plan p, int *tile, int *ctas_per_sm, int *n_items, float *tuned_ms)
{
    if (!p) return PT_ERR_ARG;
    if (tile) *tile = p->tt;
    if (ctas_per_sm) *ctas_per_sm = p->ctas_per_sm;
    if (n_items) *n_items = p->n_items;
    if (tuned_ms) *tuned_ms = p->tuned_ms;
    return PT_OK;
}

int pt_batch_plan_destroy(pt_batch_plan p)
{
    free_plan(p);
    return PT_OK;
}

}  // extern "C"
