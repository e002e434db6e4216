// pt_rows.cuh -- light curves from row tables: one kernel for every model.
//
// A light-curve call evaluates each geometry (orbit and radius ratio) at
// thousands of separations, so a preparation kernel first tabulates, per
// geometry and passband, the transit depth as a function of the separation
// (a "row"), and lc_rows_kernel does the rest in one pass:
//   - a CTA covers VT geometries x KT blocks of 256 times (VT KT <= 32, one
//     bit per (geometry, block) of a thread); it stages the geometries'
//     records and rows in shared memory;
//   - window test of every pair in plain FP32 with a margin; the pairs that
//     pass go to one list per geometry in shared memory; every flux is set
//     to 1;
//   - each lane takes a listed pair (the lists end to end, so that lanes stay
//     full), reduces its time in double-float (a pair beyond the exact window
//     keeps depth 0), solves the orbit at its supersamples and reads the
//     pair's rows there, up to NRT of them at once (1, 4 or 9: the orbit is
//     solved once for all of a geometry's rows but the 10 to 17 of a high-order
//     Gimenez law with many passbands); mean, flux, residual;
//   - residual sums per block of 256 times, in an order fixed by n_t alone: a
//     vector's sum does not depend on the other vectors of its call.
// The place of a pair in its list is not determined, but no value depends on
// it, so results are reproducible bit by bit.
// The rows and what a look-up does are the model's:
//   R_MA      piecewise polynomials in the distance to the contacts
//             (pt_device.cuh); the exact terms where a geometry has none;
//   R_GIM     piecewise polynomials of the Gimenez series;
//   R_ZI      Gimenez on z nodes (Sec. 3.3), linear;
//   R_INTERP  the Mandel-Agol table at the geometry's k (Sec. 2.2.3), linear.
// Before, the path was a set-up, a window kernel writing pair lists to memory,
// a scan, and an evaluation kernel per model that solved Kepler's equation for
// every supersample, packed the in-transit ones and evaluated the terms for
// each.  50,000 times x 256 eccentric vectors x 10 supersamples: Mandel-Agol
// 85.4 -> 45.9 us a call, from the caller's table 109 -> 43.8 us; 3,001 times x
// 800 circular geometries x 3, residual sums: 75.8 -> 38.9 us.  What bounds it:
// issue (about 67 %), two thirds of the instructions in the window test, the
// lists and the stores of a survey's mostly empty pairs.
#pragma once

#include "pt_device.cuh"

namespace rows {

using pt::GeomRec;

enum Model { R_MA = 0, R_GIM = 1, R_ZI = 2, R_INTERP = 3 };

constexpr int TB = 256;          // times per block of a tile, threads per CTA
constexpr int NW = TB / 32;
constexpr int MAX_BITS = 32;     // VT KT
constexpr int MAX_BAND_ROWS = 8; // passbands of a geometry with a row each; more share the rows of the terms

struct Args {
    const float2 *tsplit;
    int n_t;
    const GeomRec *rec;
    int n_geom;
    const float *rows;      // [n_geom][nr][row_len]
    int row_len;            // floats, a multiple of 4
    int nr;                 // rows per geometry
    int terms;              // rows hold the model's terms, combined per passband with its weights
    const float *wts;       // these weights, [n_geom n_bpg][nr]
    int n_bpg, n_b, k_per_band;
    const float *ld;        // [n_geom n_bpg][2], R_MA
    int n_ss;
    float t_exp;
    int max_iter;
    float *flux;            // [n_geom n_bpg][n_t] or null
    float *ssr_part;        // [n_geom n_bpg][n_blk] or null (needs !terms)
    int n_tiles, tile0;
    int n_blk;              // blocks of TB times
    const float *y, *wt;
    int *n_bad;
    int log_vt, log_kt;
    int flux_vec;           // 16-byte stores of whole rows are aligned
    float scale;            // R_GIM
    int n_in, n_edge;       // R_ZI
    float inv_dz;           // R_INTERP
    int n_z;
};

// The exact Mandel-Agol terms of a geometry without a table.
__device__ __noinline__ float3 exact_terms(float k, float z)
{
    float3 t;
    pt::ma_terms(k, z, &t.x, &t.y, &t.z);
    return t;
}

// A look-up: the place in the row and the offset from it.
template <int MODEL>
__device__ __forceinline__ unsigned find(const Args &A, const float4 &q, float z, float *t)
{
    if (MODEL == R_MA) {
        const float zm1 = z - 1.0f;
        return pt::mt_find(q.x, q.y, q.z, zm1, pt::mt_off_limb(zm1), t);
    }
    if (MODEL == R_GIM) {
        // u = sqrt(1 - z / (1 + k)), 0 at and beyond the contact
        const float u = pt::sqrt_a(__saturatef((q.x - (z - 1.0f)) * q.y));
        const float b = fmaf(u, A.scale, pt::MT_MAGIC);
        *t = fmaf(u, A.scale, pt::MT_MAGIC - b);
        return __float_as_uint(b);
    }
    if (MODEL == R_ZI) {   // q: k, zb, 1 / h1 (0: the first region is z = 0), 1 / h2
        if (z <= q.y) {
            const float f = z * q.z;
            const int i = q.z > 0.0f ? min((int)f, A.n_in - 2) : 0;
            *t = q.z > 0.0f ? f - (float)i : 0.0f;
            return (unsigned)i;
        }
        const float f = fminf((z - q.y) * q.w, 1e9f);
        const int c = min((int)f, A.n_edge - 1);
        *t = f - (float)c;
        return (unsigned)(A.n_in - 1 + c);
    }
    const float f = fminf(fmaxf(z, 0.0f) * A.inv_dz, (float)(A.n_z - 1));
    const int i = min((int)f, A.n_z - 2);
    *t = f - (float)i;
    return (unsigned)i;
}

constexpr int GIM_DEG = 8;   // coefficients per interval of a Gimenez row

// base: byte address in shared memory (SMEM) of the row, less the place's
// constant bits; or the row in global memory
template <int MODEL, bool SMEM>
__device__ __forceinline__ float eval(unsigned base, const float *row, const float4 &q, float z, unsigned pos, float t)
{
    if (MODEL == R_MA && SMEM) return pt::mt_eval(base, pos, t);
    if (MODEL == R_GIM || MODEL == R_MA) {
        // (8 floats per interval in both)
        float4 c, d;
        if (SMEM) {
            const unsigned at = base + 32u * pos;
            asm volatile("ld.shared.v4.f32 {%0, %1, %2, %3}, [%4];" : "=f"(c.x), "=f"(c.y), "=f"(c.z), "=f"(c.w) : "r"(at));
            asm volatile("ld.shared.v4.f32 {%0, %1, %2, %3}, [%4];" : "=f"(d.x), "=f"(d.y), "=f"(d.z), "=f"(d.w) : "r"(at + 16u));
        } else {
            const float4 *p = reinterpret_cast<const float4 *>(row + (size_t)(pos - pt::MT_BITS0) * 8);
            c = *p;
            d = p[1];
        }
        float v = MODEL == R_GIM ? fmaf(fmaf(d.w, t, d.z), t, d.y) : d.y;
        v = fmaf(v, t, d.x);
        v = fmaf(v, t, c.w);
        v = fmaf(v, t, c.z);
        v = fmaf(v, t, c.y);
        return fmaf(v, t, c.x);
    }
    float a, b;
    if (SMEM) {
        const unsigned at = base + 4u * pos;
        asm volatile("ld.shared.f32 %0, [%1];" : "=f"(a) : "r"(at));
        asm volatile("ld.shared.f32 %0, [%1];" : "=f"(b) : "r"(at + 4u));
    } else {
        a = row[pos];
        b = row[pos + 1];
    }
    return z < 1.0f + q.x ? fmaf(t, b - a, a) : 0.0f;
}

// constants of a geometry's look-ups
template <int MODEL>
__device__ __forceinline__ float4 look_up_constants(const Args &A, float k)
{
    float4 q = make_float4(k, 0.0f, 0.0f, 1.0f);
    if (MODEL == R_MA) {
        if (pt::mt_valid(k)) pt::mt_scales(k, &q.y, &q.z);
        else q.w = 0.0f;
    } else if (MODEL == R_GIM) {
        q.y = 1.0f / (1.0f + k);
    } else if (MODEL == R_ZI) {
        q.y = fmaxf(1.0f - k, 0.0f);
        q.z = q.y > 0.0f ? 1.0f / (q.y / (float)(A.n_in - 1)) : 0.0f;
        q.w = 1.0f / ((1.0f + k - q.y) / (float)A.n_edge);
    }
    return q;
}

struct Smem {   // byte offsets in dynamic shared memory
    int list, rows, sval, sred, total;
};

__host__ __device__ inline Smem smem_layout(int vt, int log_kt, int nr, int row_len, bool staged, int n_ssr)
{
    Smem s;
    const int pairs = vt * (TB << log_kt);
    int off = 0;
    s.list = off;
    off += pairs * 2;
    s.rows = off;
    if (staged) off += vt * nr * row_len * 4;
    s.sval = off;
    off += n_ssr * pairs * 4;
    s.sred = off;
    off += NW * (vt << log_kt) * n_ssr * 4;
    s.total = off;
    return s;
}

template <int MODEL, int NRT, bool SMEM>
__global__ void __launch_bounds__(TB, 4) lc_rows_kernel(Args A)
{
    pt::chain_begin();
    extern __shared__ __align__(16) unsigned char dsm[];
    __shared__ GeomRec srec[MAX_BITS];
    __shared__ float4 stest[MAX_BITS];   // 1/P, -(t0 + window centre)/P, half width + margin (periods)
    __shared__ float4 sgeo[MAX_BITS];    // constants of the look-ups
    __shared__ int sband[MAX_BITS];      // passband of each geometry's data
    __shared__ int scnt[MAX_BITS];       // pairs of each geometry
    __shared__ int soff[MAX_BITS + 1];   // ... before each geometry, lists end to end
    __shared__ float swmax[NW];
    __shared__ bool sexact;              // R_MA: a geometry without a table
    const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
    const int log_vt = A.log_vt, vt = 1 << log_vt, log_kt = A.log_kt, kt = 1 << log_kt;
    const int tile = A.tile0 + blockIdx.y;
    const int g0 = blockIdx.x << log_vt;
    const int ng = min(vt, A.n_geom - g0);
    const int tb = tile * (TB << log_kt);
    const int n_ssr = A.ssr_part ? A.nr : 0;
    const Smem L = smem_layout(vt, log_kt, A.nr, A.row_len, SMEM, n_ssr);
    const int cap = TB << log_kt;        // entries of a geometry's list
    unsigned short *list = reinterpret_cast<unsigned short *>(dsm + L.list);   // [vt][cap]: k TB + thread
    for (int i = tid; i < ng * 6; i += TB) {
        const int vl = i / 6, c = i - 6 * vl;
        reinterpret_cast<float4 *>(&srec[vl])[c] = reinterpret_cast<const float4 *>(&A.rec[g0 + vl])[c];
    }
    if (SMEM) {
        const float4 *src = reinterpret_cast<const float4 *>(A.rows + (size_t)g0 * A.nr * A.row_len);
        const unsigned dst = (unsigned)__cvta_generic_to_shared(dsm + L.rows);
        const int n4 = ng * A.nr * A.row_len / 4;
        for (int i = tid; i < n4; i += TB)
            asm volatile("cp.async.cg.shared.global [%0], [%1], 16;" ::"r"(dst + 16u * i), "l"(src + i) : "memory");
        asm volatile("cp.async.commit_group;" ::: "memory");
    }
    if (tid < MAX_BITS) scnt[tid] = 0;
    if (tid == 0) sexact = false;
    // the tile's largest |t_h| (non-negative floats order like their bits)
    float am = 0.0f;
    for (int k = 0; k < kt; ++k) {
        const int t = tb + k * TB + tid;
        if (t < A.n_t) am = fmaxf(am, fabsf(A.tsplit[t].x));
    }
    am = __int_as_float(__reduce_max_sync(0xffffffffu, __float_as_int(am)));
    if (lane == 0) swmax[warp] = am;
    __syncthreads();
    if (tid < MAX_BITS) stest[tid] = make_float4(0.0f, 0.0f, -1.0f, 0.0f);   // beyond the last geometry: never
    if (tid < ng) {
        float tmax = swmax[0];
        for (int w = 1; w < NW; ++w) tmax = fmaxf(tmax, swmax[w]);
        const GeomRec &r = srec[tid];
        // The test is in periods from the window's centre, one FMA: off by less
        // than 5 roundings of the magnitudes involved (the products with the
        // rounded 1/P, the low parts of t, t0 and P, the sum).  Where that is
        // no small part of a period, every pair is listed.
        const float mid = 0.5f * (r.win_lo + r.win_hi);
        const float m = 3.0e-7f * (tmax + fabsf(r.t0h) + fabsf(mid) + r.Ph) * r.invP + 1e-7f;
        float half = 0.5f * (r.win_hi - r.win_lo) * r.invP * 1.000001f + m;
        if (r.win_lo > r.win_hi) half = -1.0f;
        else if (!(m < 0.25f)) half = INFINITY;
        stest[tid] = make_float4(r.invP, -(r.t0h + mid) * r.invP, half, 0.0f);
        sgeo[tid] = look_up_constants<MODEL>(A, r.k);
        if (MODEL == R_MA && sgeo[tid].w == 0.0f) sexact = true;
        sband[tid] = A.k_per_band ? (g0 + tid) % A.n_b : 0;
    }
    // every flux of the tile is 1 until its pair is evaluated
    if (A.flux) {
        const int n_row = ng * A.n_bpg, n_tt = min(cap, A.n_t - tb);
        float *fp = A.flux + (size_t)g0 * A.n_bpg * A.n_t + tb;
        if (A.flux_vec) {   // rows and the array start on 16 bytes
            const float4 one = make_float4(1.0f, 1.0f, 1.0f, 1.0f);
            const int n4 = n_tt / 4;   // (n_t, and so n_tt, a multiple of 4)
            for (int r = tid >> 6; r < n_row; r += TB / 64)
                for (int i = tid & 63; i < n4; i += 64) reinterpret_cast<float4 *>(fp + (size_t)r * A.n_t)[i] = one;
        } else {
            for (int r = 0; r < n_row; ++r, fp += A.n_t)
                for (int i = tid; i < n_tt; i += TB) fp[i] = 1.0f;
        }
    }
    __syncthreads();
    unsigned bits = 0u;   // bit k vt + vl: the time of block k may be in geometry vl's window
    for (int k = 0; k < kt; ++k) {
        const int t = tb + k * TB + tid;
        const float th = t < A.n_t ? A.tsplit[t].x : __int_as_float(0x7fffffff);   // NaN: in no window
        unsigned cand = 0u;
        for (int v0 = 0; v0 < vt; v0 += 4) {
            unsigned c4 = 0u;
#pragma unroll
            for (int u = 0; u < 4; ++u) {   // (vt < 4: the entries beyond never pass)
                const float4 q = stest[v0 + u];
                const float ph = fmaf(th, q.x, q.y);
                const float fr = ph - ((ph + pt::MT_MAGIC) - pt::MT_MAGIC);
                c4 |= fabsf(fr) <= q.z ? (1u << u) : 0u;
            }
            cand |= c4 << v0;
        }
        bits |= cand << (k << log_vt);
    }
    {
        // append to the lists: one atomic per warp and geometry where the
        // warp's lanes share geometries (exposures around one planet's
        // transits), one per pair where they do not (survey cadence)
        const unsigned wbits = __reduce_or_sync(0xffffffffu, bits);
        const int wpairs = __reduce_add_sync(0xffffffffu, __popc(bits));
        if (wpairs > 4 * __popc(wbits)) {
            for (unsigned rest = wbits; rest; rest &= rest - 1u) {
                const int p = __ffs(rest) - 1, vl = p & (vt - 1), k = p >> log_vt;
                const bool in = (bits >> p) & 1u;
                const unsigned mb = __ballot_sync(0xffffffffu, in);
                int base = 0;
                if (lane == 0) base = atomicAdd(&scnt[vl], __popc(mb));
                base = __shfl_sync(0xffffffffu, base, 0);
                if (in) list[vl * cap + base + __popc(mb & ((1u << lane) - 1u))] = (unsigned short)(k * TB + tid);
            }
        } else {
            for (unsigned rest = bits; rest; rest &= rest - 1u) {
                const int p = __ffs(rest) - 1, vl = p & (vt - 1), k = p >> log_vt;
                list[vl * cap + atomicAdd(&scnt[vl], 1)] = (unsigned short)(k * TB + tid);
            }
        }
    }
    if (SMEM) asm volatile("cp.async.wait_all;" ::: "memory");
    __syncthreads();
    if (warp == 0) {
        const int v = lane < vt ? scnt[lane] : 0;
        int x = v;
#pragma unroll
        for (int o = 1; o < 32; o <<= 1) {
            const int u = __shfl_up_sync(0xffffffffu, x, o);
            if (lane >= o) x += u;
        }
        if (lane < vt) soff[lane] = x - v;
        if (lane == 31) soff[vt] = x;
    }
    __syncthreads();
    const int nq = soff[vt];
    // the lists end to end, 32 pairs per warp and turn
    const float inv_nss = 1.0f / (float)A.n_ss;
    const unsigned sbase = (unsigned)__cvta_generic_to_shared(dsm + L.rows) -
                           (MODEL == R_MA || MODEL == R_GIM ? 32u * pt::MT_BITS0 : 0u);
    float *sval = reinterpret_cast<float *>(dsm + L.sval);   // [n_ssr][kt vt][TB]
    int nbad = 0;
    auto geometry_of = [&](int e) {   // the last geometry with soff <= e
        int vl = 0;
        for (int o = vt >> 1; o > 0; o >>= 1)
            if (soff[vl + o] <= e) vl += o;
        return vl;
    };
    // a row's depth at the time with this code
    auto emit = [&](int vl, int code, int row, float dep) {
        const int t = tb + code;
        if (A.flux) A.flux[((size_t)(g0 + vl) * A.n_bpg + row) * A.n_t + t] = 1.0f - dep;
        if (n_ssr) {
            const int band = sband[vl] + (A.k_per_band ? 0 : row);
            // y - f with f = 1 - depth not rounded in between
            const float res = (A.y[(size_t)band * A.n_t + t] - 1.0f) + dep;
            const int p = ((code >> 8) << log_vt) + vl;
            sval[((row << (log_vt + log_kt)) + p) * TB + (code & (TB - 1))] =
                (A.wt ? A.wt[(size_t)band * A.n_t + t] : 1.0f) * res * res;
        }
    };
    // f(z) at the supersamples of a pair's exposure (none beyond the window).
    // Kepler's equation once, at mid-exposure; the supersamples from the f and g
    // series at offsets x0 + s dx of mean anomaly, or, where the exposure is too
    // long a part of the period for them, by Newton's method each.
#define PT_EACH_Z(COUNT, F)                                                                                         \
    if (series) {                                                                                                   \
        _Pragma("unroll 1") for (int s = 0; s < n_ss; ++s) F(pt::fg_z(o, fg, cosi, x0 + (float)s * dx));            \
    } else {                                                                                                        \
        float warm[4] = {__int_as_float(0x7fffffff), 0.0f, 0.0f, 0.0f}; /* Kepler warm start (none yet) */          \
        _Pragma("unroll 1") for (int s = 0; s < n_ss; ++s)                                                          \
        {                                                                                                           \
            bool bad = false;                                                                                       \
            const float off = A.t_exp * (((float)s + 0.5f) * inv_nss - 0.5f);                                       \
            const float z = pt::orbit_z<true, true>(r, dt + off, A.max_iter, &bad, warm);                           \
            if (bad && (COUNT)) ++nbad;                                                                             \
            F(z);                                                                                                   \
        }                                                                                                           \
    }
    for (int e = tid; e < nq; e += TB) {
        const int vl = geometry_of(e), code = list[vl * cap + (e - soff[vl])], t = tb + code;
        const GeomRec &r = srec[vl];
        const float4 q = sgeo[vl];
        if (MODEL == R_MA && q.w == 0.0f) continue;   // without a table: below
        const float2 ts = A.tsplit[t];
        const float dt = pt::reduce_time(ts.x, ts.y, r);
        const int n_ss = dt >= r.win_lo && dt <= r.win_hi ? A.n_ss : 0;
        const size_t row0 = (size_t)(g0 + vl) * A.n_bpg;
        pt::OrbitState o;
        bool bad0 = false;
        pt::orbit_state(r, dt, A.max_iter, &bad0, &o);
        const float cosi = r.cosi, dx = A.n_ss > 1 ? r.nang * A.t_exp * inv_nss : 0.0f;
        const float x0 = -0.5f * (float)(A.n_ss - 1) * dx;
        const bool series = pt::fg_valid(r, o.E1, x0);
        const pt::FgSeries fg = pt::fg_series(o.E1, o.esin);
        if (series && bad0) nbad += n_ss;
        float mean[NRT];
#pragma unroll 1
        for (int r0 = 0; r0 < A.nr; r0 += NRT) {
#pragma unroll
            for (int u = 0; u < NRT; ++u) mean[u] = 0.0f;
            const unsigned lbase = sbase + (unsigned)((vl * A.nr + r0) * A.row_len) * 4u;
            const float *grow = A.rows + ((size_t)(g0 + vl) * A.nr + r0) * A.row_len;
            auto add = [&](float z) {
                float off_t;
                const unsigned pos = find<MODEL>(A, q, z, &off_t);
#pragma unroll
                for (int u = 0; u < NRT; ++u) {
                    if (r0 + u >= A.nr) break;
                    mean[u] += eval<MODEL, SMEM>(lbase + (unsigned)(u * A.row_len) * 4u, grow + u * A.row_len, q, z, pos, off_t);
                }
            };
            PT_EACH_Z(r0 == 0, add)
            if (A.terms) {
#pragma unroll
                for (int u = 0; u < NRT; ++u) mean[u] = __fmul_rn(mean[u], inv_nss);
                // the terms' share of every passband's depth; the flux holds the
                // depth so far (this lane's alone) until the last rows
                const float *w = A.wts + row0 * A.nr + r0;
                float *fp = A.flux + row0 * A.n_t + t;
                for (int bb = 0; bb < A.n_bpg; ++bb, w += A.nr, fp += A.n_t) {
                    float dep = r0 == 0 ? 0.0f : *fp;
#pragma unroll
                    for (int u = 0; u < NRT; ++u) {
                        if (r0 + u >= A.nr) break;
                        dep += w[u] * mean[u];
                    }
                    *fp = r0 + NRT >= A.nr ? 1.0f - dep : dep;
                }
                continue;
            }
#pragma unroll
            for (int u = 0; u < NRT; ++u) {
                if (r0 + u >= A.nr) break;
                emit(vl, code, r0 + u, __fmul_rn(mean[u], inv_nss));
            }
        }
    }
    if (MODEL == R_MA && sexact) {
        // the pairs of geometries without a table: the exact terms, once for all
        // of a geometry's passbands
        for (int e = tid; e < nq; e += TB) {
            const int vl = geometry_of(e), code = list[vl * cap + (e - soff[vl])];
            if (sgeo[vl].w != 0.0f) continue;
            const GeomRec &r = srec[vl];
            const float2 ts = A.tsplit[tb + code];
            const float dt = pt::reduce_time(ts.x, ts.y, r);
            const int n_ss = dt >= r.win_lo && dt <= r.win_hi ? A.n_ss : 0;
            pt::OrbitState o;
            bool bad0 = false;
            pt::orbit_state(r, dt, A.max_iter, &bad0, &o);
            const float cosi = r.cosi, dx = A.n_ss > 1 ? r.nang * A.t_exp * inv_nss : 0.0f;
            const float x0 = -0.5f * (float)(A.n_ss - 1) * dx;
            const bool series = pt::fg_valid(r, o.E1, x0);
            const pt::FgSeries fg = pt::fg_series(o.E1, o.esin);
            if (series && bad0) nbad += n_ss;
            float3 te = make_float3(0.0f, 0.0f, 0.0f);
            auto add = [&](float z) {
                const float3 x = exact_terms(r.k, z);
                te.x += x.x;
                te.y += x.y;
                te.z += x.z;
            };
            PT_EACH_Z(true, add)
            for (int row = 0; row < A.n_bpg; ++row) {
                const size_t at = (size_t)(g0 + vl) * A.n_bpg + row;
                float we, wd, wn;
                if (A.terms) we = A.wts[3 * at], wd = A.wts[3 * at + 1], wn = A.wts[3 * at + 2];
                else pt::ma_weights(A.ld[2 * at], A.ld[2 * at + 1], &we, &wd, &wn);
                emit(vl, code, row, (we * te.x + wd * te.y + wn * te.z) * inv_nss);
            }
        }
    }
#undef PT_EACH_Z
    if (nbad && A.n_bad) atomicAdd(A.n_bad, nbad);
    if (!n_ssr) return;
    __syncthreads();
    // residual sums per geometry, passband and block of 256 times (the same sums
    // whatever the tile's shape): every thread's own time, from the evaluated
    // pair or with the flux at 1, then the warp's tree.  Eight sums or more go
    // through the tree eight together: at its first three levels each half of the
    // lanes keeps half of them, 9 shuffles in place of 40 (20,000 vectors x 4,000
    // times 461 -> 394 us a call; a lone sum would take 2 us longer that way).
    float *sred = reinterpret_cast<float *>(dsm + L.sred);     // [NW][n_sum]
    const int log_p = log_vt + log_kt, n_pair = 1 << log_p;    // pair p: block p / vt, geometry p % vt
    const int n_sum = n_ssr << log_p;                          // sum i: passband i / n_pair, pair i % n_pair
    float r1 = 0.0f;
    int k_of = -1, band_of = -1;
    auto value = [&](int i) {
        const int p = i & (n_pair - 1), vl = p & (vt - 1), k = p >> log_vt;
        if (vl >= ng) return 0.0f;
        if ((bits >> p) & 1u) return sval[i * TB + tid];
        const int band = sband[vl] + (A.k_per_band ? 0 : i >> log_p);
        if (k != k_of || band != band_of) {
            const int t = tb + k * TB + tid;
            r1 = 0.0f;
            if (t < A.n_t) {
                const float r = A.y[(size_t)band * A.n_t + t] - 1.0f;
                r1 = (A.wt ? A.wt[(size_t)band * A.n_t + t] : 1.0f) * r * r;
            }
            k_of = k;
            band_of = band;
        }
        return r1;
    };
    if (n_sum < 8) {
        for (int i = 0; i < n_sum; ++i) {
            float x = value(i);
#pragma unroll
            for (int o = 16; o > 0; o >>= 1) x += __shfl_xor_sync(0xffffffffu, x, o);
            if (lane == 0) sred[warp * n_sum + i] = x;
        }
    } else {
        const bool hi16 = lane & 16, hi8 = lane & 8, hi4 = lane & 4;
        for (int i0 = 0; i0 < n_sum; i0 += 8) {
            float v[8], x4[4], x2[2];
#pragma unroll
            for (int u = 0; u < 8; ++u) v[u] = i0 + u < n_sum ? value(i0 + u) : 0.0f;
#pragma unroll
            for (int i = 0; i < 4; ++i)
                x4[i] = (hi16 ? v[4 + i] : v[i]) + __shfl_xor_sync(0xffffffffu, hi16 ? v[i] : v[4 + i], 16);
#pragma unroll
            for (int i = 0; i < 2; ++i)
                x2[i] = (hi8 ? x4[2 + i] : x4[i]) + __shfl_xor_sync(0xffffffffu, hi8 ? x4[i] : x4[2 + i], 8);
            float x = (hi4 ? x2[1] : x2[0]) + __shfl_xor_sync(0xffffffffu, hi4 ? x2[0] : x2[1], 4);
            x += __shfl_xor_sync(0xffffffffu, x, 2);
            x += __shfl_xor_sync(0xffffffffu, x, 1);
            const int i = i0 + (lane >> 4) * 4 + (hi8 ? 2 : 0) + (hi4 ? 1 : 0);
            if ((lane & 3) == 0 && i < n_sum) sred[warp * n_sum + i] = x;
        }
    }
    __syncthreads();
    for (int i = tid; i < n_sum; i += TB) {
        const int p = i & (n_pair - 1), vl = p & (vt - 1), blk = tile * kt + (p >> log_vt);
        if (vl >= ng || blk >= A.n_blk) continue;
        float x = 0.0f;
        for (int w = 0; w < NW; ++w) x += sred[w * n_sum + i];
        A.ssr_part[((size_t)(g0 + vl) * A.n_bpg + (i >> log_p)) * A.n_blk + blk] = x;
    }
}

}  // namespace rows
