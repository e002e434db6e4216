// pt_gim.cuh -- row tables of the Gimenez series (Sec. 2.1).
//
// The transit depth of one geometry and passband,
//   1 - f = sum_n C_n alpha_n,
//   alpha_n = b^2 (1 - c^2)^(nu+1) sum_{j < n_j} T_{n,j} G_j(nu+2, 1; c^2),
// with T_{n,j} = A_{n,j} G_j(nu+2, nu+1; 1-b)^2 (Sec. 2.1.4), nu = (n + 2)/2,
// c = z/(1+k), is linear in T, and the functions of c,
//   Phi_{n,j}(c) = (1 - c^2)^(nu+1) G_j(nu+2, 1; c^2),
// are the same for every geometry.  A plan therefore holds their piecewise
// polynomials once: in u = sqrt(1 - c), nearly uniform in arccos c, degree 7
// on n_int equal intervals (the first one half as long, as in the
// Mandel-Agol rows).  A call forms, per row,
//   coefficients = sum_n C_n sum_j (b^2 T_{n,j}) Phi_{n,j} coefficients,
// per geometry and order a product over the n_j of that order, and every
// (time, supersample) then costs one look-up instead of the (N+1) n_j
// multiply-adds of the series.  The truncated series is kept as it is: the
// polynomials follow its alpha_n to (largest error over z, n = 0, 1, N, in 64
// bits, N = 1 .. 16, n_j = 2 .. 512)
//   k      0.05   0.1    0.2    0.3    0.5    0.7    1      1.5    3
//          2e-9   3e-9   6e-9   8e-9   3e-8   7e-8   6e-7   1e-7   1e-7
// (near k = 1 the inner contact lies at c = 0 and the terms do not fall off
// there), below the FP32 rounding of the flux up to k = 0.5, and the sums are
// well conditioned (at k <= 0.4 the sum of magnitudes is below four times the
// result), where the Chebyshev form used before cancelled by 10^2 to 10^3 and
// was off by about 1e-6 near k = 1.
// The product is FP32 on the FMA pipe: rows and sums stay 32-bit.
#pragma once

#include <algorithm>

#include "pt_rows.cuh"

namespace gim {

using pt::DF;
using pt::df_add;
using pt::df_mad;
using pt::df_mul;

constexpr int Q = rows::GIM_DEG;   // coefficients per interval
constexpr int GPC = 16;            // geometries per table CTA (one warp's lanes)

// Intervals of a row: W = 2 n_j + N + 4 bounds the frequency of the terms in
// arccos c; H of it per half interval.  A degree-7 fit leaves H^8 of the last
// terms' amplitude, and that falls with n_j, so longer series take wider
// intervals.  H grows such that the error at k = 0.3 stays between 1e-9 and
// 8e-9 from n_j = 24 on (shorter series: less), and not beyond 3.75: there
// the product below is already the wider rows' cost, and the error at k >= 0.7
// would pass 1e-7.
inline int intervals(int N, int n_j)
{
    const double H = fmin(2.76 * pow(n_j / 64.0, 0.28), 3.75);
    return (int)((2.0 * n_j + N + 4.0) / H) + 2;
}
inline float row_scale(int n_int) { return ((float)n_int - 0.5f) * (1.0f - 2e-6f); }

// ---------------------------------------------------------------------------
// Plan: the polynomials' coefficients, from the values of Phi_{n,j} at eight
// Chebyshev points per interval.  One CTA per order and four intervals: its
// first warp runs the recursion of G_j(nu+2, 1; x) at the 32 points, one a
// lane, in double-float arithmetic (a chain of n_j steps; FP64 has a 64th of
// the FP32 rate here), and the other three turn the previous BJ terms' values into
// coefficients.  The points are symmetric, so even and odd Chebyshev
// coefficients come from the sums and differences of four pairs; in powers of
// x in [-1, 1] they are 4 x 4 products, and t = x / 2 scales them by powers of
// two.  Only the first interval, t in [0, 1/2], shifts them (x = 4 t - 1).
// The high powers cancel to about 2^-6 of their terms, which double-float
// sums leave far below the rounding to FP32 at the end.  The same work in
// two FP64 passes with the node values in global memory took 83 us at N = 8,
// n_j = 192 and 454 at N = 16, n_j = 512; here launch and wait take 42 and 155.
// ---------------------------------------------------------------------------
constexpr int BJ = 32;          // terms per step
constexpr int BASIS_TB = 128;   // threads

struct Basis {
    const double *A, *recb;   // uploaded: A_{n,j}; [N+1][n_j][3] recursion of G_j(nu+2, nu+1; x)
    const float2 *rec;        // uploaded: recursion of G_j(nu+2, 1; x), double-float
    float4 *coef;             // the same in FP32
    float2 *dA, *drb;         // A and recb as double-float pairs
    float *B;                 // [(N+1) n_j][n_int][8]
    int NP1, n_j, n_int;
    double scale;
    double xq[Q];             // the points in [-1, 1]
    float2 m[2][4][4];        // [parity][power / 2][pair]: pair sums, differences -> powers of x
};

__global__ void __launch_bounds__(BASIS_TB) basis_kernel(const __grid_constant__ Basis P)
{
    extern __shared__ __align__(16) unsigned char bsm[];
    float2 *srec = reinterpret_cast<float2 *>(bsm);   // [n_j][3]
    __shared__ float2 sv[2][BJ][32];                  // node values
    __shared__ float sF[Q][Q];                        // powers of x -> powers of t, first interval
    const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5, n_j = P.n_j;
    const int n = blockIdx.y, i0 = 4 * blockIdx.x, q = lane & 7, i = min(i0 + (lane >> 3), P.n_int - 1);

    // the other forms of the uploaded tables, a share of them per CTA
    const int id0 = (blockIdx.y * gridDim.x + blockIdx.x) * BASIS_TB + tid, nth = gridDim.x * gridDim.y * BASIS_TB;
    for (int at = id0; at < P.NP1 * n_j; at += nth) {
        const DF a = pt::df_of(P.A[at]);
        P.dA[at] = make_float2(a.h, a.l);
        for (int c = 0; c < 3; ++c) {
            const DF r = pt::df_of(P.recb[3 * at + c]);
            P.drb[3 * at + c] = make_float2(r.h, r.l);
        }
        P.coef[at] = make_float4(P.rec[3 * at].x, P.rec[3 * at + 1].x, P.rec[3 * at + 2].x, 0.0f);
    }
    for (int at = tid; at < 3 * n_j; at += BASIS_TB) srec[at] = P.rec[(size_t)n * n_j * 3 + at];
    if (tid < Q * Q) {   // (4 t - 1)^c by powers r of t: binomial(c, r) 4^r (-1)^(c - r)
        const int r = tid / Q, c = tid % Q;
        float bin = r <= c ? 1.0f : 0.0f;
        for (int m = 1; m <= r && r <= c; ++m) bin = bin * (float)(c - r + m) / (float)m;
        sF[r][c] = bin * (float)(1 << (2 * r)) * ((c - r) & 1 ? -1.0f : 1.0f);
    }
    DF g = {}, gp = {}, x = {};
    DF M[4];
    if (warp == 0) {
        const double xq = P.xq[q], u = (i == 0 ? 0.25 * (1.0 + xq) : i + 0.5 * xq) / P.scale, c = 1.0 - u * u;
        const double sn = u * sqrt(2.0 - u * u);   // sqrt(1 - c^2)
        double pw = 1.0;
        for (int m = 0; m < n + 4; ++m) pw *= sn;
        x = pt::df_of(c * c);
        g = pt::df_of(pw);
    } else {
        for (int p = 0; p < 4; ++p) {
            const float2 v = P.m[q >> 2][q & 3][p];
            M[p] = DF{v.x, v.y};
        }
    }
    const int pw = q < 4 ? 2 * q : 2 * q - 7;   // the power of this lane's coefficient
    const float two = (float)(1 << pw);
    __syncthreads();
    const int n_step = (n_j + BJ - 1) / BJ;
    for (int st = 0; st <= n_step; ++st) {
        if (warp == 0 && st < n_step) {
            const int j1 = min(BJ, n_j - st * BJ);
            for (int j = 0; j < j1; ++j) {
                sv[st & 1][j][lane] = make_float2(g.h, g.l);
                const float2 *r = srec + 3 * (st * BJ + j);
                const DF al = df_mad(DF{r[1].x, r[1].y}, x, DF{r[0].x, r[0].y});
                const DF gn = df_mad(al, g, df_mul(DF{r[2].x, r[2].y}, gp));
                gp = g;
                g = gn;
            }
        }
        if (warp > 0 && st > 0) {
            const int j0 = (st - 1) * BJ, j1 = min(BJ, n_j - j0);
            for (int j = warp - 1; j < j1; j += BASIS_TB / 32 - 1) {
                const float2 v = sv[(st - 1) & 1][j][lane], o = sv[(st - 1) & 1][j][lane ^ 7];
                const float sg = q < 4 ? 1.0f : -1.0f;   // lanes 0..3 the pairs' sums, 4..7 differences (pair 7 - q)
                const DF sd = df_add(DF{o.x, o.y}, DF{sg * v.x, sg * v.y});
                DF b = {};
                for (int p = 0; p < 4; ++p) {
                    const int src = (lane & 24) + (q < 4 ? p : 7 - p);
                    const DF w = {__shfl_sync(~0u, sd.h, src), __shfl_sync(~0u, sd.l, src)};
                    b = p == 0 ? df_mul(M[0], w) : df_mad(M[p], w, b);
                }
                float out = two * b.h;
                if (i0 == 0) {
                    DF a = {};
                    for (int c = 0; c < Q; ++c) {
                        const int src = c & 1 ? 4 + c / 2 : c / 2;
                        const DF w = {__shfl_sync(~0u, b.h, src), __shfl_sync(~0u, b.l, src)};
                        a = df_mad(DF{sF[pw][c], 0.0f}, w, a);
                    }
                    // the depth is exactly 0 at the contact (u = 0)
                    if (lane < 8) out = pw == 0 ? 0.0f : a.h;
                }
                if (i0 + (lane >> 3) < P.n_int)
                    P.B[(((size_t)n * n_j + j0 + j) * P.n_int + i) * Q + pw] = out;
            }
        }
        __syncthreads();
    }
}

// ---------------------------------------------------------------------------
// Call: b^2 T_{n,j} of GPC geometries of one order.  The Jacobi recursion
// G_{j+1} = (r1 + r2 x) G_j + r3 G_{j-1}, x = 1 - b, is a chain of n_j dependent
// steps in double-float arithmetic, one geometry per thread; a chain runs alone
// on its scheduler, so its time is the length of its instruction stream, and
// everything else is done by all threads before it (r1 + r2 x) and after it
// (T).  The plan's coefficients are kept as double-float pairs: converting
// them from FP64 in every CTA cost more than the chain.  The CTAs of order 0
// also form the passbands' weights C_n.
// ---------------------------------------------------------------------------
struct Table {
    const float2 *dA;    // [N+1][n_j] A_{n,j}
    const float2 *drb;   // [N+1][n_j][3] recursion of G_j(nu+2, nu+1; x)
    int NP1, n_j;
    float *At;           // [(N+1) n_j][Gp] b^2 T, geometry fastest
    int Gp;              // geometries, rounded up to 32
    float *W;            // [n_geom n_bpg][N+1] C_n of every geometry and passband
};

inline size_t table_smem(int n_j)
{
    return 2 * (size_t)GPC * (n_j + 1) * sizeof(DF) + GPC * sizeof(DF) + (size_t)n_j * sizeof(DF) + GPC * sizeof(float);
}

__device__ __forceinline__ DF df2(float2 v) { return DF{v.x, v.y}; }

__device__ __forceinline__ void table_cta(const Table &T, const float *k, int n_geom, int n_bpg, const float *ld, int n,
                                          int gb)
{
    extern __shared__ __align__(16) unsigned char tsm[];
    const int n_j = T.n_j, rs = n_j + 1;   // rows of n_j + 1: chain lanes in distinct banks
    DF *sal = reinterpret_cast<DF *>(tsm);   // [GPC][rs]: r1_j + r2_j x
    DF *sG = sal + GPC * rs;                 // [GPC][rs]: G_j
    DF *sx = sG + GPC * rs;                  // [GPC]
    DF *sr3 = sx + GPC;                      // [n_j]: r3_j
    float *sb2 = reinterpret_cast<float *>(sr3 + n_j);   // [GPC]: b^2
    const float2 *rb = T.drb + (size_t)n * n_j * 3, *dA = T.dA + (size_t)n * n_j;
    const int tid = threadIdx.x, nt = blockDim.x;
    const int g0 = gb * GPC, ng = min(GPC, n_geom - g0), N = T.NP1 - 1;
    if (tid < ng) {
        const float kf = k[g0 + tid], b = kf / (1.0f + kf);
        const double kk = kf;
        sx[tid] = pt::df_of(1.0 - kk / (1.0 + kk));
        sb2[tid] = b * b;
    }
    for (int j = tid; j < n_j; j += nt) sr3[j] = df2(rb[3 * j + 2]);
    __syncthreads();
    for (int j = tid; j < n_j; j += nt) {
        const DF r1 = df2(rb[3 * j]), r2 = df2(rb[3 * j + 1]);
        for (int gl = 0; gl < ng; ++gl) sal[gl * rs + j] = df_add(r1, df_mul(r2, sx[gl]));
    }
    __syncthreads();
    if (tid < ng) {
        const DF *al = sal + tid * rs;
        DF *G = sG + tid * rs;
        // q = r3_j G_{j-1} is formed one step ahead, so each step's dependent
        // path is one df_mad
        DF gc = DF{1.0f, 0.0f}, q = DF{0.0f, 0.0f};
        for (int j = 0; j < n_j; ++j) {
            G[j] = gc;
            const DF gn = df_mad(al[j], gc, q);
            if (j + 1 < n_j) q = df_mul(sr3[j + 1], gc);
            gc = gn;
        }
    }
    if (n == 0 && tid >= 32) {
        // beside the chains: C_0 = (1 - sum u)/D, C_n = u_n/D, D = 1 - sum n u_n/(n+2)   (Sec. 2.1.3)
        for (long long i = tid - 32; i < (long long)ng * n_bpg; i += nt - 32) {
            const size_t row = (size_t)g0 * n_bpg + i;
            const float *u = ld + row * N;
            float su = 0.0f, sd = 0.0f;
            for (int m = 1; m <= N; ++m) {
                su += u[m - 1];
                sd += (float)m * u[m - 1] / (float)(m + 2);
            }
            float *w = T.W + row * T.NP1;
            w[0] = (1.0f - su) / (1.0f - sd);
            for (int m = 1; m <= N; ++m) w[m] = u[m - 1] / (1.0f - sd);
        }
    }
    __syncthreads();
    for (int e = tid; e < n_j * ng; e += nt) {
        const int j = e / ng, gl = e - j * ng;
        const DF gc = sG[gl * rs + j];
        const DF t = df_mul(df_mul(df2(__ldg(dA + j)), gc), gc);
        T.At[((size_t)n * n_j + j) * T.Gp + g0 + gl] = (t.h + t.l) * sb2[gl];
    }
}

// ---------------------------------------------------------------------------
// The rows: term n of geometry g is P_n = At_n^T B_n, a product over the n_j of
// its order, and a passband's row sum_n C_n P_n.  The terms cost what one
// passband's row would (each order meets its own n_j only), and any number of
// passbands sharing a radius ratio takes the same product: with a row of
// (N+1) n_j factors per passband, as before, eight passbands of 1,000 vectors
// took 750 us at N = 8, n_j = 192, and the zero factors of rows of the terms
// another nine times the work.
// A CTA covers RT geometries x CT = 256 C / RT columns, a warp one order at a
// time, 8 geometries x C columns per lane as pairs of geometries in
// fma.rn.f32x2; operands come from L2 through a ring of cp.async stages per
// warp (loads straight to registers left an SM with a third of the bytes in
// flight that the L2 latency asks for).  An order is cut into chains(N) sums of
// consecutive j, added in order, so that a CTA has 9 to 20 warps: `spread`
// gives each chain a warp, which ends a lone wave soonest; else a warp takes
// its order's chains in turn, and two CTAs share an SM.  Every form adds up a
// row in the same order, so a row depends neither on the other geometries nor on the other
// passbands of its call.
// What bounds it: shared-memory loads and FMA issue about equally (41 TFLOP/s
// on 5,000 rows at N = 8, n_j = 192, half the FP32 peak; 33 by direct loads).
// ---------------------------------------------------------------------------
constexpr int CHAIN_STEP = 16;      // chains are whole stages of every form
constexpr int KS = 8, STAGES = 3;   // j per stage of a ring
constexpr int MAX_WARPS = 20;

// j per chain, and chains per order
inline int chain_len(int NP1, int n_j)
{
    const int c = std::max(1, (16 + NP1 / 2) / NP1), per = (n_j + c - 1) / c;
    return (per + CHAIN_STEP - 1) / CHAIN_STEP * CHAIN_STEP;
}
inline int chains(int NP1, int n_j) { return (n_j + chain_len(NP1, n_j) - 1) / chain_len(NP1, n_j); }

template <int RT, int C>
struct Shape {
    static constexpr int CT = 256 * C / RT;        // columns per CTA
    static constexpr int STAGE = KS * (RT + CT);   // floats
    static constexpr int RING = STAGES * STAGE, SLOT = RT * CT;
    // a warp's sums: in its ring's place after its only chain, else beside the ring
    static constexpr int warp_floats(bool one_chain) { return one_chain ? (RING > SLOT ? RING : SLOT) : RING + SLOT; }
    // ... and the weights of up to eight passbands
    static constexpr size_t SMEM_MAX = ((size_t)MAX_WARPS * (RING > SLOT ? RING : SLOT) + RT * rows::MAX_BAND_ROWS * 17) * sizeof(float);
    static_assert(SMEM_MAX <= 200 * 1024 && 10 * (RING + SLOT) <= MAX_WARPS * (RING > SLOT ? RING : SLOT), "shared memory");
};

struct Product {
    const float *At;   // [(N+1) n_j][Gp]
    int Gp, G;
    const float *B;    // [(N+1) n_j][Nc]
    int n_j, NP1, per, chains, spread, Nc;
    const float *W;    // [G nr][N+1]; null: the terms themselves
    int nr;
    float *out;        // [G][nr or N+1][Nc]
};

constexpr int TALL = 128, TALL_KS = CHAIN_STEP, TALL_STAGES = 4;
constexpr size_t TALL_SMEM = (size_t)TALL_STAGES * TALL_KS * 2 * TALL * sizeof(float);

// What a call runs: tiles of 32 geometries x 32 or 48 columns with a warp per
// chain, x 32 columns with a warp per order, of 8 geometries x 32 or 64 columns
// with a warp per chain (few geometries), or of 128 x 128 (many).  The one of
// least cost in whole waves; the weights are measured times of a wave at N = 8,
// n_j = 192 in units of 0.1 us (17, 25; 22 alone and 13.7 each when they share an
// SM; 12.4, 14.5), which keep their proportions at other orders and depths: over
// 90 calls of 1 to 5,000 geometries the choice was the fastest form or within 2 us
// or 10 % of it.  Tiles of 128 x 128 take 12 waves of 32 x 32 where orders are one
// chain of 128 j or more, and 14 or more where they are shorter (N = 8: 186 us
// against 152 on 2,000 rows) and are left out there, and where a geometry has
// several rows (their sums in memory: 1,985 us against 1,384 with eight).
struct Form {
    int rt, c, spread;
};

inline bool tall_fits(int NP1, int n_j, bool one_row) { return one_row && n_j >= 128 && chains(NP1, n_j) == 1; }

inline Form product_form(size_t G, int Nc, bool tall, int n_sm)
{
    const Form cand[6] = {{32, 4, 0}, {32, 4, 1}, {32, 6, 1}, {8, 1, 1}, {8, 2, 1}, {TALL, 0, 0}};
    const size_t wave[6] = {137, 170, 250, 124, 145, 1610};
    Form best = cand[0];
    size_t cost = 0;
    for (int i = 0; i < (tall ? 6 : 5); ++i) {
        const size_t ct = cand[i].rt == TALL ? (size_t)TALL : (size_t)(256 * cand[i].c / cand[i].rt);
        const size_t w = ((G + cand[i].rt - 1) / cand[i].rt * (((size_t)Nc + ct - 1) / ct) + n_sm - 1) / n_sm;
        const size_t t = i == 0 && w == 1 ? 220 : w * wave[i] + (i == 0 ? 40 : 0);
        if (i == 0 || t < cost) {
            best = cand[i];
            cost = t;
        }
    }
    return best;
}

__device__ __forceinline__ void copy16(unsigned dst, const float *src, bool ok)
{
    const int bytes = ok ? 16 : 0;   // 0: zero-fill
    asm volatile("cp.async.cg.shared.global [%0], [%1], 16, %2;" ::"r"(dst), "l"(src), "r"(bytes) : "memory");
}

template <int RT, int C>
__global__ void __launch_bounds__(32 * MAX_WARPS, 1) product_kernel(Product A)
{
    pt::chain_begin();
    using S = Shape<RT, C>;
    constexpr int CT = S::CT;
    extern __shared__ __align__(16) float psm[];
    const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
    const int n_ct = (A.Nc + CT - 1) / CT;
    const int ct = (int)(blockIdx.x % n_ct), rt = (int)(blockIdx.x / n_ct);   // column and geometry tile
    const int cols = min(CT, A.Nc - ct * CT);                                // a multiple of 8
    const int wpn = A.spread ? A.chains : 1, n = warp / wpn;                 // warps per order, this warp's
    const bool one = A.spread || A.chains == 1;
    const int unit = S::warp_floats(one);
    // the passbands' weights of the tile, on their way beside the products
    float *sw = psm + (size_t)(A.spread ? A.chains : 1) * A.NP1 * unit;   // [RT][nr][N+1]
    if (A.W) {
        const int row = A.nr * A.NP1, n_w = min(RT, A.G - rt * RT) * row;
        const float *w = A.W + (size_t)rt * RT * row;   // this call's: not by __ldg
        for (int i = tid; i < n_w; i += blockDim.x) sw[i] = w[i];
    }
    float *ring = psm + (size_t)warp * unit, *slot = ring + (one ? 0 : S::RING);
    const unsigned ring_at = (unsigned)__cvta_generic_to_shared(ring);
    const int rl = (lane / (CT / C)) * 8, cl = (lane % (CT / C)) * C;
    const int j0 = A.spread ? (warp - n * wpn) * A.per : 0, len = A.spread ? min(A.n_j - j0, A.per) : A.n_j;
    const float *ga = A.At + ((size_t)n * A.n_j + j0) * A.Gp + (size_t)rt * RT;
    const float *gb = A.B + ((size_t)n * A.n_j + j0) * A.Nc + (size_t)ct * CT;
    auto fetch = [&](int st) {
        const int k0 = st * KS;
        if (k0 < len) {
            const unsigned d = ring_at + 4u * (unsigned)((st % STAGES) * S::STAGE);
#pragma unroll
            for (int q = 0; q < (KS * RT / 4 + 31) / 32; ++q) {
                const int e = q * 32 + lane, kk = e / (RT / 4), x = 4 * (e % (RT / 4));
                if (KS * RT / 4 % 32 == 0 || e < KS * RT / 4)
                    copy16(d + 16u * e, ga + (size_t)min(k0 + kk, len - 1) * A.Gp + x, k0 + kk < len);
            }
#pragma unroll
            for (int q = 0; q < (KS * CT / 4 + 31) / 32; ++q) {
                const int e = q * 32 + lane, kk = e / (CT / 4), x = 4 * (e % (CT / 4));
                if (KS * CT / 4 % 32 == 0 || e < KS * CT / 4) {
                    const bool ok = k0 + kk < len && x < cols;
                    copy16(d + 4u * KS * RT + 16u * e, ok ? gb + (size_t)(k0 + kk) * A.Nc + x : gb, ok);
                }
            }
        }
        asm volatile("cp.async.commit_group;" ::: "memory");
    };
    unsigned long long acc[4][C];   // pairs of geometries
#pragma unroll
    for (int i = 0; i < 4; ++i)
#pragma unroll
        for (int j = 0; j < C; ++j) acc[i][j] = 0ull;
    auto to_slot = [&](bool first) {
#pragma unroll
        for (int i = 0; i < 4; ++i)
#pragma unroll
            for (int j = 0; j < C; ++j) {
                float *d = slot + (rl + 2 * i) * CT + cl + j;
                const float x = pt::f2_lo(acc[i][j]), y = pt::f2_hi(acc[i][j]);
                d[0] = first ? x : d[0] + x;
                d[CT] = first ? y : d[CT] + y;
                acc[i][j] = 0ull;
            }
    };
#pragma unroll
    for (int st = 0; st < STAGES - 1; ++st) fetch(st);
    int left = A.per;   // of the chain, when this warp takes several
    for (int st = 0; st * KS < len; ++st) {
        asm volatile("cp.async.wait_group %0;" ::"n"(STAGES - 2) : "memory");
        __syncwarp();   // stage st has landed for every lane, stage st - 1 is no longer read
        fetch(st + STAGES - 1);
        const float *sa = ring + (st % STAGES) * S::STAGE + rl, *sb = ring + (st % STAGES) * S::STAGE + KS * RT + cl;
#pragma unroll
        for (int kk = 0; kk < KS; ++kk) {
            const ulonglong2 a0 = *reinterpret_cast<const ulonglong2 *>(sa + kk * RT);
            const ulonglong2 a1 = *reinterpret_cast<const ulonglong2 *>(sa + kk * RT + 4);
            const unsigned long long a[4] = {a0.x, a0.y, a1.x, a1.y};
            float b[C];
            if constexpr (C == 4) {
                const float4 v = *reinterpret_cast<const float4 *>(sb + kk * CT);
                b[0] = v.x, b[1] = v.y, b[2] = v.z, b[3] = v.w;
            } else if constexpr (C % 2 == 0) {
#pragma unroll
                for (int j = 0; j < C; j += 2) {
                    const float2 v = *reinterpret_cast<const float2 *>(sb + kk * CT + j);
                    b[j] = v.x, b[j + 1] = v.y;
                }
            } else {
#pragma unroll
                for (int j = 0; j < C; ++j) b[j] = sb[kk * CT + j];
            }
#pragma unroll
            for (int j = 0; j < C; ++j) {
                const unsigned long long bb = pt::f2_pack(b[j], b[j]);
#pragma unroll
                for (int i = 0; i < 4; ++i) acc[i][j] = pt::f2_fma(a[i], bb, acc[i][j]);
            }
        }
        left -= KS;
        if (!one && left == 0) {
            to_slot(st * KS < A.per);
            left = A.per;
        }
    }
    asm volatile("cp.async.wait_all;" ::: "memory");
    __syncwarp();   // the ring is no longer read: the sums may take its place
    if (one || left < A.per) to_slot(one || A.n_j <= A.per);
    __syncthreads();
    const int step = wpn * unit;   // from order to order
    for (int e = tid; e < RT * CT; e += blockDim.x) {
        const int g = rt * RT + e / CT, x = e % CT;
        if (g >= A.G || x >= cols) continue;
        float *p = psm + (one ? 0 : S::RING) + e;   // (a thread's own elements)
        if (wpn > 1)
            for (int m = 0; m < A.NP1; ++m) {
                float v = p[(size_t)m * step];
                for (int q = 1; q < wpn; ++q) v += p[(size_t)m * step + (size_t)q * unit];
                p[(size_t)m * step] = v;
            }
        float *out = A.out + (size_t)g * (A.W ? A.nr : A.NP1) * A.Nc + ct * CT + x;
        if (!A.W) {
            for (int m = 0; m < A.NP1; ++m) out[(size_t)m * A.Nc] = p[(size_t)m * step];
            continue;
        }
        const float *w = sw + (e / CT) * A.nr * A.NP1;
        for (int r = 0; r < A.nr; ++r, w += A.NP1) {
            float v = 0.0f;
            for (int m = 0; m < A.NP1; ++m) v = fmaf(w[m], p[(size_t)m * step], v);
            out[(size_t)r * A.Nc] = v;
        }
    }
}

// The same for many geometries, long orders of one chain, and one row per
// geometry (or the terms): a CTA covers 128 geometries x 128 columns and all of
// it shares its operands, 8 x 8 per thread; an order's sums go to the row when
// it ends (row += C_n P_n by the thread that holds P_n: the fma chain of the
// other form).  47 TFLOP/s on 1,000 rows at N = 16, n_j = 512: 835 us, 1,041 by
// tiles of 32 x 32.
__global__ void __launch_bounds__(256, 1) product_tall_kernel(Product A)
{
    pt::chain_begin();
    constexpr int STAGE = TALL_KS * 2 * TALL;
    extern __shared__ __align__(16) float psm[];
    const int tid = threadIdx.x, tx = tid & 15, ty = tid >> 4;   // rows 4 ty, 64 + 4 ty, columns 4 tx, 64 + 4 tx (+ 0 .. 3)
    const int n_ct = (A.Nc + TALL - 1) / TALL;
    const int c0 = (int)(blockIdx.x % n_ct) * TALL, g0 = (int)(blockIdx.x / n_ct) * TALL;
    const int per_n = (A.n_j + TALL_KS - 1) / TALL_KS, n_st = A.NP1 * per_n;   // stages: an order's, all
    const unsigned at = (unsigned)__cvta_generic_to_shared(psm);
    auto fetch = [&](int st) {
        if (st < n_st) {
            const int n = st / per_n, k0 = (st - n * per_n) * TALL_KS;
            const float *ga = A.At + ((size_t)n * A.n_j + k0) * A.Gp + g0, *gb = A.B + ((size_t)n * A.n_j + k0) * A.Nc + c0;
            const unsigned d = at + 4u * (unsigned)((st % TALL_STAGES) * STAGE);
#pragma unroll
            for (int q = 0; q < TALL_KS * TALL / 4 / 256; ++q) {
                const int e = q * 256 + tid, kk = e / (TALL / 4), x = 4 * (e % (TALL / 4));
                const bool in = k0 + kk < A.n_j, oa = in && g0 + x < A.Gp, ob = in && c0 + x < A.Nc;
                copy16(d + 16u * e, oa ? ga + (size_t)kk * A.Gp + x : A.At, oa);
                copy16(d + 4u * TALL_KS * TALL + 16u * e, ob ? gb + (size_t)kk * A.Nc + x : A.B, ob);
            }
        }
        asm volatile("cp.async.commit_group;" ::: "memory");
    };
    unsigned long long acc[4][8];   // pairs of geometries
#pragma unroll
    for (int i = 0; i < 4; ++i)
#pragma unroll
        for (int j = 0; j < 8; ++j) acc[i][j] = 0ull;
#pragma unroll
    for (int st = 0; st < TALL_STAGES - 1; ++st) fetch(st);
    int n = 0, in_n = 0;
    for (int st = 0; st < n_st; ++st) {
        asm volatile("cp.async.wait_group %0;" ::"n"(TALL_STAGES - 2) : "memory");
        __syncthreads();   // stage st has landed, stage st - 1 is no longer read
        fetch(st + TALL_STAGES - 1);
        const float *sa = psm + (st % TALL_STAGES) * STAGE + 4 * ty, *sb = psm + (st % TALL_STAGES) * STAGE + TALL_KS * TALL + 4 * tx;
#pragma unroll
        for (int kk = 0; kk < TALL_KS; ++kk) {
            const ulonglong2 a0 = *reinterpret_cast<const ulonglong2 *>(sa + kk * TALL);
            const ulonglong2 a1 = *reinterpret_cast<const ulonglong2 *>(sa + kk * TALL + TALL / 2);
            const float4 b0 = *reinterpret_cast<const float4 *>(sb + kk * TALL);
            const float4 b1 = *reinterpret_cast<const float4 *>(sb + kk * TALL + TALL / 2);
            const unsigned long long a[4] = {a0.x, a0.y, a1.x, a1.y};
            const float b[8] = {b0.x, b0.y, b0.z, b0.w, b1.x, b1.y, b1.z, b1.w};
#pragma unroll
            for (int j = 0; j < 8; ++j) {
                const unsigned long long bb = pt::f2_pack(b[j], b[j]);
#pragma unroll
                for (int i = 0; i < 4; ++i) acc[i][j] = pt::f2_fma(a[i], bb, acc[i][j]);
            }
        }
        if (++in_n < per_n) continue;
        // the order ends: into the row
#pragma unroll
        for (int i = 0; i < 8; ++i) {
            const int g = g0 + (i >> 2) * (TALL / 2) + 4 * ty + (i & 3);
            if (g >= A.G) continue;
            const float w = A.W ? A.W[(size_t)g * A.NP1 + n] : 1.0f;
            float *out = A.out + (A.W ? (size_t)g : (size_t)g * A.NP1 + n) * A.Nc;
#pragma unroll
            for (int h = 0; h < 2; ++h) {
                const int c = c0 + h * (TALL / 2) + 4 * tx;
                if (c >= A.Nc) continue;   // (Nc a multiple of 8)
                float4 *d = reinterpret_cast<float4 *>(out + c);
                float4 v = make_float4(0.0f, 0.0f, 0.0f, 0.0f);
                if (A.W && n > 0) v = *d;
                float p[4];
#pragma unroll
                for (int j = 0; j < 4; ++j) p[j] = i & 1 ? pt::f2_hi(acc[i >> 1][4 * h + j]) : pt::f2_lo(acc[i >> 1][4 * h + j]);
                *d = A.W ? make_float4(fmaf(w, p[0], v.x), fmaf(w, p[1], v.y), fmaf(w, p[2], v.z), fmaf(w, p[3], v.w))
                         : make_float4(p[0], p[1], p[2], p[3]);
            }
        }
#pragma unroll
        for (int i = 0; i < 4; ++i)
#pragma unroll
            for (int j = 0; j < 8; ++j) acc[i][j] = 0ull;
        ++n;
        in_n = 0;
    }
}

// Rows on z nodes (Sec. 3.3) read from the series' rows: node i of a row.
__global__ void zi_rows_kernel(rows::Args A, const float *k, int n_row, int zi_len, float *out)
{
    pt::chain_begin();
    const long long id = (long long)blockIdx.x * blockDim.x + threadIdx.x;
    const long long row = id / zi_len;
    if (row >= n_row) return;
    const int i = (int)(id - row * zi_len);
    float v = 0.0f;
    if (i < A.n_in + A.n_edge) {
        const float kk = k[row / A.nr];
        const float zb = fmaxf(1.0f - kk, 0.0f);
        const float h1 = zb / (float)(A.n_in - 1), h2 = (1.0f + kk - zb) / (float)A.n_edge;
        const float z = i < A.n_in ? (float)i * h1 : zb + (float)(i - A.n_in + 1) * h2;
        const float4 q = rows::look_up_constants<rows::R_GIM>(A, kk);
        float t;
        const unsigned pos = rows::find<rows::R_GIM>(A, q, z, &t);
        v = rows::eval<rows::R_GIM, false>(0u, A.rows + row * A.row_len, q, z, pos, t);
        if (!(z < 1.0f + kk)) v = 0.0f;
    }
    out[id] = v;
}

}  // namespace gim
