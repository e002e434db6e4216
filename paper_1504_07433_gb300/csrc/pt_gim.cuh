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
//   coefficients = sum_{n,j} (C_n b^2 T_{n,j}) Phi coefficients,
// a product of [rows] x [(N+1) n_j] with [(N+1) n_j] x [8 n_int], and every
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

#include "pt_rows.cuh"

namespace gim {

using pt::DF;
using pt::df_add;
using pt::df_mad;
using pt::df_mul;

constexpr int Q = rows::GIM_DEG;   // coefficients per interval
constexpr int GPC = 16;            // geometries per table CTA

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
// Plan: node values of Phi_{n,j}, then coefficients.  rec [N+1][n_j][3]: the
// recursion of G_j(nu+2, 1; x); all in FP64 (once per plan).
// ---------------------------------------------------------------------------
__global__ void basis_nodes_kernel(const double *rec, int NP1, int n_j, int n_int, double scale, double *V)
{
    const int n_node = Q * n_int;
    const int id = blockIdx.x * blockDim.x + threadIdx.x;
    if (id >= NP1 * n_node) return;
    const int n = id / n_node, node = id - n * n_node, i = node / Q, q = node - i * Q;
    const double xq = cospi((q + 0.5) / Q);
    const double u = (i == 0 ? 0.25 * (1.0 + xq) : i + 0.5 * xq) / scale;
    const double c = 1.0 - u * u, x = c * c;
    const double sn = u * sqrt(2.0 - u * u);   // sqrt(1 - c^2)
    double pw = 1.0;
    for (int m = 0; m < n + 4; ++m) pw *= sn;
    double g = pw, gp = 0.0;
    for (int j = 0; j < n_j; ++j) {
        V[((size_t)n * n_j + j) * n_node + node] = g;
        const double *r = rec + ((size_t)n * n_j + j) * 3;
        const double gn = (r[0] + r[1] * x) * g + r[2] * gp;
        gp = g;
        g = gn;
    }
}

// mat [2][Q][Q]: node values -> monomial coefficients (first interval, others)
__global__ void basis_coef_kernel(const double *V, const double *mat, int K, int n_int, float *B)
{
    const long long id = (long long)blockIdx.x * blockDim.x + threadIdx.x;
    if (id >= (long long)K * n_int) return;
    const long long k = id / n_int;
    const int i = (int)(id - k * n_int);
    const double *v = V + (k * n_int + i) * Q, *m = mat + (i == 0 ? 0 : Q * Q);
    for (int c = 0; c < Q; ++c) {
        double a = 0.0;
        for (int q = 0; q < Q; ++q) a += m[c * Q + q] * v[q];
        // the depth is exactly 0 at the contact (u = 0)
        B[(k * n_int + i) * Q + c] = (i == 0 && c == 0) ? 0.0f : (float)a;
    }
}

// ---------------------------------------------------------------------------
// Call: the weighted T_{n,j} of GPC geometries of one order.  The Jacobi
// recursion G_{j+1} = (r1 + r2 x) G_j + r3 G_{j-1}, x = 1 - b, is a chain of
// n_j dependent steps in double-float arithmetic, one geometry per thread; a
// chain runs alone on its scheduler, so its time is the length of its
// instruction stream, and everything else is done by all threads before it
// (r1 + r2 x) and after it (T, the weights).  The plan's coefficients are kept
// as double-float pairs: converting them from FP64 in every CTA cost more than
// the chain.
// ---------------------------------------------------------------------------
struct Table {
    const float2 *dA;    // [N+1][n_j] A_{n,j}
    const float2 *drb;   // [N+1][n_j][3] recursion of G_j(nu+2, nu+1; x)
    int NP1, n_j;
    float *At;           // [(N+1) n_j][Rp] weighted T, row fastest
    int Rp;              // rows, rounded up to 32
};

inline size_t table_smem(int n_j, int nr)
{
    return 2 * (size_t)GPC * (n_j + 1) * sizeof(DF) + GPC * sizeof(DF) + (size_t)n_j * sizeof(DF) + (size_t)GPC * nr * sizeof(float);
}

__device__ __forceinline__ DF df2(float2 v) { return DF{v.x, v.y}; }

__device__ __forceinline__ void table_cta(const Table &T, const float *k, int n_geom, int nr, int terms, int n_bpg,
                                          const float *ld, int n, int gb)
{
    extern __shared__ __align__(16) unsigned char tsm[];
    const int n_j = T.n_j, rs = n_j + 1;   // rows of n_j + 1: chain lanes in distinct banks
    DF *sal = reinterpret_cast<DF *>(tsm);   // [GPC][rs]: r1_j + r2_j x
    DF *sG = sal + GPC * rs;                 // [GPC][rs]: G_j
    DF *sx = sG + GPC * rs;                  // [GPC]
    DF *sr3 = sx + GPC;                      // [n_j]: r3_j
    float *sw = reinterpret_cast<float *>(sr3 + n_j);   // [GPC][nr]: C_n b^2
    const float2 *rb = T.drb + (size_t)n * n_j * 3, *dA = T.dA + (size_t)n * n_j;
    const int tid = threadIdx.x, nt = blockDim.x;
    const int g0 = gb * GPC, ng = min(GPC, n_geom - g0), N = T.NP1 - 1;
    if (tid < ng) {
        const double kk = k[g0 + tid];
        sx[tid] = pt::df_of(1.0 - kk / (1.0 + kk));
    }
    for (int j = tid; j < n_j; j += nt) sr3[j] = df2(rb[3 * j + 2]);
    for (int i = tid; i < ng * nr; i += nt) {
        const int gl = i / nr, r = i - gl * nr;
        const float kk = k[g0 + gl], b = kk / (1.0f + kk);
        float w = r == n ? 1.0f : 0.0f;
        if (!terms) {   // C_0 = (1 - sum u)/D, C_n = u_n/D, D = 1 - sum n u_n/(n+2)   (Sec. 2.1.3)
            const float *u = ld + ((size_t)(g0 + gl) * n_bpg + r) * N;
            float su = 0.0f, sd = 0.0f;
            for (int m = 1; m <= N; ++m) {
                su += u[m - 1];
                sd += (float)m * u[m - 1] / (float)(m + 2);
            }
            w = (n == 0 ? 1.0f - su : u[n - 1]) / (1.0f - sd);
        }
        sw[i] = w * b * b;
    }
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
    __syncthreads();
    const int n_row = ng * nr;
    for (int e = tid; e < n_j * n_row; e += nt) {
        const int j = e / n_row, i = e - j * n_row, gl = i / nr;
        const DF gc = sG[gl * rs + j];
        const DF t = df_mul(df_mul(df2(__ldg(dA + j)), gc), gc);
        T.At[((size_t)n * n_j + j) * T.Rp + (size_t)g0 * nr + i] = (t.h + t.l) * sw[i];
    }
}

// ---------------------------------------------------------------------------
// rows [R][Nc] = At^T [R][K] B [K][Nc].  A CTA covers RT rows x 256 C / RT
// columns and splits K into PARTS parts over its warps (the parts' sums meet in
// shared memory, in order), because rows and columns alone would not fill the
// chip.  Operands come straight from L2 (each is read once per CTA); a thread
// holds 8 rows x C columns: C = 8 or 6 at RT = 32, 3, 2 or 1 at RT = 8 (for few
// rows: more loads in flight per warp).  The width is the one whose CTAs, one
// per multiprocessor, need the least time in whole waves (product_width): 256
// rows of n_j = 192 are 112 CTAs of 64 columns, 36.6 us, or 144 of 48, 29.4
// (ncu, cold); 100 rows 182 of 64, 27.1 us, or 117 of 96, 20.6.  Every form adds
// up a row in the same order, so a row does not depend on the others of its
// call.
// ---------------------------------------------------------------------------
constexpr int PARTS = 16;

template <int RT, int C>
struct Split {
    static constexpr int WARPS = PARTS;
    static constexpr int CT = 256 * C / RT;   // columns per CTA
    static constexpr size_t SMEM = (size_t)PARTS * RT * CT * sizeof(float);
};

// C for r row tiles of RT rows: a step of a thread is 8 C multiply-adds and
// about 6 other instructions.
template <int RT>
inline int product_width(size_t r, int Nc, int n_sm)
{
    const int cand[2][3] = {{8, 6, 6}, {3, 2, 1}};
    int best = 0;
    size_t cost = 0;
    for (int c : cand[RT == 32 ? 0 : 1]) {
        const size_t ct = (size_t)(256 * c / RT), ctas = r * (((size_t)Nc + ct - 1) / ct);
        const size_t t = (ctas + n_sm - 1) / n_sm * (size_t)(8 * c + 6);
        if (best == 0 || t < cost) {
            best = c;
            cost = t;
        }
    }
    return best;
}

template <int RT, int C>
__global__ void __launch_bounds__(32 * PARTS, 1) product_kernel(const float *At, int Rp, const float *B, int K, int Nc,
                                                                int R, float *out)
{
    pt::chain_begin();
    constexpr int WARPS = PARTS, CT = Split<RT, C>::CT;
    extern __shared__ __align__(16) float psm[];   // [PARTS][RT][CT]
    const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
    const int n_ct = (Nc + CT - 1) / CT;
    const int ct = (int)(blockIdx.x % n_ct), rt = (int)(blockIdx.x / n_ct);   // column and row tile
    const int rl = (lane / (CT / C)) * 8;
    // Columns beyond the last: the last C again (the same sums; a tile has at
    // least 8 columns, Nc being a multiple of 8).
    const int cl = min((lane % (CT / C)) * C, Nc - C - ct * CT);
    const float *pa = At + (size_t)rt * RT + rl;
    const float *pb = B + ct * CT + cl;
    const int per = (K + PARTS - 1) / PARTS;
    {
        const int part = warp;
        const int k0 = part * per, k1 = min(K, k0 + per);
        float acc[8][C];
#pragma unroll
        for (int i = 0; i < 8; ++i)
#pragma unroll
            for (int j = 0; j < C; ++j) acc[i][j] = 0.0f;
#pragma unroll(RT == 32 ? (C == 8 ? 3 : 4) : (C == 3 ? 8 : 12))
        for (int k = k0; k < k1; ++k) {
            const float4 a0 = *reinterpret_cast<const float4 *>(pa + (size_t)k * Rp);   // this call's: not by __ldg
            const float4 a1 = *reinterpret_cast<const float4 *>(pa + (size_t)k * Rp + 4);
            const float a[8] = {a0.x, a0.y, a0.z, a0.w, a1.x, a1.y, a1.z, a1.w};
            float b[C];
            const float *bk = pb + (size_t)k * Nc;
            if constexpr (C == 8) {
#pragma unroll
                for (int j = 0; j < C; j += 4) {
                    const float4 v = __ldg(reinterpret_cast<const float4 *>(bk + j));
                    b[j] = v.x, b[j + 1] = v.y, b[j + 2] = v.z, b[j + 3] = v.w;
                }
            } else if constexpr (C % 2 == 0) {
#pragma unroll
                for (int j = 0; j < C; j += 2) {
                    const float2 v = __ldg(reinterpret_cast<const float2 *>(bk + j));
                    b[j] = v.x, b[j + 1] = v.y;
                }
            } else {
#pragma unroll
                for (int j = 0; j < C; ++j) b[j] = __ldg(bk + j);
            }
#pragma unroll
            for (int i = 0; i < 8; ++i)
#pragma unroll
                for (int j = 0; j < C; ++j) acc[i][j] = fmaf(a[i], b[j], acc[i][j]);
        }
        float *mine = psm + (size_t)part * RT * CT;
#pragma unroll
        for (int i = 0; i < 8; ++i)
#pragma unroll
            for (int j = 0; j < C; ++j) mine[(rl + i) * CT + cl + j] = acc[i][j];
    }
    __syncthreads();
    for (int e = tid; e < RT * CT; e += 32 * WARPS) {
        float x = 0.0f;
#pragma unroll
        for (int w = 0; w < PARTS; ++w) x += psm[(size_t)w * RT * CT + e];
        const int row = rt * RT + e / CT, col = ct * CT + e % CT;
        if (row < R && col < Nc) out[(size_t)row * Nc + col] = x;
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
