// pt_adjoint.cu -- hand-written adjoint of the quadratic Mandel-Agol light
// curve: SSR = sum_t wt (y - f)^2 and dSSR/dtheta for
// theta = (t0, P, a, b, e, w, k, u1, u2), one CTA per parameter vector, the
// forward model recomputed in registers (nothing saved between passes).  What
// depends on the separation alone comes, for a vector with many points, from
// a row of polynomials made at the start of its CTA; the chain rule through
// the orbit is applied to sums over the points, not to each of them.
//
// The paper has no gradients (it cites analytic MA derivatives, Pal 2008).
// They follow from the definition of the occulted flux: with
// I_g = int int_overlap g dA for g in {1, mu, mu^2},
//   F = 1 - [(1 - u1 - u2) I_1 + (u1 + 2 u2) I_mu - u2 I_mu2] / (pi (1 - u1/3 - u2/6)),
// and only the planet's edge inside the star moves with k or z, so
//   dI_g/dk = k int_arc g dphi,   dI_g/dz = k int_arc g cos(phi) dphi,
// complete elliptic integrals for g = mu.  The orbit part is the chain rule
// through z = sqrt(U^2 + V^2 cos^2 i), Kepler's equation (solved in the same
// differential FP32 form as the forward kernels) and the conjunction anchor.
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

constexpr float PI_F = 3.14159265358979f;

// cel(kc, 1, a, b) for two (a, b) pairs sharing kc and p = 1 (so the whole
// Landen sequence, including p, is shared): returns K and E.
__device__ __forceinline__ void ellke(float kc, float *K, float *E)
{
    float a1 = 1.0f, b1 = 1.0f;          // K
    float a2 = 1.0f, b2 = kc * kc;       // E
    float p = 1.0f, m = 1.0f, e = kc;
#pragma unroll 1
    for (int it = 0; it < 10; ++it) {
        float ip = pt::rcp_a(p);   // p, kc, e, m normal throughout (as in pt::cel2)
        float g = e * ip;
        float f = a1;
        a1 = fmaf(b1, ip, a1);
        b1 = 2.0f * fmaf(f, g, b1);
        f = a2;
        a2 = fmaf(b2, ip, a2);
        b2 = 2.0f * fmaf(f, g, b2);
        p += g;
        g = m;
        m = kc + m;
        if (fabsf(g - kc) <= g * 3e-4f) break;
        kc = 2.0f * pt::sqrt_a(e);
        e = kc * m;
    }
    float den = pt::rcp_a(m * (m + p));
    *K = (0.5f * PI_F) * fmaf(a1, m, b1) * den;
    *E = (0.5f * PI_F) * fmaf(a2, m, b2) * den;
}

// S(m) = int_0^{pi/2} sin^2 cos^2 / sqrt(1 - m sin^2): binomial series below
// m = 1/2 (terms fall as m^n n^-2; 24 terms reach 1e-9), closed form in K, E
// at and above it.  Term n is c_n (w_n - w_{n+1}) m^n with c_n the binomial
// coefficients of (1 - x)^(-1/2) and w_n = int_0^{pi/2} sin^(2n) = (pi/2)
// (2n-1)!!/(2n)!!; the coefficients are constants, formed at compile time,
// and the sum runs by Horner's rule.
struct S2C2Coef {
    float a[24];
};

constexpr S2C2Coef make_s2c2()
{
    S2C2Coef r{};
    double c = 1.0, w1 = 0.25 * 3.14159265358979323846, w2 = w1 * 0.75;
    for (int n = 0; n < 24; ++n) {
        r.a[n] = (float)(c * (w1 - w2));
        c *= (2.0 * n + 1.0) / (2.0 * n + 2.0);
        double w3 = w2 * (2.0 * n + 5.0) / (2.0 * n + 6.0);
        w1 = w2;
        w2 = w3;
    }
    return r;
}

__device__ __forceinline__ float s2c2_int(float m, float K, float E)
{
    if (m < 0.5f) {
        constexpr S2C2Coef C = make_s2c2();
        float s = C.a[23];
#pragma unroll
        for (int n = 22; n >= 0; --n) s = fmaf(s, m, C.a[n]);
        return s;
    }
    return ((2.0f - m) * E - 2.0f * (1.0f - m) * K) * pt::rcp_a(3.0f * m * m);   // m >= 1/2
}

// Derivatives d[0..5] = dI_1/dk, dI_1/dz, dI_mu/dk, dI_mu/dz, dI_mu2/dk,
// dI_mu2/dz of the overlap integrals, from the distances dd = z - (1 - p) and
// e1 = (1 + p) - z to the contacts (a caller that knows them better than
// their rounded difference passes them).
__device__ __forceinline__ void overlap_derivs(float p, float z, float dd, float e1, float *d, bool have_ke = false,
                                               float Kin = 0.0f, float Ein = 0.0f)
{
    for (int i = 0; i < 6; ++i) d[i] = 0.0f;
    if (!(e1 > 0.0f) || !(p > 0.0f)) return;
    if (p >= 1.0f && z <= p - 1.0f) return;
    float oma = e1 * (1.0f + z - p);
    float al = 1.0f - z * z - p * p;
    if (dd < 0.0f) {                                   // full circle inside the star
        // oma, -dd and z p are normal numbers here (as in pt::ma_terms)
        const float ioma = pt::rcp_a(oma);
        float m = 4.0f * z * p * ioma;
        float K = Kin, E = Ein;
        if (!have_ke) ellke(pt::sqrt_a(-dd * (1.0f + z + p) * ioma), &K, &E);
        float so = pt::sqrt_a(oma);
        d[0] = 2.0f * PI_F * p;
        d[2] = 4.0f * p * so * E;
        d[3] = -p * 4.0f * so * m * s2c2_int(m, K, E);
        d[4] = p * al * 2.0f * PI_F;
        d[5] = -p * 2.0f * z * p * PI_F;
        return;
    }
    float bm1 = dd * (1.0f + z + p);
    float fa = pt::sqrt_a(fmaxf(0.0f, oma * bm1));
    float kap0 = pt::atan2_pos(fa, p * p + z * z - 1.0f);
    float ipz = pt::rcp_a(2.0f * p * z);
    float sk = fa * ipz, ck = (p * p + z * z - 1.0f) * ipz;
    float m1 = 0.5f * oma * ipz, mc1 = 0.5f * bm1 * ipz;
    const float szp = pt::sqrt_a(z * p);
    float K, E, mcK;
    if (dd == 0.0f) {                                  // contact with the limb from inside: m1 = 1
        E = 1.0f;
        mcK = 0.0f;
    } else {
        if (have_ke) {
            K = Kin;
            E = Ein;
        } else {
            ellke(pt::sqrt_a(mc1), &K, &E);
        }
        mcK = mc1 * K;
    }
    float icos = -2.0f * sk, icos2 = kap0 + sk * ck;
    d[0] = 2.0f * p * kap0;
    d[1] = p * icos;
    d[2] = 8.0f * p * szp * (E - mcK);
    d[3] = -p * (8.0f / 3.0f) * szp * ((2.0f * m1 - 1.0f) * E + mcK);
    d[4] = p * (al * 2.0f * kap0 - 2.0f * z * p * icos);
    d[5] = p * (al * icos - 2.0f * z * p * icos2);
}

struct VecConst {
    pt::GeomRec g;          // phase reduction, window, anchor, position coefficients
    float q2, q3, xq;       // start of Newton's method: dE = x + q2 x^2 + q3 x^3, x = dM / (1 - e cos E_tr), for |x| <= xq
    float ci2, c0, c2, u2, invPD, inv3D, inv6D;   // c0 = 1 - u1 - u2, c2 = u1 + 2 u2; 1 / (pi D), 1 / (3 D), 1 / (6 D)
    float e, ise2, dci_a, dci_b, dci_e, dci_w, Ke, dMtr_dw, Wc;   // Wc = Us - e U'_tr
};

// By one whole warp: the anomalies at conjunction and at the two ends of the
// window are one evaluation, on lanes 2, 0 and 1 (three in a row on one lane
// were a third of a block's start).
__device__ void make_const(const pt_theta &th, int v, float half_exp, VecConst *c)
{
    const float PI2 = 6.28318530717958f;
    const int lane = threadIdx.x & 31;
    const double t0 = th.t0[v], P = th.P[v], iP = 1.0 / P;
    const float a = th.a[v], b = th.b[v], e = th.e ? th.e[v] : 0.0f, w = th.w ? th.w[v] : 0.5f * PI_F;
    const float k = th.k[v];
    float sw, cw;
    sincosf(w, &sw, &cw);
    const float ome2 = (1.0f - e) * (1.0f + e), se = sqrtf(ome2);
    const float ci = b * (1.0f + e * sw) / (a * ome2), ci2 = ci * ci;
    // conservative window (as the forward set-up): |sin th| > sqrt(((1+k)^2/rmin^2 - ci^2)/(1 - ci^2))
    const float rr = (1.0f + k) * 1.0001f + 1e-5f;
    const float rmin = a * (1.0f - e);
    const float s2 = (rr * rr / (rmin * rmin) - ci2) / fmaxf(1.0f - ci2, 1e-30f);
    const float thw = asinf(sqrtf(fminf(1.0f, fmaxf(s2, 0.0f)))) * 1.001f + 1e-5f;
    // eccentric and mean anomaly at true anomaly ftr (conjunction) and ftr -+ thw
    const float ftr = 0.5f * PI_F - w;
    const float f = ftr + (lane == 0 ? -thw : (lane == 1 ? thw : 0.0f));
    float sf, cf, sEf, cEf;
    sincosf(0.5f * f, &sf, &cf);
    const float Ef = 2.0f * atan2f(sqrtf(1.0f - e) * sf, sqrtf(1.0f + e) * cf);
    sincosf(Ef, &sEf, &cEf);
    const float Mf = Ef - e * sEf;
    const float sE = __shfl_sync(0xffffffffu, sEf, 2), cE = __shfl_sync(0xffffffffu, cEf, 2);
    const float Mtr = __shfl_sync(0xffffffffu, Mf, 2);
    float Ml = __shfl_sync(0xffffffffu, Mf, 0) - Mtr, Mh = __shfl_sync(0xffffffffu, Mf, 1) - Mtr;
    if (lane != 0) return;
    pt::GeomRec &r = c->g;
    r.t0h = (float)t0;
    r.t0l = (float)(t0 - (double)r.t0h);
    r.Ph = (float)P;
    r.Pl = (float)(P - (double)r.Ph);
    r.invP = (float)iP;
    r.nang = (float)(2.0 * 3.14159265358979323846 * iP);
    // conjunction anchor (FP32: it enters only as coefficients of small terms)
    const float ecEt = 1.0f - e * cE;
    c->e = e;
    c->ise2 = 1.0f / ome2;
    c->ci2 = ci2;
    c->dci_a = -ci / a;
    c->dci_b = (1.0f + e * sw) / (a * ome2);
    c->dci_e = b / a * (sw * ome2 + 2.0f * e * (1.0f + e * sw)) / (ome2 * ome2);
    c->dci_w = b / a * e * cw / ome2;
    c->dMtr_dw = -ecEt * ecEt / se;
    c->Ke = -ecEt * sE / ome2;   // dM_tr/de + sin E_tr
    // The series of E about E_tr in M has dE/dM = 1 / (1 - e cos E_tr) = E1,
    // then -e sin E E1^3 and (3 (e sin E)^2 E1 - e cos E) E1^4.  It is the start
    // where its last two terms are small against the first.
    {
        const float E1 = 1.0f / ecEt, s1 = e * sE * E1, c1 = e * cE * E1;
        c->q2 = -0.5f * s1;
        c->q3 = (3.0f * s1 * s1 - c1) * (1.0f / 6.0f);
        c->xq = fminf(0.5f, fminf(0.25f / (fabsf(c->q2) + 1e-6f), sqrtf(0.1f / (fabsf(c->q3) + 1e-6f))));
    }
    r.a = a;
    r.cosi = ci;
    r.k = k;
    r.ecc = 1.0f;
    r.ecE = e * cE;
    r.esE = e * sE;
    r.cE = cE;
    r.sE = sE;
    r.Uc = a * cw;
    r.Us = a * se * sw;
    r.Vs = a * sw;
    r.Vc = a * se * cw;
    r.Vtr = a * ecEt;
    c->Wc = r.Us + e * (r.Uc * sE + r.Us * cE) / ecEt;
    float lo, hi;
    const float full = 1.5f * (float)P;
    if (rmin * fabsf(ci) >= rr) {
        lo = 1.0f;
        hi = -1.0f;
    } else {
        const float margin = half_exp + 1e-6f + 1e-6f * (float)P;
        Ml = Ml - PI2 * floorf(Ml / PI2);
        Ml = (Ml > 0.0f) ? Ml - PI2 : 0.0f;
        Mh = Mh - PI2 * floorf(Mh / PI2);
        if (Mh >= PI2) Mh = 0.0f;
        if (s2 >= 1.0f || Mh - Ml >= 3.0f) {
            lo = -full;
            hi = full;
        } else {
            lo = Ml * 1.0005f / r.nang - margin;
            hi = Mh * 1.0005f / r.nang + margin;
        }
    }
    r.win_lo = lo;
    r.win_hi = hi;
    r.nq = e / (1.0f - e);
    r.pad1 = r.pad2 = 0.0f;
    const float u1 = th.u1[v], u2 = th.u2[v], D = 1.0f - u1 * (1.0f / 3.0f) - u2 * (1.0f / 6.0f);
    c->c0 = 1.0f - u1 - u2;
    c->c2 = u1 + 2.0f * u2;
    c->u2 = u2;
    c->invPD = 1.0f / (PI_F * D);
    c->inv3D = 1.0f / (3.0f * D);
    c->inv6D = 1.0f / (6.0f * D);
}

// The quantities that depend on the separation alone (for one vector's k, u1,
// u2): the depth 1 - F and dF/du1, dF/du2, dF/dk, dF/dz.
struct LimbTerms {
    float dep, du1, du2, dk, dz;
};
constexpr int N_LT = 5;

struct LimbConst {
    float c0, c2, u2, invPD, inv3D, inv6D;
};

__device__ __forceinline__ LimbTerms limb_terms(const LimbConst &c, float le, float ld, float ed, const float *d)
{
    const float I0 = PI_F * le, I1 = PI_F * ld, I2 = PI_F * (le - ed);
    LimbTerms o;
    o.dep = (c.c0 * I0 + c.c2 * I1 - c.u2 * I2) * c.invPD;
    o.du1 = -((I1 - I0) * c.invPD + o.dep * c.inv3D);
    o.du2 = -((2.0f * I1 - I0 - I2) * c.invPD + o.dep * c.inv6D);
    o.dk = -(c.c0 * d[0] + c.c2 * d[2] - c.u2 * d[4]) * c.invPD;
    o.dz = -(c.c0 * d[1] + c.c2 * d[3] - c.u2 * d[5]) * c.invPD;
    return o;
}

// From the exact terms, for the vectors that have no rows.
__device__ __forceinline__ LimbTerms limb_exact(const LimbConst &c, float p, float z)
{
    float le, ld, ed, Kc = 0.0f, Ec = 0.0f, d[6];
    bool have_ke = false;
    pt::ma_terms<true>(p, z, &le, &ld, &ed, &Kc, &Ec, &have_ke);
    if (!(z < 1.0f + p)) return LimbTerms{0.0f, 0.0f, 0.0f, 0.0f, 0.0f};
    overlap_derivs(p, z, (z - 1.0f) + p, (1.0f - z) + p, d, have_ke, Kc, Ec);
    return limb_terms(c, le, ld, ed, d);
}

// Rows: the five quantities as piecewise polynomials in the square root of
// the distance to the contacts, on the intervals of pt_device.cuh's row
// tables, made per vector in shared memory.  The derivatives have a
// w^2 log w term at the inner contact z = 1 - p (the depth only w^4 log w),
//   dI_mu/dk, dI_mu/dz ~ -+ 2 sqrt(p / (1 - p)) w^2 log w  (inside -, limb +),
// which the polynomial would miss by 1e-5 of the derivative in the first
// intervals: those carry it as a seventh coefficient, of t^2 log2 t, and the
// error is then below 1e-6 (dz) and 3e-7 (dk) of the largest derivative at
// k >= 0.1 and 3.4e-6 at GR_PMIN, in the second interval (measured in 64 bits;
// the FP32 elliptic integrals are good to about 1e-6).
// A row costs 144 evaluations of the exact terms, 5,000 to 6,000 warp
// instructions a vector; an evaluation from it is about 60 instructions
// against 350.
// Layout: 8 floats per (interval, quantity), interval-major.
constexpr float GR_PMIN = 0.02f;
constexpr int GR_ROW = 8 * N_LT * pt::MT_N;
constexpr unsigned GR_STEP = 32u * N_LT;   // bytes per interval

__device__ __forceinline__ float first_interval_log(int i, float p, float c2, float invPD)
{
    if (i != 0 && i != pt::MT_NA) return 0.0f;
    float sA, sL;
    pt::mt_scales(p, &sA, &sL);
    const float h = 1.0f / (i == 0 ? sA : sL);
    const float C = 2.0f * 0.69314718056f * sqrtf(p / (1.0f - p)) * c2 * invPD * h * h;
    return i == 0 ? C : -C;   // of dF = -dI / (pi D)
}

__device__ void row_node(const LimbConst &c, float p, int n, float *node)
{
    const int i = n / pt::MT_Q, q = n - i * pt::MT_Q;
    float le, ld, ed, d[6];
    pt::mt_node(p, i, q, &le, &ld, &ed);
    float z, dd, e1, t;
    pt::mt_node_at(p, i, q, &z, &dd, &e1, &t);
    overlap_derivs(p, z, dd, e1, d);
    const LimbTerms o = limb_terms(c, le, ld, ed, d);
    const float lg = first_interval_log(i, p, c.c2, c.invPD) * t * t * log2f(fmaxf(t, 1e-6f));
    node[0 * pt::MT_NODES + n] = o.dep;
    node[1 * pt::MT_NODES + n] = o.du1;
    node[2 * pt::MT_NODES + n] = o.du2;
    node[3 * pt::MT_NODES + n] = o.dk - lg;
    node[4 * pt::MT_NODES + n] = o.dz - lg;
}

// The polynomial at byte OFF of the interval's coefficients.
template <int OFF>
__device__ __forceinline__ float row_poly(unsigned at, float t)
{
    float4 c;
    float2 g;
    asm volatile("ld.shared.v4.f32 {%0, %1, %2, %3}, [%4+%5];"
                 : "=f"(c.x), "=f"(c.y), "=f"(c.z), "=f"(c.w) : "r"(at), "n"(OFF));
    asm volatile("ld.shared.v2.f32 {%0, %1}, [%2+%3];" : "=f"(g.x), "=f"(g.y) : "r"(at), "n"(OFF + 16));
    return fmaf(fmaf(fmaf(fmaf(fmaf(g.y, t, g.x), t, c.w), t, c.z), t, c.y), t, c.x);
}

__device__ __forceinline__ LimbTerms limb_row(unsigned base, float p, float sA, float sL, float z)
{
    const float zm1 = z - 1.0f;
    float t;
    const unsigned at = base + GR_STEP * pt::mt_find(p, sA, sL, zm1, pt::mt_off_limb(zm1), &t);
    LimbTerms o;
    o.dep = row_poly<0>(at, t);
    o.du1 = row_poly<32>(at, t);
    o.du2 = row_poly<64>(at, t);
    float lg, ck;   // the coefficient is the same for both derivatives
    asm("lg2.approx.ftz.f32 %0, %1;" : "=f"(lg) : "f"(fmaxf(t, 1e-6f)));
    asm volatile("ld.shared.f32 %0, [%1+120];" : "=f"(ck) : "r"(at));
    lg *= ck * t * t;
    o.dk = row_poly<96>(at, t) + lg;
    o.dz = row_poly<128>(at, t) + lg;
    return o;
}

// The sums from which the gradient is formed.  With G = (dF/dz) / z and
// dz/dtheta = (U dU/dtheta + cos^2 i V dV/dtheta + V^2 cos i d cos i/dtheta) / z,
// every parameter's derivative is a combination, with the vector's constants,
// of a few sums over the points; per point that leaves about 25 instructions
// against 90 for the derivative of each parameter.  X = dE/dM G (U dU/dE +
// cos^2 i V dV/dE) is the derivative by the mean anomaly.  The derivative by w
// is summed per point (S_W): of its two parts, the turn of the orbit and the
// shift of the anomaly that keeps the conjunction at t0, all but the order of
// e dM cancels, which is taken out beforehand (kap = dM_tr/dw),
//   dU/dw = kap U' - V = -(kap dE/dM (Uc dS + Wc dC) + (V - V_tr)),  dV/dw = kap V' + U.
enum { S_X, S_XT, S_XS, S_VV, S_UU, S_W, S_U, S_V, S_US, S_VS, S_K, S_U1, S_U2, S_SSR, N_SUM };

struct PointConst {   // the registers of the loop over points
    float nang, ecE, esE, nq, E1, q2, q3, xq, cE, sE, Uc, Us, Vs, Vc, Vtr, ci2, ci, invP, kap, Wc;
    float k, sA, sL;
    unsigned base;
    LimbConst lc;   // the exact terms' weights
};

// Adds w times the point's terms to S; returns the depth.
template <bool ROWS>
__device__ __forceinline__ float point_sums(const PointConst &c, float dts, float n_ep, int max_iter, bool *bad,
                                            float yw, float w, bool ss1, float *S)
{
    // Newton's method on Kepler's equation relative to the conjunction anchor,
    // with pt::orbit_z's stopping rule (the error left is below 3e-8 |dE|).
    // From the third-order start it takes one step over a transit.
    const float dM = c.nang * dts;
    float dE = dM * c.E1;
    if (fabsf(dE) <= c.xq) dE = fmaf(dE * dE, fmaf(dE, c.q3, c.q2), dE);
    float sh = 0.0f, ch = 1.0f, step = 0.0f;
    bool conv = false;
    for (int it = 0; it < max_iter; ++it) {
        pt::sincos_near0(0.5f * dE, &sh, &ch);
        const float sn = 2.0f * sh * ch, omc = 2.0f * sh * sh;
        const float F = (dE - c.ecE * sn) + (c.esE * omc - dM);
        const float Fp = 1.0f - c.ecE * (1.0f - omc) + c.esE * sn;
        step = F * pt::rcp_a(Fp);   // Fp lies in [1 - e, 1 + e]
        dE -= step;
        if (c.nq * step * step <= 6e-8f * fabsf(dE) + 1e-12f) {
            conv = true;
            break;
        }
        if (it + 1 >= pt::KEPLER_FREE) dE = pt::kepler_bracket(dE, dM, c.esE, c.nq);
    }
    if (!conv) *bad = true;
    // sin and cos of dE/2 at the solution (as in pt::orbit_z)
    const float h = 0.5f * step;
    const float cr = fmaf(-0.5f * h, h, 1.0f);
    const float s1 = fmaf(-ch, h, sh * cr);
    ch = fmaf(sh, h, ch * cr);
    const float sn = 2.0f * s1 * ch, omc = 2.0f * s1 * s1;
    const float dC = -c.cE * omc - c.sE * sn;
    const float dS = c.cE * sn - c.sE * omc;
    const float U = c.Uc * dC - c.Us * dS;
    const float dV = c.Vs * dC + c.Vc * dS;
    const float V = c.Vtr + dV;
    if (V <= 0.0f) return 0.0f;
    const float Vi = V * c.ci;
    // z and w dF/dz / z: approximate root and reciprocal, each once corrected by its
    // remainder, for the errors of sqrtf and a division (4,096 vectors x 10,000 times:
    // 182 us so, 195 with those two, 179 uncorrected).  At z = 0 dF/dz is 0 but for a
    // row's rounding; z is then 1e-18.
    const float zz = fmaxf(fmaf(U, U, Vi * Vi), 1e-36f), z0 = pt::sqrt_a(zz), iz = pt::rcp_a(z0);
    const float z = fmaf(0.5f * fmaf(-z0, z0, zz), iz, z0);
    const LimbTerms l = ROWS ? limb_row(c.base, c.k, c.sA, c.sL, z) : limb_exact(c.lc, c.k, z);
    if (ss1) w *= 2.0f * (yw - l.dep);   // one supersample: w is the point's weight
    const float cE = c.cE + dC, sE = c.sE + dS;
    const float iecE = pt::rcp_a(1.0f - c.ecE * (1.0f - omc) + c.esE * sn);   // 1 - e cos E
    const float wdz = w * l.dz, g0 = wdz * iz, G = fmaf(fmaf(-g0, z, wdz), iz, g0);
    const float GU = G * U, GV = G * V;
    const float GVc = GV * c.ci2, Vp = iecE * (c.Vc * cE - c.Vs * sE);
    const float X = GVc * Vp - GU * (iecE * (c.Uc * sE + c.Us * cE));
    const float Uw = fmaf(c.kap * iecE, fmaf(c.Uc, dS, c.Wc * dC), dV);   // -dU/dw
    S[S_W] += GVc * fmaf(c.kap, Vp, U) - GU * Uw;
    S[S_X] += X;
    S[S_XT] = fmaf(X, fmaf(dts, c.invP, n_ep), S[S_XT]);
    S[S_XS] = fmaf(X, dS, S[S_XS]);
    S[S_VV] = fmaf(GV, V, S[S_VV]);
    S[S_UU] = fmaf(GU, U, S[S_UU]);
    S[S_U] += GU;
    S[S_V] += GV;
    S[S_US] = fmaf(GU, dS, S[S_US]);
    S[S_VS] = fmaf(GV, dS, S[S_VS]);
    S[S_K] = fmaf(w, l.dk, S[S_K]);
    S[S_U1] = fmaf(w, l.du1, S[S_U1]);
    S[S_U2] = fmaf(w, l.du2, S[S_U2]);
    return l.dep;
}

// dSSR/dtheta_j from the sums, theta = (t0, P, a, b, e, w, k, u1, u2).  M =
// n (t - t0 - n_ep P) moves with t0 and P, E with e and w also through the
// anchor, U and V with a in proportion, and cos i with a, b, e, w.
__device__ __forceinline__ float gradient_of(const VecConst &c, const float *S, int j)
{
    const pt::GeomRec &r = c.g;
    const float ci = r.cosi, bv = ci * S[S_VV], gu = S[S_U], gv = c.ci2 * S[S_V];
    if (j == 2) return (S[S_UU] + ci * bv) / r.a + c.dci_a * bv;
    if (j == 3) return c.dci_b * bv;
    if (j == 4)
        return S[S_XS] + c.Ke * S[S_X] - (r.Uc * gu + r.Vs * gv) -
               c.e * c.ise2 * (r.Vc * (r.sE * gv + c.ci2 * S[S_VS]) - r.Us * (r.sE * gu + S[S_US])) + c.dci_e * bv;
    if (j == 5)   // a circular orbit does not depend on w: the terms cancel, and their rounding is left out
        return c.e == 0.0f ? 0.0f : S[S_W] + c.dci_w * bv;
    if (j < 2) return -r.nang * S[j == 0 ? S_X : S_XT];
    return S[S_K + j - 6];
}

struct BwdArgs {
    const float2 *tsplit;
    const float2 *tile_mm;    // [n_tiles] smallest and largest time of each tile of TT times
    const double *tile_ssr;   // [n_tiles] sum of wt (y - 1)^2 over each tile
    int n_t;
    pt_theta th;
    int n_ss;
    float t_exp;
    int max_iter;
    const float *y, *wt;
    float *grad, *ssr, *flux;
    int *n_bad;
};

// Per tile of TT times (one CTA of TT threads): the double-float split of
// each time, the tile's smallest and largest time (rounded outward to FP32)
// and the residual sum of its times with the flux at 1, sum wt (y - 1)^2, in
// FP64 and a fixed order.  The adjoint kernel skips tiles that meet no
// transit window, where the flux is exactly 1 and every derivative zero, and
// takes their residual sums from here.
constexpr int TT = 64;   // times per tile

// Blocks of 384 threads for few vectors, where the chip has room and a
// vector's passes are one chain.  Two of them fit on an SM: as many vectors
// as that take one wave (304 vectors x 3,000 times 16.4 us, in blocks of 128
// 18.5; x 40,000 49.1 and 83.3; x 30 to 300 the same to 2 us).  Vectors of a
// second wave pay its start: 400 x 301 18.5 us and 12.4, x 3,000 24.6 and
// 18.6, so up to 600 vectors they come in wide blocks only where they are long,
// from about 12,000 points (400 x 10,000 32.8 and 34.9, 599 x 20,000 54.9 and
// 57.4; 599 x 5,000 x 3 supersamples 50.5 and 49.2, x 10,000 x 3 74.1 and 81.1).
constexpr int WIDE_PER_SM = 2, WIDE_MAX_VECTORS = 600, WIDE_LONG_POINTS = 12000;

// Rows pay from about 1,280 in-transit points a vector (4,096 vectors, a
// quarter of the points in transit: 3,000 times 93 us with rows, 82 with the
// exact terms; 2,000 x 3 supersamples at 3,000 vectors 103 and 108; 10,000
// times 167 and 197).  Their number is estimated, from the length of a
// central transit, P (1 + k) / (pi a), and the span of the times as evenly
// covered; it depends neither on the order of the times nor on the window,
// which is not known yet.
constexpr float ROWS_MIN_POINTS = 1280.0f;
__device__ bool rows_pay(float a, float P, float k, float n, const float2 *tile_mm, int n_tiles)
{
    if (n < ROWS_MIN_POINTS) return false;
    float lo = INFINITY, hi = -INFINITY;
    for (int j = threadIdx.x & 31; j < n_tiles; j += 32) {
        const float2 mm = tile_mm[j];
        lo = fminf(lo, mm.x);
        hi = fmaxf(hi, mm.y);
    }
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) {
        lo = fminf(lo, __shfl_xor_sync(0xffffffffu, lo, o));
        hi = fmaxf(hi, __shfl_xor_sync(0xffffffffu, hi, o));
    }
    const float length = P * (1.0f + k) / (PI_F * a);
    return n * length >= ROWS_MIN_POINTS * fmaxf(length, fminf(P, hi - lo));
}

__global__ void __launch_bounds__(TT) tile_kernel(const double *t, const float *y, const float *wt, int n,
                                                  float2 *tsplit, float2 *tile_mm, double *tile_ssr)
{
    pt::chain_next();
    __shared__ double smin[TT / 32], smax[TT / 32], ssum[TT / 32];
    const int i = blockIdx.x * TT + threadIdx.x;
    double lo = INFINITY, hi = -INFINITY, r2 = 0.0;
    if (i < n) {
        const double x = t[i];
        const float h = (float)x;
        tsplit[i] = make_float2(h, (float)(x - (double)h));
        lo = hi = x;
        const double r = 1.0 - (double)y[i];
        r2 = (wt ? (double)wt[i] : 1.0) * r * r;
    }
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) {
        lo = fmin(lo, __shfl_xor_sync(0xffffffffu, lo, o));
        hi = fmax(hi, __shfl_xor_sync(0xffffffffu, hi, o));
        r2 += __shfl_xor_sync(0xffffffffu, r2, o);
    }
    if (lane == 0) {
        smin[warp] = lo;
        smax[warp] = hi;
        ssum[warp] = r2;
    }
    __syncthreads();
    if (threadIdx.x == 0) {
        for (int w = 1; w < TT / 32; ++w) {
            lo = fmin(lo, smin[w]);
            hi = fmax(hi, smax[w]);
            r2 += ssum[w];
        }
        float flo = (float)lo, fhi = (float)hi;
        if ((double)flo > lo) flo = nextafterf(flo, -INFINITY);
        if ((double)fhi < hi) fhi = nextafterf(fhi, INFINITY);
        tile_mm[blockIdx.x] = make_float2(flo, fhi);
        tile_ssr[blockIdx.x] = r2;
    }
}

// Can a time in [tmin, tmax] lie in the transit window of some epoch,
// t - t0 - n P in [win_lo, win_hi]?  That is, is there an integer n with
// (tmin - t0 - win_hi) / P <= n <= (tmax - t0 - win_lo) / P?  The interval
// is widened by m, 1e-6 of the magnitudes involved, which exceeds the FP32
// rounding of these expressions, so the test never misses an epoch.
__device__ __forceinline__ bool tile_meets_window(const pt::GeomRec &g, float tmin, float tmax)
{
    if (g.win_lo > g.win_hi) return false;                // never in transit
    if (g.win_hi - g.win_lo >= 0.5f * g.Ph) return true;  // a wide window: no test
    const float m = 1e-6f * (fabsf(tmin) + fabsf(tmax) + fabsf(g.t0h) + g.Ph) + 1e-9f;
    const float n_lo = ceilf((tmin - g.t0h - g.win_hi - m) * g.invP);
    const float n_hi = floorf((tmax - g.t0h - g.win_lo + m) * g.invP);
    return n_lo <= n_hi;
}


// One vector's points: the sums of this thread's share, and its share of the
// skipped tiles' residual sums.
template <int TB, bool SS1, bool ROWS>
__device__ __forceinline__ void vector_sums(const BwdArgs &A, const VecConst &sc, const float *srow, int *slist,
                                            int *swcnt, float *acc, double *ssr_skipped, bool *bad_out)
{
    constexpr int NW = TB / 32;
    const int v = blockIdx.x;
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    PointConst c;
    {
        const pt::GeomRec &r = sc.g;
        c.nang = r.nang;
        c.ecE = r.ecE;
        c.esE = r.esE;
        c.nq = r.nq;
        c.E1 = 1.0f / (1.0f - r.ecE);
        c.q2 = sc.q2;
        c.q3 = sc.q3;
        c.xq = sc.xq;
        c.cE = r.cE;
        c.sE = r.sE;
        c.Uc = r.Uc;
        c.Us = r.Us;
        c.Vs = r.Vs;
        c.Vc = r.Vc;
        c.Vtr = r.Vtr;
        c.ci = r.cosi;
        c.ci2 = sc.ci2;
        c.kap = sc.dMtr_dw;
        c.Wc = sc.Wc;
        c.invP = r.invP;
        c.k = r.k;
        pt::mt_scales(r.k, &c.sA, &c.sL);
        c.base = (unsigned)__cvta_generic_to_shared(srow) - GR_STEP * pt::MT_BITS0;
        c.lc = LimbConst{sc.c0, sc.c2, sc.u2, sc.invPD, sc.inv3D, sc.inv6D};
    }
    const pt::GeomRec &g = sc.g;
    bool bad = false;
    const float inv_ss = 1.0f / (float)A.n_ss;
    const int n_tiles = (A.n_t + TT - 1) / TT;
    double ssr_out = 0.0;   // this thread's share of the skipped tiles' residual sums
    // Tile j holds times j TT .. j TT + TT - 1.  A tile that meets no transit
    // window has flux 1 and zero derivatives: it is skipped and its residual
    // sum comes from tile_kernel.  Chunks of TB tiles: one window test per
    // thread, the evaluated tiles listed in order in shared memory, then
    // passes over TB / TT of them at a time (thread tid takes time tid % TT of
    // list entry tid / TT), each pass's inputs loaded during the previous one.
    constexpr int TPP = TB / TT;   // tiles per pass
    for (int c0 = 0; c0 < n_tiles; c0 += TB) {
        const int jt = c0 + (int)threadIdx.x;
        bool ev = false;
        if (jt < n_tiles) {
            const float2 mm = A.tile_mm[jt];
            ev = tile_meets_window(g, mm.x, mm.y);
            if (!ev) ssr_out += A.tile_ssr[jt];
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
        if (A.flux) {
            // flux 1 on this chunk's skipped tiles: thread tid writes time
            // tid % TT of every (TB / TT)-th tile
            const int c1 = min(n_tiles, c0 + TB);
            for (int tj = c0 + (int)(threadIdx.x / TT); tj < c1; tj += TPP) {
                const int i = tj * TT + (int)(threadIdx.x % TT);
                const float2 mm = A.tile_mm[tj];
                if (i < A.n_t && !tile_meets_window(g, mm.x, mm.y)) A.flux[(size_t)v * A.n_t + i] = 1.0f;
            }
        }
        __syncthreads();
        // pass q takes list entries q TPP .. q TPP + TPP - 1
        auto time_of = [&](int q) {
            const int e = q * TPP + (int)(threadIdx.x / TT);
            return e < n_ev ? slist[e] * TT + (int)(threadIdx.x % TT) : -1;
        };
        const int n_pass = (n_ev + TPP - 1) / TPP;
        int i_n = n_pass > 0 ? time_of(0) : -1;
        float2 ts_n = make_float2(0.0f, 0.0f);
        float y_n = 0.0f, w_n = 1.0f;
        if (i_n >= 0 && i_n < A.n_t) {
            ts_n = A.tsplit[i_n];
            y_n = A.y[i_n];
            w_n = A.wt ? A.wt[i_n] : 1.0f;
        }
        for (int q = 0; q < n_pass; ++q) {
            const int i = i_n;
            const float2 ts = ts_n;
            const float yw = 1.0f - y_n, wi = w_n;
            i_n = q + 1 < n_pass ? time_of(q + 1) : -1;
            if (i_n >= 0 && i_n < A.n_t) {
                ts_n = A.tsplit[i_n];
                y_n = A.y[i_n];
                w_n = A.wt ? A.wt[i_n] : 1.0f;
            }
            if (i < 0 || i >= A.n_t) continue;
            // epoch and offset (double-float phase reduction)
            const float n_ep = rintf((ts.x - g.t0h) * c.invP);
            const float dt = pt::reduce_time(ts.x, ts.y, g);
            float dep = 0.0f;
            const bool inw = dt >= g.win_lo && dt <= g.win_hi;
            if (SS1) {
                if (inw) dep = point_sums<ROWS>(c, dt, n_ep, A.max_iter, &bad, yw, wi, true, acc);
            } else {
                float S[N_SUM];
#pragma unroll
                for (int j = 0; j < N_SUM; ++j) S[j] = 0.0f;
                if (inw) {
                    for (int ss = 0; ss < A.n_ss; ++ss) {
                        const float dts = dt + A.t_exp * (((float)ss + 0.5f) * inv_ss - 0.5f);
                        dep += point_sums<ROWS>(c, dts, n_ep, A.max_iter, &bad, 0.0f, inv_ss, false, S);
                    }
                    dep *= inv_ss;
                }
                const float tw = 2.0f * wi * (yw - dep);
#pragma unroll
                for (int j = 0; j < S_SSR; ++j) acc[j] = fmaf(tw, S[j], acc[j]);
            }
            const float res = yw - dep;
            acc[S_SSR] = fmaf(wi * res, res, acc[S_SSR]);
            if (A.flux) A.flux[(size_t)v * A.n_t + i] = 1.0f - dep;
        }
    }
    *ssr_skipped = ssr_out;
    *bad_out = bad;
}

// One block per vector.  What bounds it: instruction issue (65% of the cycles;
// 4,096 vectors x 10,000 times, a quarter in transit: 290 instructions per
// warp of in-transit points, 9,000 per vector for its constants, row and sums).  Measured
// there 183 us against 274 when every point took the exact terms (540
// instructions) and the derivative of each parameter by itself; with the exact
// terms and these sums it is 197.  72 registers: seven blocks per multiprocessor
// (six took 3% longer, eight the same).
template <int TB, bool SS1>
__global__ void __launch_bounds__(TB, 896 / TB) ma_bwd_kernel(BwdArgs A)
{
    pt::chain_next();
    constexpr int NW = TB / 32;
    __shared__ VecConst sc;
    __shared__ __align__(16) float srow[GR_ROW];
    __shared__ float snode[N_LT * pt::MT_NODES];
    __shared__ float sred[NW][N_SUM];
    __shared__ float ssum[N_SUM];
    __shared__ double sout[NW];
    __shared__ int slist[TB];          // the current chunk's evaluated tiles, in order
    __shared__ int swcnt[NW];
    __shared__ int sbad;
    __shared__ bool srows;
    const int v = blockIdx.x;
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    const float k = A.th.k[v];
    // The first warp forms the vector's constants; the warps beside it evaluate the
    // row's nodes, two the 48 inside the disk (double-float terms), the others
    // those across the limb.
    if (warp == 0) make_const(A.th, v, 0.5f * A.t_exp, &sc);
    if (threadIdx.x == 0) sbad = 0;
    // the inputs were there before tile_kernel was launched; its results are waited for here
    pt::chain_wait();
    if (warp > 0) {
        const bool r = k >= GR_PMIN && k <= pt::MT_PMAX &&
                       rows_pay(A.th.a[v], (float)A.th.P[v], k, (float)A.n_t * (float)A.n_ss, A.tile_mm,
                                (A.n_t + TT - 1) / TT);
        if (threadIdx.x == 32) srows = r;
        if (r) {
            const float u1 = A.th.u1[v], u2 = A.th.u2[v], D = 1.0f - u1 * (1.0f / 3.0f) - u2 * (1.0f / 6.0f);
            const LimbConst lc{1.0f - u1 - u2, u1 + 2.0f * u2, u2, 1.0f / (PI_F * D), 1.0f / (3.0f * D),
                               1.0f / (6.0f * D)};
            constexpr int NIN = pt::MT_Q * pt::MT_NA;
            const int n0 = warp <= 2 ? (int)threadIdx.x - 32 : NIN + (int)threadIdx.x - 96;
            const int end = warp <= 2 ? NIN : pt::MT_NODES, step = warp <= 2 ? 64 : TB - 96;
            for (int n = n0; n < end; n += step) row_node(lc, k, n, snode);
        }
    }
    __syncthreads();
    const bool rows = srows;
    if (rows) {
        // one thread per (interval, quantity): the matrix entries are then the same for a warp's lanes
        const int j = threadIdx.x;
        if (j < N_LT * pt::MT_N) {
            const int i = j / N_LT, f = j - i * N_LT;
            float x[pt::MT_Q];
#pragma unroll
            for (int q = 0; q < pt::MT_Q; ++q) x[q] = snode[f * pt::MT_NODES + i * pt::MT_Q + q];
#pragma unroll
            for (int q = 0; q < pt::MT_Q; ++q) srow[8 * j + q] = pt::mt_coef(i, q, x);
            if (f == 3) srow[8 * j + 6] = first_interval_log(i, k, sc.c2, sc.invPD);
        }
        __syncthreads();
    }
    float acc[N_SUM];
#pragma unroll
    for (int i = 0; i < N_SUM; ++i) acc[i] = 0.0f;
    double ssr_out;
    bool bad;
    if (rows)
        vector_sums<TB, SS1, true>(A, sc, srow, slist, swcnt, acc, &ssr_out, &bad);
    else
        vector_sums<TB, SS1, false>(A, sc, srow, slist, swcnt, acc, &ssr_out, &bad);
    if (bad) atomicAdd(&sbad, 1);
    // deterministic block reduction (the skipped tiles' sums in FP64)
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) ssr_out += __shfl_xor_sync(0xffffffffu, ssr_out, o);
    if (lane == 0) sout[warp] = ssr_out;
#pragma unroll
    for (int j = 0; j < N_SUM; ++j) {
        float x = acc[j];
#pragma unroll
        for (int o = 16; o > 0; o >>= 1) x += __shfl_xor_sync(0xffffffffu, x, o);
        if (lane == 0) sred[warp][j] = x;
    }
    __syncthreads();
    if (threadIdx.x < N_SUM) {
        float x = 0.0f;
        for (int w = 0; w < NW; ++w) x += sred[w][threadIdx.x];
        ssum[threadIdx.x] = x;
    }
    __syncthreads();
    if (threadIdx.x < 9) A.grad[(size_t)v * 9 + threadIdx.x] = gradient_of(sc, ssum, threadIdx.x);
    if (threadIdx.x == 32 && A.ssr) {
        double so = 0.0;
        for (int w = 0; w < NW; ++w) so += sout[w];
        A.ssr[v] = (float)((double)ssum[S_SSR] + so);
    }
    if (threadIdx.x == 0 && sbad && A.n_bad) atomicAdd(A.n_bad, sbad);
}

}  // namespace

extern "C" {

// work buffer: [n_t] time split, then per tile of TT times its time range
// and its residual sum with the flux at 1, each part 256-byte aligned
static size_t bwd_split_bytes(int n_t) { return ((size_t)n_t * sizeof(float2) + 255) & ~(size_t)255; }
static size_t bwd_tiles(int n_t) { return ((size_t)n_t + TT - 1) / TT; }

size_t pt_ma_quad_bwd_work_bytes(int n_t)
{
    if (n_t <= 0) return 256;
    const size_t nt = bwd_tiles(n_t);
    return bwd_split_bytes(n_t) + ((nt * sizeof(float2) + 255) & ~(size_t)255) + ((nt * sizeof(double) + 255) & ~(size_t)255);
}

int pt_ma_quad_bwd(const double *t, int n_t, const pt_theta *th, int n_ss, double t_exp, int max_iter,
                   const float *y, const float *wt, float *grad, float *ssr, float *flux, void *work,
                   size_t work_bytes, int *n_bad, pt_stream_t stream)
{
    if (!th || th->n_v < 0 || n_t < 0 || n_ss < 1 || n_ss > 256 || max_iter < 1 || max_iter > 64)
        return PT_ERR_ARG;
    if (!(t_exp >= 0.0 && t_exp < 1.0e30))
        return pt_internal::set_error(PT_ERR_DOMAIN, "pt_ma_quad_bwd", "exposure time must be finite and >= 0");
    if (n_t == 0 || th->n_v == 0) return PT_OK;
    if (!th->t0 || !th->P || !th->a || !th->b || !th->k || !th->u1 || !th->u2) return PT_ERR_ARG;
    if ((th->e == nullptr) != (th->w == nullptr)) return PT_ERR_ARG;
    if (!t || !y || !grad) return PT_ERR_ARG;
    if (!work) return PT_ERR_WORKSPACE;
    if (work_bytes < pt_ma_quad_bwd_work_bytes(n_t)) return PT_ERR_WORKSPACE;
    if (th->n_v > 0x7fffffff) return PT_ERR_ARG;
    if (((uintptr_t)work & 15u) != 0u)
        return pt_internal::set_error(PT_ERR_WORKSPACE, "pt_ma_quad_bwd", "work buffer must be 16-byte aligned");
    cudaStream_t s = (cudaStream_t)stream;
    const size_t nt = bwd_tiles(n_t);
    float2 *ts = (float2 *)work;
    float2 *tmm = (float2 *)((char *)work + bwd_split_bytes(n_t));
    double *tssr = (double *)((char *)tmm + ((nt * sizeof(float2) + 255) & ~(size_t)255));
    tile_kernel<<<(unsigned)nt, TT, 0, s>>>(t, y, wt, n_t, ts, tmm, tssr);
    cudaError_t e = cudaGetLastError();
    if (e != cudaSuccess) return pt_internal::set_error(PT_ERR_CUDA, "tile_kernel", cudaGetErrorString(e));
    BwdArgs A;
    A.tsplit = ts;
    A.tile_mm = tmm;
    A.tile_ssr = tssr;
    A.n_t = n_t;
    A.th = *th;
    A.n_ss = n_ss;
    A.t_exp = (float)t_exp;
    A.max_iter = max_iter;
    A.y = y;
    A.wt = wt;
    A.grad = grad;
    A.ssr = ssr;
    A.flux = flux;
    A.n_bad = n_bad;
    int dev = 0, n_sm = 0;
    e = cudaGetDevice(&dev);
    if (e == cudaSuccess) e = cudaDeviceGetAttribute(&n_sm, cudaDevAttrMultiProcessorCount, dev);
    if (e != cudaSuccess) return pt_internal::set_error(PT_ERR_CUDA, "SM count", cudaGetErrorString(e));
    if (th->n_v > (n_t * (int64_t)n_ss < WIDE_LONG_POINTS ? WIDE_PER_SM * n_sm : WIDE_MAX_VECTORS - 1))
        pt::launch_chained(n_ss == 1 ? ma_bwd_kernel<128, true> : ma_bwd_kernel<128, false>, th->n_v, 128, 0, s, A);
    else
        pt::launch_chained(n_ss == 1 ? ma_bwd_kernel<384, true> : ma_bwd_kernel<384, false>, th->n_v, 384, 0, s, A);
    e = cudaGetLastError();
    return e == cudaSuccess ? PT_OK : pt_internal::set_error(PT_ERR_CUDA, "ma_bwd_kernel", cudaGetErrorString(e));
}

}  // extern "C"
