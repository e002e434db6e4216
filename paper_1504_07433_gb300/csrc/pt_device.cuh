// pt_device.cuh -- device-side building blocks of the transit-model kernels.
//
// Everything here is FP32 except where a comment says otherwise.  The
// numerical choices are documented next to the code; the formulas follow
// Parviainen (2015) Sec. 2.2.1, Eq. (ma_model), with the lambda/eta functions
// of Mandel & Agol (2002), which the paper defers to.
#pragma once

#include <cuda_runtime.h>
#include <math.h>
#include <stdint.h>

#define PT_PI_F 3.14159265358979f
#define PT_ZBEHIND 1.0e30f

namespace pt {

// ---------------------------------------------------------------------------
// Per-geometry record, written by the set-up kernel and staged in shared
// memory by the light-curve kernels.  One record per (vector) or, when every
// passband has its own radius ratio, per (vector, passband).
//
// Time is reduced in double-float arithmetic: t0 and P are split into a
// high float and the float of the remainder, so that t - t0 - n P keeps
// ~1e-11 d absolute accuracy at |t| ~ 1e3 d without FP64 instructions on the
// hot path.  The eccentric-orbit anchor (the eccentric anomaly at
// conjunction) is computed in FP64 by the set-up kernel and enters the hot
// path only multiplied by small quantities (see orbit_z below).
// ---------------------------------------------------------------------------
struct __align__(16) GeomRec {
    float t0h, t0l, Ph, Pl;   // double-float t0 and P
    float invP, nang;         // 1/P, 2 pi / P
    float win_lo, win_hi;     // transit window in (t - t0 - nP) [days]; empty if lo > hi
    float a, cosi, k, ecc;    // a/R*, cos i, radius ratio, 0 = circular / 1 = eccentric
    float ecE, esE, cE, sE;   // e cos E_tr, e sin E_tr, cos E_tr, sin E_tr
    float Uc, Us, Vs, Vc;     // a cos w, a sqrt(1-e^2) sin w, a sin w, a sqrt(1-e^2) cos w
    float Vtr, nq, pad1, pad2;    // r at conjunction = a (1 - e cos E_tr); e / (1 - e) (Newton's error factor)
};
static_assert(sizeof(GeomRec) == 96, "GeomRec layout");

// t - t0 - n P for the nearest epoch n, in double-float arithmetic.
// (th, tl) is the double-float split of t.  Two-sum error terms are exact.
__device__ __forceinline__ float reduce_time(float th, float tl, const GeomRec &r)
{
    float s = th - r.t0h;
    float bv = s - th;
    float e1 = (th - (s - bv)) + (-r.t0h - bv);
    float n = rintf(s * r.invP);
    float p = n * r.Ph;
    float pe = fmaf(n, r.Ph, -p);          // n*Ph = p + pe exactly
    float d = s - p;
    float bv2 = d - s;
    float e2 = (s - (d - bv2)) + (-p - bv2);
    float lo = ((e1 + e2) - pe) + (tl - r.t0l) - n * r.Pl;
    return d + lo;
}

// One-instruction hardware approximations (PTX rcp.approx.ftz, sqrt.approx.ftz:
// about one ulp, denormal inputs and results flushed to zero).  Without the
// .ftz form each call also carries the scaling that handles denormals.  The
// Mandel-Agol core uses them only where its arguments are normal numbers or
// exact zeros by construction (stated at each use).
__device__ __forceinline__ float rcp_a(float x)
{
    float r;
    asm("rcp.approx.ftz.f32 %0, %1;" : "=f"(r) : "f"(x));
    return r;
}
__device__ __forceinline__ float sqrt_a(float x)
{
    float r;
    asm("sqrt.approx.ftz.f32 %0, %1;" : "=f"(r) : "f"(x));
    return r;
}

// The same, or the correctly rounded forms (for the nodes of tables that are
// read many times: their cost is shared, and so is their error).
template <bool IEEE>
__device__ __forceinline__ float rcp_t(float x) { return IEEE ? __frcp_rn(x) : rcp_a(x); }
template <bool IEEE>
__device__ __forceinline__ float sqrt_t(float x) { return IEEE ? __fsqrt_rn(x) : sqrt_a(x); }

// ---------------------------------------------------------------------------
// Double-float arithmetic, for the few values that many others are formed
// from (the Gimenez table recursion, the nodes of the row tables): a value is
// the unevaluated sum h + l of two floats (about 48 significant bits).  Sums
// and products carry their rounding errors exactly (Knuth's two-sum; the FMA
// form of Dekker's product); reciprocal and root are one Newton correction of
// the FP32 ones.  GB300's FP64 rate is a small fraction of its FP32 rate, so
// FP64 operations would dominate that work.
// ---------------------------------------------------------------------------
struct DF {
    float h, l;
};

__device__ __forceinline__ DF df_of(double v)
{
    float h = (float)v;
    return DF{h, (float)(v - (double)h)};
}

__device__ __forceinline__ DF df_norm(float s, float e)   // |s| >= |e|
{
    float h = s + e;
    return DF{h, e - (h - s)};
}

__device__ __forceinline__ DF df_add(DF a, DF b)
{
    float s = a.h + b.h;
    float bb = s - a.h;
    float e = (a.h - (s - bb)) + (b.h - bb);
    return df_norm(s, e + (a.l + b.l));
}

__device__ __forceinline__ DF df_neg(DF a) { return DF{-a.h, -a.l}; }

__device__ __forceinline__ DF df_mul(DF a, DF b)
{
    float p = a.h * b.h;
    float e = fmaf(a.h, b.h, -p);
    e = fmaf(a.h, b.l, fmaf(a.l, b.h, e));
    return df_norm(p, e);
}

__device__ __forceinline__ DF df_scale(float a, DF b)   // a a power of two
{
    return DF{a * b.h, a * b.l};
}

// a b + c with one two-sum: the product's rounding error (fmaf), the two-sum
// error of p + c_h, the cross terms and c_l go into the low part
__device__ __forceinline__ DF df_mad(DF a, DF b, DF c)
{
    const float p = a.h * b.h;
    const float e = fmaf(a.h, b.h, -p);
    const float s = p + c.h;
    const float bb = s - p;
    const float err = (p - (s - bb)) + (c.h - bb);
    return df_norm(s, fmaf(a.h, b.l, fmaf(a.l, b.h, c.l)) + (e + err));
}

__device__ __forceinline__ DF df_rcp(DF a)   // a normal
{
    const float x = rcp_a(a.h);
    const float e = fmaf(-a.l, x, fmaf(-a.h, x, 1.0f));
    return df_norm(x, x * e);
}

__device__ __forceinline__ DF df_sqrt(DF a)   // a > 0, normal
{
    const float r = sqrt_a(a.h);
    const float e = fmaf(-r, r, a.h) + a.l;
    return df_norm(r, 0.5f * e * rcp_a(r));
}

// atan2(y, x) for y >= 0 (an angle in [0, pi]), for the lens angles of the
// Mandel-Agol terms.  r = min(y, |x|) / max(y, |x|) lies in [0, 1] and
// atan(r) = r P(r^2) with P of degree 8, fitted to atan(r)/r on [0, 1] by
// Lawson's iteratively reweighted least squares (towards the minimax fit;
// csrc/atan_poly.py recomputes the coefficients): 1.4e-8 absolute in FP64,
// about 1.2e-7 evaluated in FP32.  Then atan2 = pi/2 - atan(r) when y > |x|,
// and pi minus that when x < 0.  Both arguments zero give 0.
__device__ __forceinline__ float atan2_pos(float y, float x)
{
    const float ax = fabsf(x);
    const float mx = fmaxf(y, ax), mn = fminf(y, ax);
    const float r = mx > 0.0f ? mn * rcp_a(mx) : 0.0f;   // mx is 0 or a normal number here
    const float s = r * r;
    float q = 2.903584391e-03f;
    q = fmaf(q, s, -1.628314145e-02f);
    q = fmaf(q, s, 4.303959757e-02f);
    q = fmaf(q, s, -7.533697039e-02f);
    q = fmaf(q, s, 1.065468788e-01f);
    q = fmaf(q, s, -1.420713663e-01f);
    q = fmaf(q, s, 1.999305487e-01f);
    q = fmaf(q, s, -3.333309293e-01f);
    q = fmaf(q, s, 1.0f);
    float t = r * q;
    if (y > ax) t = 0.5f * PT_PI_F - t;
    if (x < 0.0f) t = PT_PI_F - t;
    return t;
}

// First pass of the window test, in plain FP32: false only when t - t0 - nP
// is certainly outside [win_lo, win_hi].  One FMA does the reduction with
// the same epoch n as reduce_time; against the double-float result it drops
// the rounding of s, the low parts of t, t0 and P and rounds once more, so
// it is off by less than 2^-24 (|s| + |t_h| + |t0_h| + |n| P_h + |d|); the
// margin doubles that (plus a nanosecond-scale floor).
__device__ __forceinline__ bool maybe_in_window(float th, const GeomRec &r)
{
    float s = th - r.t0h;
    float n = rintf(s * r.invP);
    float d = fmaf(-n, r.Ph, s);
    float m = 1.2e-7f * (fabsf(s) + fabsf(th) + fabsf(r.t0h) + fabsf(n) * r.Ph + fabsf(d)) + 1e-9f;
    return (d + m >= r.win_lo) && (d - m <= r.win_hi);
}

// sin h and cos h by their Taylor series through h^9 and h^10, for the
// small angles of the transit window (|h| <= 0.4: the first omitted terms,
// h^11/11! and h^12/12!, are below 1e-11 relative); other angles take
// sincosf.
__device__ __forceinline__ void sincos_near0(float h, float *s, float *c)
{
    if (fabsf(h) <= 0.4f) {
        const float h2 = h * h;
        float ps = fmaf(h2, 1.0f / 362880.0f, -1.0f / 5040.0f);
        ps = fmaf(h2, ps, 1.0f / 120.0f);
        ps = fmaf(h2, ps, -1.0f / 6.0f);
        *s = fmaf(h * h2, ps, h);
        float pc = fmaf(h2, -1.0f / 3628800.0f, 1.0f / 40320.0f);
        pc = fmaf(h2, pc, -1.0f / 720.0f);
        pc = fmaf(h2, pc, 1.0f / 24.0f);
        pc = fmaf(h2, pc, -0.5f);
        *c = fmaf(h2, pc, 1.0f);
    } else {
        sincosf(h, s, c);
    }
}

// Projected separation z at time offset dt from conjunction (Sec. 1; the
// paper prints no orbit formula).
//   Circular:  phi = 2 pi dt / P,  z = a sqrt(sin^2 phi + cos^2 i cos^2 phi).
//   Eccentric: Kepler's equation is solved relative to the conjunction
//     anchor E_tr (M_tr = E_tr - e sin E_tr):
//       dE - e cos E_tr sin dE + e sin E_tr (1 - cos dE) = dM,  dM = 2 pi dt / P,
//     by Newton's method.  Position in the sky plane relative to conjunction:
//       U = r cos(w + f) = a cos w dC - a sqrt(1-e^2) sin w dS        (U_tr = 0)
//       V = r sin(w + f) = V_tr + a sin w dC + a sqrt(1-e^2) cos w dS
//     with dC = cos E - cos E_tr, dS = sin E - sin E_tr formed from sin dE and
//     1 - cos dE = 2 sin^2(dE/2).  Every term is small near transit, so FP32
//     keeps relative accuracy there; z = sqrt(U^2 + V^2 cos^2 i).
//   Behind the star (cos phi <= 0, or V <= 0) returns PT_ZBEHIND.
// Newton stops once the error left after a step, at most (e / (2 (1 - e)))
// step^2 (|f''| <= e, f' >= 1 - e for this f), is below 3e-8 |dE|: the
// rounding level of the FP32 evaluation, so no step is spent on merely
// confirming convergence.  *bad is set when that did not happen within
// max_iter steps.
// Warm start: a caller stepping through the supersamples of one exposure
// passes warm[4] = {dE, dM, dE/dM, (1/2) d2E/dM2} of the previous solution
// (warm[0] NaN for none); the start is the second-order step, off by
// ~e (dM' - dM)^3 / 6, so one Newton step converges on every lane (after a
// first-order step some lane of most warps took a second).  The solution is
// written back.
// FAST takes the Newton quotient with the one-instruction reciprocal (its
// denominator 1 - e cos E lies in [1 - e, 1 + e]) and the final root with the
// one-instruction square root (an argument below 2^-126, a separation under
// 1e-19, gives 0): about one ulp more in z.  ROT takes sin and cos of dE/2 at the solution
// from the last step's values (below) instead of a second series; the
// supersample loop of the row kernel gains from it, while in the
// batched and tile kernels the extra live values cost more than the series.

// E = M + e sin E puts dE within e of dM - e sin E_tr.  Far from transit at a high
// eccentricity Newton's method, from either start, can leap out of that interval and
// not come back (e = 0.9, exposures of 0.4 d at P = 3 d: 2.6 % of the exposures did
// not converge from the second-order start, none from a first-order one; over
// the whole orbit 14 % from the cold start), so from the fourth step on its iterate is
// brought back into it: then every one converges, in eight steps at most up to e
// = 0.9 and ten at 0.95.  The steps before are free: over a transit there are one
// to three.
constexpr int KEPLER_FREE = 4;

__device__ __forceinline__ float kepler_bracket(float dE, float dM, float esE, float nq)
{
    const float e = 1.0001f * nq * rcp_a(1.0f + nq), c = dM - esE;   // nq = e / (1 - e)
    return fminf(fmaxf(dE, c - e), c + e);
}

template <bool FAST = false, bool ROT = false>
__device__ __forceinline__ float orbit_z(const GeomRec &r, float dt, int max_iter, bool *bad, float *warm = nullptr)
{
    if (r.ecc == 0.0f) {
        float s, c;
        sincos_near0(r.nang * dt, &s, &c);
        if (c <= 0.0f) return PT_ZBEHIND;
        float ci = r.cosi * c;
        return r.a * (FAST ? sqrt_a(fmaf(s, s, ci * ci)) : sqrtf(fmaf(s, s, ci * ci)));
    }
    float dM = r.nang * dt;
    float dE;
    if (warm && warm[0] == warm[0]) {
        const float x = dM - warm[1];
        dE = fmaf(x, fmaf(x, warm[3], warm[2]), warm[0]);
    } else {
        dE = dM / (1.0f - r.ecE);
    }
    float sh = 0.0f, ch = 1.0f, dEdM = 1.0f, step = 0.0f, esin = 0.0f;
    auto newton = [&]() {
        sincos_near0(0.5f * dE, &sh, &ch);
        float sn = 2.0f * sh * ch, omc = 2.0f * sh * sh;
        float F = (dE - r.ecE * sn) + (r.esE * omc - dM);
        float Fp = 1.0f - r.ecE * (1.0f - omc) + r.esE * sn;
        if (warm) esin = fmaf(r.esE, 1.0f - omc, r.ecE * sn);   // e sin E
        if (FAST) {
            dEdM = rcp_a(Fp);
            step = F * dEdM;
        } else {
            step = F / Fp;
            if (warm) dEdM = __fdividef(1.0f, Fp);
        }
        dE -= step;
        return r.nq * step * step <= 6e-8f * fabsf(dE) + 1e-12f;
    };
    // (the bracketed steps in a loop of their own: in one loop their test cost the
    // batch kernel 1 %, so 0.5 %; the other way round in orbit_state and the adjoint)
    bool conv = false;
    int it = 0;
#pragma unroll 1
    for (; it < min(max_iter, KEPLER_FREE) && !conv; ++it) conv = newton();
#pragma unroll 1
    for (; it < max_iter && !conv; ++it) {
        dE = kepler_bracket(dE, dM, r.esE, r.nq);
        conv = newton();
    }
    if (!conv) *bad = true;
    if (warm) {
        warm[0] = dE;
        warm[1] = dM;
        warm[2] = dEdM;
        warm[3] = -0.5f * esin * dEdM * dEdM * dEdM;
    }
    if (ROT) {
        // sin and cos of dE/2 at the solution: the last step's values rotated
        // by -step/2 with cos(step/2) ~ 1 - step^2/8, sin(step/2) ~ step/2.
        // The dropped terms are third order in step/2: the stopping rule
        // accepts |step| <= sqrt(6e-8 |dE| / nq) (< 1e-3 unless e is tiny,
        // where the Newton step itself is at most e |dM|), so they stay
        // below 1e-10.
        const float h = 0.5f * step;
        const float c = fmaf(-0.5f * h, h, 1.0f);
        const float sh1 = fmaf(-ch, h, sh * c);
        ch = fmaf(sh, h, ch * c);
        sh = sh1;
    } else {
        sincos_near0(0.5f * dE, &sh, &ch);
    }
    float sn = 2.0f * sh * ch, omc = 2.0f * sh * sh;
    float dC = -r.cE * omc - r.sE * sn;
    float dS = r.cE * sn - r.sE * omc;
    float U = r.Uc * dC - r.Us * dS;
    float V = r.Vtr + (r.Vs * dC + r.Vc * dS);
    if (V <= 0.0f) return PT_ZBEHIND;
    float Vi = V * r.cosi;
    return FAST ? sqrt_a(fmaf(U, U, Vi * Vi)) : sqrtf(fmaf(U, U, Vi * Vi));
}


// Sky position over one exposure from a single solution of Kepler's equation.
// OrbitState is the position (U, V) and its derivative by the mean anomaly at
// one time; in units of the mean anomaly the motion obeys r'' = -u r with
// u = (a/r)^3, so at an offset x the position is f(x) (U, V) + g(x) (U', V')
// with the f and g series (Bate, Mueller & White 1971, Sec. 5.2, to x^5),
//   f = 1 - u x^2/2 + u p x^3/2 + (3uq - 15up^2 + u^2) x^4/24
//         + (7up^3 - 3upq - u^2 p) x^5/8,
//   g = x - u x^3/6 + u p x^4/4 + (9uq - 45up^2 + u^2) x^5/120,
// p = r'/r, q = v^2/r^2 - u.  With E1 = dE/dM = a/r these are u = E1^3,
// p = e sin E E1^2, q = E1^2 (E1 - 1).  The remainder, in units of a, is below
// (0.02 + 0.4 e^2) (u x^2)^3 (measured in 64 bits over e = 0 .. 0.95 and all
// phases); fg_valid asks for 5e-9 stellar radii, under the rounding of an
// FP32 separation.  A supersample costs about 20 instructions against 100 to
// 170 for a Newton solution (warm-started) and its position.
struct OrbitState {
    float U, V, Up, Vp, E1, esin;
};

__device__ __forceinline__ void orbit_state(const GeomRec &r, float dt, int max_iter, bool *bad, OrbitState *o)
{
    if (r.ecc == 0.0f) {
        float s, c;
        sincos_near0(r.nang * dt, &s, &c);
        o->U = r.a * s;
        o->V = r.a * c;
        o->Up = o->V;
        o->Vp = -o->U;
        o->E1 = 1.0f;
        o->esin = 0.0f;
        return;
    }
    // as in orbit_z
    const float dM = r.nang * dt;
    float dE = dM / (1.0f - r.ecE);
    float sh = 0.0f, ch = 1.0f, step = 0.0f;
    bool conv = false;
    for (int it = 0; it < max_iter; ++it) {
        sincos_near0(0.5f * dE, &sh, &ch);
        const float sn = 2.0f * sh * ch, omc = 2.0f * sh * sh;
        const float F = (dE - r.ecE * sn) + (r.esE * omc - dM);
        const float Fp = 1.0f - r.ecE * (1.0f - omc) + r.esE * sn;
        step = F * rcp_a(Fp);
        dE -= step;
        if (r.nq * step * step <= 6e-8f * fabsf(dE) + 1e-12f) {
            conv = true;
            break;
        }
        if (it + 1 >= KEPLER_FREE) dE = kepler_bracket(dE, dM, r.esE, r.nq);
    }
    if (!conv) *bad = true;
    const float h = 0.5f * step;
    const float c = fmaf(-0.5f * h, h, 1.0f);
    const float sh1 = fmaf(-ch, h, sh * c);
    ch = fmaf(sh, h, ch * c);
    sh = sh1;
    const float sn = 2.0f * sh * ch, omc = 2.0f * sh * sh;
    const float dC = -r.cE * omc - r.sE * sn;
    const float dS = r.cE * sn - r.sE * omc;
    o->U = r.Uc * dC - r.Us * dS;
    o->V = r.Vtr + (r.Vs * dC + r.Vc * dS);
    o->esin = fmaf(r.esE, 1.0f - omc, r.ecE * sn);
    o->E1 = rcp_a(1.0f - r.ecE * (1.0f - omc) + r.esE * sn);   // 1 - e cos E, in [1 - e, 1 + e]
    const float cE = r.cE + dC, sE = r.sE + dS;
    o->Up = -(r.Uc * sE + r.Us * cE) * o->E1;
    o->Vp = (r.Vc * cE - r.Vs * sE) * o->E1;
}

// Are the series good enough for offsets up to x?
__device__ __forceinline__ bool fg_valid(const GeomRec &r, float E1, float x)
{
    const float e = r.ecc == 0.0f ? 0.0f : r.nq * rcp_a(1.0f + r.nq);   // nq = e / (1 - e)
    const float s = E1 * E1 * E1 * x * x;
    return r.a * fmaf(0.4f * e, e, 0.02f) * s * s * s <= 5e-9f;
}

struct FgSeries {
    float f2, f3, f4, f5, g3, g4, g5;
};

__device__ __forceinline__ FgSeries fg_series(float E1, float esin)
{
    FgSeries c;
    const float u = E1 * E1 * E1, p = esin * E1 * E1, q = E1 * E1 * (E1 - 1.0f), pp = p * p;
    c.f2 = -0.5f * u;
    c.f3 = 0.5f * u * p;
    c.f4 = u * (3.0f * q - 15.0f * pp + u) * (1.0f / 24.0f);
    c.f5 = u * p * (7.0f * pp - 3.0f * q - u) * 0.125f;
    c.g3 = -u * (1.0f / 6.0f);
    c.g4 = 0.25f * u * p;
    c.g5 = u * (9.0f * q - 45.0f * pp + u) * (1.0f / 120.0f);
    return c;
}

// separation at offset x
__device__ __forceinline__ float fg_z(const OrbitState &o, const FgSeries &c, float cosi, float x)
{
    const float x2 = x * x;
    const float f1 = fmaf(fmaf(fmaf(c.f5, x, c.f4), x, c.f3), x, c.f2) * x2;   // f - 1
    const float g = fmaf(fmaf(fmaf(c.g5, x, c.g4), x, c.g3), x2 * x, x);
    const float U = o.U + fmaf(f1, o.U, g * o.Up), V = o.V + fmaf(f1, o.V, g * o.Vp);
    const float Vi = V * cosi;
    return V > 0.0f ? sqrt_a(fmaf(U, U, Vi * Vi)) : PT_ZBEHIND;
}

// ---------------------------------------------------------------------------
// Bulirsch's general complete elliptic integral (Bulirsch 1969, Numer. Math.
// 13, 305),
//   cel(kc, p, a, b) = int_0^{pi/2} (a cos^2 + b sin^2) /
//                      ((cos^2 + p sin^2) sqrt(cos^2 + kc^2 sin^2)) dth,
// evaluated for two (p, a, b) triples that share kc: the Gauss/Landen
// sequence of (kc, m) does not depend on (p, a, b), so the two integrals
// share its square roots.  The first triple has p = 1 (the K/E combination
// a K + (b - a) ... is folded into (a, b) by the caller), the second has
// p = rho > 0 and b = 0.  Converged when the arithmetic-geometric means agree
// to 3e-4 (quadratic convergence then leaves ~1e-7); at most 10 steps.
// The two integrals' updates run as the two lanes of fma/mul/add.rn.f32x2
// (one instruction for both; each lane rounded as the scalar operation).
// ---------------------------------------------------------------------------
// two-lane FP32 helpers (sm_100 and later); each lane is one IEEE operation
// rounded once, the same result as the scalar instruction
__device__ __forceinline__ unsigned long long f2_pack(float lo, float hi)
{
    return ((unsigned long long)__float_as_uint(hi) << 32) | __float_as_uint(lo);
}
__device__ __forceinline__ float f2_lo(unsigned long long v) { return __uint_as_float((unsigned)v); }
__device__ __forceinline__ float f2_hi(unsigned long long v) { return __uint_as_float((unsigned)(v >> 32)); }
__device__ __forceinline__ unsigned long long f2_fma(unsigned long long a, unsigned long long b, unsigned long long c)
{
    unsigned long long d;
    asm("fma.rn.f32x2 %0, %1, %2, %3;" : "=l"(d) : "l"(a), "l"(b), "l"(c));
    return d;
}
__device__ __forceinline__ unsigned long long f2_mul(unsigned long long a, unsigned long long b)
{
    unsigned long long d;
    asm("mul.rn.f32x2 %0, %1, %2;" : "=l"(d) : "l"(a), "l"(b));
    return d;
}
__device__ __forceinline__ unsigned long long f2_add(unsigned long long a, unsigned long long b)
{
    unsigned long long d;
    asm("add.rn.f32x2 %0, %1, %2;" : "=l"(d) : "l"(a), "l"(b));
    return d;
}

template <bool IEEE = false>
__device__ __forceinline__ void cel2(float kc, float a1, float b1, float srho, float a2, float *r1,
                                     float *r2)
{
    // lanes: (first integral, second integral); srho = sqrt(rho).  The lanes'
    // p start at 1 and sqrt(rho) >= 1 and only grow, kc in (0, 1] and e = kc m
    // stay normal numbers, so the .ftz approximations never meet a denormal.
    unsigned long long A = f2_pack(a1, a2), B = f2_pack(b1, 0.0f), P = f2_pack(1.0f, srho);
    float m = 1.0f, e = kc;
#pragma unroll 1
    for (int it = 0; it < 10; ++it) {
        const unsigned long long ip = f2_pack(rcp_t<IEEE>(f2_lo(P)), rcp_t<IEEE>(f2_hi(P)));
        const unsigned long long F = A;
        A = f2_fma(B, ip, A);
        const unsigned long long G = f2_mul(f2_pack(e, e), ip);
        B = f2_fma(F, G, B);
        B = f2_add(B, B);
        P = f2_add(P, G);
        float g = m;
        m = kc + m;
        if (fabsf(g - kc) <= g * 3e-4f) break;
        kc = 2.0f * sqrt_t<IEEE>(e);
        e = kc * m;
    }
    *r1 = (0.5f * PT_PI_F) * fmaf(f2_lo(A), m, f2_lo(B)) * rcp_t<IEEE>(m * (m + f2_lo(P)));
    *r2 = (0.5f * PT_PI_F) * fmaf(f2_hi(A), m, f2_hi(B)) * rcp_t<IEEE>(m * (m + f2_hi(P)));
}

// cel2's loop carrying K = cel(kc, 1, 1, 1) and E = cel(kc, 1, 1, kc^2) in place
// of one combination of them (cel with p = 1 is linear in (a, b), so
// cel(kc, 1, cK + cE, cK + cE kc^2) = cK K + cE E), for callers that also need
// K and E themselves.
__device__ __forceinline__ void cel3(float kc, float srho, float a2, float *K, float *E, float *r2)
{
    float p1 = 1.0f;
    float p2 = srho;   // argument ranges as in cel2
    float aK = 1.0f, bK = 1.0f, aE = 1.0f, bE = kc * kc, b2 = 0.0f;
    float m = 1.0f, e = kc;
#pragma unroll 1
    for (int it = 0; it < 10; ++it) {
        float ip1 = rcp_a(p1);
        float ip2 = rcp_a(p2);
        float g = e * ip1;
        float f = aK;
        aK = fmaf(bK, ip1, aK);
        bK = 2.0f * fmaf(f, g, bK);
        f = aE;
        aE = fmaf(bE, ip1, aE);
        bE = 2.0f * fmaf(f, g, bE);
        p1 += g;
        f = a2;
        a2 = fmaf(b2, ip2, a2);
        g = e * ip2;
        b2 = 2.0f * fmaf(f, g, b2);
        p2 += g;
        g = m;
        m = kc + m;
        if (fabsf(g - kc) <= g * 3e-4f) break;
        kc = 2.0f * sqrt_a(e);
        e = kc * m;
    }
    const float den = (0.5f * PT_PI_F) * rcp_a(m * (m + p1));
    *K = fmaf(aK, m, bK) * den;
    *E = fmaf(aE, m, bE) * den;
    *r2 = (0.5f * PT_PI_F) * fmaf(a2, m, b2) * rcp_a(m * (m + p2));
}

// ---------------------------------------------------------------------------
// Mandel & Agol (2002) terms for the quadratic law, FP32.
//   le = lambda_e, ld = lambda_d + 2/3 Theta(p - z), ed = eta_d.
//
// Geometry: d = z + p - 1, 1 - a = (1 - z + p)(1 + z - p), b - 1 = d (1 + z + p),
// q = (p - z)(p + z); all formed from single differences so they keep
// relative precision at the contact points.  kap0, kap1 and the triangle
// area come from atan2 of the Heron area (no acos of a rounded cosine).
//
// lambda_1 (partial) and lambda_2 (inside) are Mandel & Agol's
//   pref {cK K(k) + cE E(k) + cP Pi(n, k)}.
// Near z = 1 - p the modulus tends to 1 and K, Pi diverge logarithmically
// while their divergences cancel.  The kernel removes the cancellation
// algebraically:  with rho = 1 - n,
//   cP Pi = (cP/rho) K + cP (rho - 1)/rho * cel(kc, rho, 1, 0),
// and cK' = cK + cP/rho factors through b - 1:
//   lambda_1: cK' = -(b-1)(6 p^2 + 2 p z - 3),              cR = -3 q (1-a)/a
//   lambda_2: cK' = (b-1)(p^3 - p^2 z - p z^2 + 2p + z^3 - 4z)/(p+z),
//             cR = -12 q z p / (a b)
// so the brace is cel(kc, 1, cK'+cE, cK'+cE kc^2) + cel(kc, rho, cR, 0), two
// bounded integrals evaluated in one shared loop (cel2).  With a = (z-p)^2,
// b = (z+p)^2 and q = -(z-p)(z+p) these reduce exactly to
//   lambda_1: sqrt(rho) = 1/|z-p|,        cR = 3 (z+p)(1-a)/(z-p),
//   lambda_2: sqrt(rho) = (z+p)/|z-p|,    cR = 12 z p / ((z-p)(z+p)),
// which the kernel evaluates (fewer roundings; z = p is a separate case).
// Reciprocals and square roots are the one-instruction approximations.  For
// p >= 1e-15 every argument they get is a normal number or zero: d and z - p
// are 0 (separate cases) or at least an ulp of p, z or 1, and the products
// formed from them stay far above 2^-126.
// Exact special cases of Mandel & Agol's Table 1 that the general formulas
// cannot evaluate (z = 1 - p, z = p, p = z = 1/2, star covered) are taken
// separately; near them the general formulas stay accurate in FP32.
// ---------------------------------------------------------------------------
// With KE, K and E of the general cases' modulus (cases 2, 3, 8, 9: the
// partial and inside overlaps) come back too, *have_ke = true; other cases
// leave *have_ke false.
// ma_terms_core takes d = z + p - 1 and e1 = 1 - z + p beside p and z, for
// callers that know the distances to the contacts better than the rounded z
// does (the nodes of the row tables below); it is for points in transit
// (e1 > 0, p > 0) that do not cover the star.
template <bool KE = false, bool IEEE = false>
__device__ __forceinline__ void ma_terms_core(float p, float z, float d, float e1, float *le, float *ld, float *ed,
                                              float *Kout = nullptr, float *Eout = nullptr, bool *have_ke = nullptr)
{
    const float pi = PT_PI_F;
    float p2 = p * p, z2 = z * z;
    float oma = e1 * (1.0f + z - p);
    float bm1 = d * (1.0f + z + p);
    float zmp = z - p;
    float eta2 = 0.5f * p2 * (p2 + 2.0f * z2);
    bool inside = d < 0.0f;

    // lens geometry: only the partial (and contact) cases need it
    float le_part = p2, eta1 = eta2;
    if (!inside) {
        float fa = sqrt_t<IEEE>(oma * bm1);                    // 4 x triangle area (oma, bm1 >= 0)
        float k1 = atan2_pos(fa, 1.0f - p2 + z2);
        float k0 = atan2_pos(fa, p2 + z2 - 1.0f);
        le_part = (p2 * k0 + k1 - 0.5f * fa) * (1.0f / pi);
        eta1 = (k1 + 2.0f * eta2 * k0 - 0.25f * (1.0f + 5.0f * p2 + z2) * fa) * (0.5f / pi);
    }

    // parameters of the shared elliptic evaluation
    float kc, cKp, cE, srho = 1.0f, cR = 0.0f, pref, cst = 0.0f;
    bool need_cel = true;
    float e_out = inside ? eta2 : eta1;
    if (d == 0.0f) {                                 // case 4: lambda_5, z = 1 - p
        cst = 2.0f / (3.0f * pi) * acosf(1.0f - 2.0f * p) -
              4.0f / (9.0f * pi) * (3.0f + 2.0f * p - 8.0f * p2) * sqrtf(p * (1.0f - p)) -
              (p > 0.5f ? 2.0f / 3.0f : 0.0f);
        e_out = eta2;
        need_cel = false;
        kc = 1.0f; cKp = 0.0f; cE = 0.0f; pref = 0.0f;
    } else if (zmp == 0.0f) {                        // z = p
        if (p == 0.5f) {                             // case 6
            cst = 1.0f / 3.0f - 4.0f / (9.0f * pi);
            e_out = 3.0f / 32.0f;
            need_cel = false;
            kc = 1.0f; cKp = 0.0f; cE = 0.0f; pref = 0.0f;
        } else if (p < 0.5f) {                       // case 5: lambda_4, modulus 2p
            kc = sqrtf((1.0f - 2.0f * p) * (1.0f + 2.0f * p));
            cKp = 1.0f - 4.0f * p2;
            cE = 4.0f * (2.0f * p2 - 1.0f);
            pref = 2.0f / (9.0f * pi);
            cst = 1.0f / 3.0f;
            e_out = eta2;
        } else {                                     // case 7: lambda_3, modulus 1/(2p)
            kc = sqrtf((2.0f * p - 1.0f) * (2.0f * p + 1.0f)) / (2.0f * p);
            cKp = -(1.0f - 4.0f * p2) * (3.0f - 8.0f * p2) / p;
            cE = 16.0f * p * (2.0f * p2 - 1.0f);
            pref = 1.0f / (9.0f * pi);
            cst = 1.0f / 3.0f;
            e_out = eta1;
        }
    } else if (inside) {                             // cases 3, 9: lambda_2
        kc = sqrt_t<IEEE>(-bm1 * rcp_t<IEEE>(oma));
        cKp = bm1 * (p2 * p - p2 * z - p * z2 + 2.0f * p + z2 * z - 4.0f * z) * rcp_t<IEEE>(p + z);
        cE = oma * (z2 + 7.0f * p2 - 4.0f);
        srho = (p + z) * rcp_t<IEEE>(fabsf(zmp));
        cR = (12.0f * z * p) * rcp_t<IEEE>(zmp * (z + p));
        pref = 2.0f * rcp_t<IEEE>(9.0f * pi * sqrt_t<IEEE>(oma));
    } else {                                         // cases 2, 8: lambda_1
        kc = sqrt_t<IEEE>(bm1 * rcp_t<IEEE>(4.0f * z * p));
        cKp = -bm1 * (6.0f * p2 + 2.0f * p * z - 3.0f);
        cE = 4.0f * p * z * (z2 + 7.0f * p2 - 4.0f);
        srho = rcp_t<IEEE>(fabsf(zmp));
        cR = (3.0f * (p + z) * oma) * rcp_t<IEEE>(zmp);
        pref = rcp_t<IEEE>(9.0f * pi * sqrt_t<IEEE>(p * z));
    }
    float lam = cst;
    if (need_cel) {
        float r1, r2;
        if (KE && d != 0.0f && zmp != 0.0f) {
            float K, E;
            cel3(kc, srho, cR, &K, &E, &r2);
            r1 = fmaf(cKp, K, cE * E);
            *Kout = K;
            *Eout = E;
            *have_ke = true;
        } else {
            cel2<IEEE>(kc, cKp + cE, fmaf(cE, kc * kc, cKp), srho, cR, &r1, &r2);
        }
        lam = fmaf(pref, r1 + r2, cst);
    }
    if (p > z) lam += 2.0f / 3.0f;
    *le = inside ? p2 : le_part;
    *ld = lam;
    *ed = e_out;
}

template <bool KE = false>
__device__ __forceinline__ void ma_terms(float p, float z, float *le, float *ld, float *ed, float *Kout = nullptr,
                                         float *Eout = nullptr, bool *have_ke = nullptr)
{
    if (KE) *have_ke = false;
    *le = 0.0f;
    *ld = 0.0f;
    *ed = 0.0f;
    if (!(z < 1.0f + p) || !(p > 0.0f)) return;    // out of transit (also PT_ZBEHIND, NaN)
    if (p >= 1.0f && z <= p - 1.0f) {               // case 11: star covered
        *le = 1.0f;
        *ld = 2.0f / 3.0f;
        *ed = 0.5f;
        return;
    }
    ma_terms_core<KE>(p, z, (z - 1.0f) + p, 1.0f - z + p, le, ld, ed, Kout, Eout, have_ke);
}

// ---------------------------------------------------------------------------
// Row tables: a Mandel-Agol quantity of one radius ratio p as a function of z,
// as piecewise polynomials good to the rounding of the FP32 terms themselves.
//
// Where a kernel evaluates one radius ratio at thousands of separations, the
// elliptic integrals need not be summed for each of them: between the
// contacts z = 1 - p and z = 1 + p the terms are analytic in z, and at the
// contacts they are analytic in the square root of the distance up to
// w^4 log w terms.  So with
//   region A, planet inside the disk:  w^2 = (1 - p) - z,
//   region B, limb, z < 1:             w^2 = z - (1 - p),
//   region C, limb, z >= 1:            w^2 = (1 + p) - z,
// and MT_NA, MT_NL, MT_NL equal intervals in w, a degree-5 polynomial per
// interval is within 1e-9 of the terms (measured in 64 bits over p = 0.001 ..
// 0.5: 4e-10 at p = 0.05, 7e-10 at 0.3, 8e-10 at 0.5), below the ~1e-8 to
// 1e-7 of the FP32 evaluation.  A table is 144 evaluations of the exact terms
// at Chebyshev nodes; a look-up is about 22 instructions against 170 (inside)
// to 230 (limb) of the terms.
// With u = w s, interval i covers u in [i - 1/2, i + 1/2] (the first of a
// region only its upper half), t = u - i, so one FMA with a large constant
// rounds to the interval and one more gives t.  The scales s keep u below the
// region's last interval's end by 2e-6, more than the rounding of w.
// Radius ratios outside [MT_PMIN, MT_PMAX] (where another contact's
// singularity comes within an interval's width) take the exact terms.
// Layout of a row: 8 floats per interval, c0..c5 and two unused, so that one
// address serves a 16-byte and an 8-byte load.  c0 of
// region C's first interval is set to 0, so a separation at or beyond 1 + p
// reads exactly 0.
// ---------------------------------------------------------------------------
constexpr int MT_NA = 8, MT_NL = 8, MT_N = MT_NA + 2 * MT_NL, MT_Q = 6, MT_NODES = MT_N * MT_Q;
constexpr int MT_ROW = 8 * MT_N;                    // floats per row
constexpr float MT_PMIN = 1e-6f, MT_PMAX = 0.5f;
constexpr float MT_MAGIC = 12582912.0f;             // 1.5 2^23: adding it rounds to an integer

// values at the interval's Chebyshev nodes -> monomial coefficients in t, for
// a region's first interval (nodes t = (1 + x) / 4) and the others (t = x / 2)
struct MtMat {
    float m[2][MT_Q][MT_Q];   // [first ? 0 : 1][coefficient][node]
};
constexpr MtMat make_mt()
{
    const double x[MT_Q] = {0.96592582628906828675, 0.70710678118654752440,  0.25881904510252076235,
                            -0.25881904510252076235, -0.70710678118654752440, -0.96592582628906828675};
    MtMat r{};
    for (int kind = 0; kind < 2; ++kind) {
        // T_k(y), y = al t + be, as polynomials in t
        const double al = kind == 0 ? 4.0 : 2.0, be = kind == 0 ? -1.0 : 0.0;
        double T[MT_Q][MT_Q] = {};
        T[0][0] = 1.0;
        T[1][0] = be;
        T[1][1] = al;
        for (int k = 2; k < MT_Q; ++k)
            for (int c = 0; c < MT_Q; ++c)
                T[k][c] = 2.0 * be * T[k - 1][c] + (c > 0 ? 2.0 * al * T[k - 1][c - 1] : 0.0) - T[k - 2][c];
        for (int q = 0; q < MT_Q; ++q) {
            double tk[MT_Q] = {1.0, x[q]};
            for (int k = 2; k < MT_Q; ++k) tk[k] = 2.0 * x[q] * tk[k - 1] - tk[k - 2];
            for (int c = 0; c < MT_Q; ++c) {
                double v = 0.0;
                for (int k = 0; k < MT_Q; ++k) v += (k == 0 ? 1.0 : 2.0) / MT_Q * tk[k] * T[k][c];
                r.m[kind][c][q] = (float)v;
            }
        }
    }
    return r;
}
static __constant__ MtMat c_mt = make_mt();

__device__ __forceinline__ bool mt_valid(float p) { return p >= MT_PMIN && p <= MT_PMAX; }

// scales of regions A and B, C
__device__ __forceinline__ void mt_scales(float p, float *sA, float *sL)
{
    *sA = ((float)MT_NA - 0.5f) * (1.0f - 2e-6f) / sqrtf(1.0f - p);
    *sL = ((float)MT_NL - 0.5f) * (1.0f - 2e-6f) / sqrtf(p);
}

// Coefficient c of interval i from the interval's node values f.  The rows of
// the matrix alternate in sign and reach 10^3, so they are applied to the
// differences from one node (the constant goes to c0 alone): applied to the
// values, their FP32 rounding would show (3e-6 at p = 0.5).
__device__ __forceinline__ float mt_coef(int i, int c, const float *f)
{
    const int kind = (i == 0 || i == MT_NA || i == MT_NA + MT_NL) ? 0 : 1;   // a region's first interval
    float a = 0.0f;
#pragma unroll
    for (int q = 0; q < MT_Q; ++q) a = fmaf(c_mt.m[kind][c][q], f[q] - f[2], a);
    if (c != 0) return a;
    return i == MT_NA + MT_NL ? 0.0f : a + f[2];
}

// lambda_2 + 2/3 Theta(p - z) with the planet wholly inside the disk, at
// z = 1 - p - w^2, in double-float arithmetic.  The brace's two integrals are
// of order one and cancel to the order of p^2: in FP32 that leaves 2e-8 to
// 4e-8, which averages out over the rounding of many separations but would be
// frozen into the rows of a table.  Formulas as in ma_terms_core (cases 3, 9)
// with a = (z - p)^2 and the distances as polynomials in p and w^2.
__device__ __forceinline__ float mt_lambda_inside(float p, float w)
{
    const float w2h = w * w;
    const DF W = DF{w2h, fmaf(w, w, -w2h)};                 // w^2
    const DF one = DF{1.0f, 0.0f}, P = DF{p, 0.0f};
    const DF zpp = df_add(one, df_neg(W));                  // z + p = 1 - w^2
    const DF z = df_add(zpp, DF{-p, 0.0f});
    const DF zmp = df_add(z, DF{-p, 0.0f});
    const DF oma = df_mul(df_add(DF{2.0f * p, 0.0f}, W), df_add(one, zmp));   // (1 - z + p)(1 + z - p)
    const DF bm1 = df_neg(df_mul(W, df_add(one, zpp)));     // (z + p - 1)(z + p + 1)
    const DF izpp = df_rcp(zpp), izmp = df_rcp(zmp), ioma = df_rcp(oma);
    const DF kc2 = df_neg(df_mul(bm1, ioma));
    DF kc = df_sqrt(kc2);
    // cK' = (b - 1) (a + (2p - 4z)/(z + p)), cE = (1 - a)(z^2 + 7 p^2 - 4)
    const DF cK = df_mul(bm1, df_mad(df_add(DF{2.0f * p, 0.0f}, df_scale(-4.0f, z)), izpp, df_mul(zmp, zmp)));
    const DF p2 = df_mul(P, P);
    const DF cE = df_mul(oma, df_add(df_mad(z, z, df_mul(DF{7.0f, 0.0f}, p2)), DF{-4.0f, 0.0f}));
    const float sg = zmp.h < 0.0f ? -1.0f : 1.0f;
    DF A1 = df_add(cK, cE), B1 = df_mad(cE, kc2, cK), P1 = one;
    DF A2 = df_mul(df_mul(DF{12.0f, 0.0f}, df_mul(z, P)), df_mul(izmp, izpp)), B2 = DF{0.0f, 0.0f};
    DF P2 = df_mul(zpp, df_scale(sg, izmp));
    DF m = one, e = kc;
#pragma unroll 1
    for (int it = 0; it < 10; ++it) {
        DF ip = df_rcp(P1);
        DF f = A1, g = df_mul(e, ip);
        A1 = df_mad(B1, ip, A1);
        B1 = df_scale(2.0f, df_mad(f, g, B1));
        P1 = df_add(P1, g);
        ip = df_rcp(P2);
        f = A2;
        g = df_mul(e, ip);
        A2 = df_mad(B2, ip, A2);
        B2 = df_scale(2.0f, df_mad(f, g, B2));
        P2 = df_add(P2, g);
        const float mh = m.h;
        m = df_add(kc, m);
        if (fabsf(mh - kc.h) <= mh * 1e-4f) break;   // quadratic convergence leaves ~1e-9
        kc = df_scale(2.0f, df_sqrt(e));
        e = df_mul(kc, m);
    }
    const DF r1 = df_mul(df_mad(A1, m, B1), df_rcp(df_mul(m, df_add(m, P1))));
    const DF r2 = df_mul(df_mad(A2, m, B2), df_rcp(df_mul(m, df_add(m, P2))));
    // pref (pi/2) = 1 / (9 sqrt(1 - a))
    const DF lam = df_mul(df_add(r1, r2), df_rcp(df_mul(DF{9.0f, 0.0f}, df_sqrt(oma))));
    return zmp.h < 0.0f ? df_add(lam, DF{0.666666687f, -1.98682151e-08f}).h : lam.h;
}

// Node q of interval i: its offset t, the separation and the distances
// d = z - (1 - p) and e1 = (1 + p) - z, formed from w; returns w.
__device__ __forceinline__ float mt_node_at(float p, int i, int q, float *z, float *d, float *e1, float *t)
{
    const int q3 = q < 3 ? q : 5 - q;
    const float xa = q3 == 0 ? 0.96592582629f : (q3 == 1 ? 0.70710678119f : 0.25881904510f);
    const float x = q < 3 ? xa : -xa;
    float sA, sL;
    mt_scales(p, &sA, &sL);
    const int reg = i < MT_NA ? 0 : (i < MT_NA + MT_NL ? 1 : 2);
    const int il = i - (reg == 0 ? 0 : (reg == 1 ? MT_NA : MT_NA + MT_NL));
    *t = il == 0 ? 0.25f * (1.0f + x) : 0.5f * x;
    const float u = il == 0 ? 0.25f * (1.0f + x) : (float)il + 0.5f * x;
    const float w = u / (reg == 0 ? sA : sL);
    const float w2 = w * w;
    *d = reg == 0 ? -w2 : (reg == 1 ? w2 : 2.0f * p - w2);
    *e1 = reg == 0 ? 2.0f * p + w2 : (reg == 1 ? 2.0f * p - w2 : w2);
    *z = reg == 2 ? (1.0f + p) - w2 : (1.0f - p) + *d;
    return w;
}

// The exact terms at that node, with the distances to the contacts formed
// from w (not from the rounded z).
__device__ __forceinline__ void mt_node(float p, int i, int q, float *le, float *ld, float *ed)
{
    float z, d, e1, t;
    const float w = mt_node_at(p, i, q, &z, &d, &e1, &t);
    // (z = p, where the second integral's parameters are infinite, keeps the FP32 terms and their separate case)
    if (i < MT_NA && fabsf(z - p) > 1e-5f) {
        const float p2 = p * p;
        *le = p2;
        *ed = 0.5f * p2 * (p2 + 2.0f * z * z);
        *ld = mt_lambda_inside(p, w);
    } else {
        ma_terms_core<false, true>(p, z, d, e1, le, ld, ed);
    }
}

// Interval and offset of separation z.  zm1 = z - 1; off_limb is the constant
// of region B (z < 1) or C (z >= 1, or NaN), which depends on z alone.
// |z - (1 - p)| and (1 + p) - z: the smaller one is w^2 in every region
// (p <= 1/2).  z >= 1 + p gives w = 0 of region C, where the polynomial is 0.
__device__ __forceinline__ float mt_off_limb(float zm1)
{
    return zm1 < 0.0f ? MT_MAGIC + (float)MT_NA : MT_MAGIC + (float)(MT_NA + MT_NL);
}

// The bits of the rounded w s: MT_BITS0 plus the interval.  (1 + p) - z
// saturated to [0, 1] costs nothing; where it saturates at 1, |z - (1 - p)| is
// below 1 and the smaller.
constexpr unsigned MT_BITS0 = 0x4B400000u;

__device__ __forceinline__ unsigned mt_find(float p, float sA, float sL, float zm1, float off_limb, float *t)
{
    const float d = zm1 + p;
    const float w = sqrt_a(fminf(fabsf(d), __saturatef(p - zm1)));
    const bool in_a = d < 0.0f;
    const float s = in_a ? sA : sL;
    const float off = in_a ? MT_MAGIC : off_limb;
    const float b = fmaf(w, s, off);
    *t = fmaf(w, s, off - b);
    return __float_as_uint(b);
}

// The polynomial of the row at shared-memory address row (bytes) - 32 MT_BITS0
// (mt_base of the row): the interval's bits, shifted, are added as they are.
__device__ __forceinline__ unsigned mt_base(const float *row)
{
    return (unsigned)__cvta_generic_to_shared(row) - 32u * MT_BITS0;
}

__device__ __forceinline__ float mt_eval(unsigned base, unsigned bits, float t)
{
    const unsigned at = base + 32u * bits;
    float4 c;
    float2 g;
    asm volatile("ld.shared.v4.f32 {%0, %1, %2, %3}, [%4];" : "=f"(c.x), "=f"(c.y), "=f"(c.z), "=f"(c.w) : "r"(at));
    asm volatile("ld.shared.v2.f32 {%0, %1}, [%2];" : "=f"(g.x), "=f"(g.y) : "r"(at + 16u));
    return fmaf(fmaf(fmaf(fmaf(fmaf(g.y, t, g.x), t, c.w), t, c.z), t, c.y), t, c.x);
}

// Bilinear interpolation of the tabulated Mandel-Agol terms (Sec. 2.2.3):
// node (i, j) holds the terms at k_i = k_lo + i dk, z_j = j dz with
// dz = (1 + k_hi) / (n_z - 1).  Out of transit (z >= 1 + k, also the
// behind-the-star sentinel and NaN) the terms are zero; k is clamped to the
// table's range.
__device__ __forceinline__ void ma_interp(const float4 *tab, int n_k, int n_z, float k_lo, float k_hi,
                                          float inv_dk, float inv_dz, float k, float z, float *le, float *ld,
                                          float *ed)
{
    *le = 0.0f;
    *ld = 0.0f;
    *ed = 0.0f;
    if (!(z < 1.0f + k)) return;
    float fk = (fminf(fmaxf(k, k_lo), k_hi) - k_lo) * inv_dk;
    int ik = min((int)fk, n_k - 2);
    float wk = fk - (float)ik;
    float fz = fminf(fmaxf(z, 0.0f) * inv_dz, (float)(n_z - 1));
    int iz = min((int)fz, n_z - 2);
    float wz = fz - (float)iz;
    const float4 *r0 = tab + (size_t)ik * n_z + iz;
    const float4 *r1 = r0 + n_z;
    float4 a = __ldg(r0), b = __ldg(r0 + 1), c = __ldg(r1), d = __ldg(r1 + 1);
    float a0 = fmaf(wz, b.x - a.x, a.x), a1 = fmaf(wz, b.y - a.y, a.y), a2 = fmaf(wz, b.z - a.z, a.z);
    float c0 = fmaf(wz, d.x - c.x, c.x), c1 = fmaf(wz, d.y - c.y, c.y), c2 = fmaf(wz, d.z - c.z, c.z);
    *le = fmaf(wk, c0 - a0, a0);
    *ld = fmaf(wk, c1 - a1, a1);
    *ed = fmaf(wk, c2 - a2, a2);
}

// Network coordinate across the ingress/egress band: theta = acos(1 - 2 s)
// mapped to [-1, 1].  Near both contacts (s -> 0, s -> 1) the MA terms
// behave like powers of sqrt(s) and sqrt(1 - s); in theta they are regular.
__device__ __forceinline__ float band_coord(float s)
{
    return acosf(fminf(1.0f, fmaxf(-1.0f, 1.0f - 2.0f * s))) * (2.0f / PT_PI_F) - 1.0f;
}

// lambda_e alone (the lens area over pi), for callers that take lambda_d and
// eta_d from elsewhere: the same geometry as ma_terms.
__device__ __forceinline__ float lens_le(float p, float z)
{
    if (!(z < 1.0f + p) || !(p > 0.0f)) return 0.0f;
    if (p >= 1.0f && z <= p - 1.0f) return 1.0f;
    float d = (z - 1.0f) + p;
    if (d <= 0.0f) return p * p;
    float p2 = p * p, z2 = z * z;
    float oma = (1.0f - z + p) * (1.0f + z - p);
    float fa = sqrtf(fmaxf(0.0f, oma * d * (1.0f + z + p)));
    float k1 = atan2f(fa, 1.0f - p2 + z2);
    float k0 = atan2f(fa, p2 + z2 - 1.0f);
    return (p2 * k0 + k1 - 0.5f * fa) * (1.0f / PT_PI_F);
}

// Quadratic-law weights of Eq. (ma_model): f = 1 - (we le + wd ld + wn ed),
// with c = u1 + 2 u2 and the normalisation 1 - u1/3 - u2/6.
__device__ __forceinline__ void ma_weights(float u1, float u2, float *we, float *wd, float *wn)
{
    float inv = 1.0f / (1.0f - u1 * (1.0f / 3.0f) - u2 * (1.0f / 6.0f));
    float c = u1 + 2.0f * u2;
    *we = (1.0f - c) * inv;
    *wd = c * inv;
    *wn = u2 * inv;
}

constexpr double PT_PI_D = 3.14159265358979323846;

__device__ __forceinline__ float wrap_pos(float x)   // into [0, 2 pi); closed form, no loop
{
    const float tp = 6.28318530717958f;
    float y = x - tp * floorf(x / tp);
    return (y >= tp) ? 0.0f : y;
}

__device__ __forceinline__ float wrap_neg(float x)   // into (-2 pi, 0]
{
    const float tp = 6.28318530717958f;
    float y = wrap_pos(x);
    return (y > 0.0f) ? y - tp : 0.0f;
}

// Per-geometry record (see GeomRec): double-float t0/P, the conjunction
// anchor of an eccentric orbit (FP64 here; it enters the hot path only as
// coefficients of small terms), sky-plane position coefficients, and a
// conservative transit window in time for radius ratio k, widened by half
// an exposure.
__device__ __forceinline__ void make_geom_rec(double t0, double P, float a_f, float inc, bool ecc, float e_f,
                                              float w_f, float k, float half_exp, GeomRec *out)
{
    GeomRec r;
    r.t0h = (float)t0;
    r.t0l = (float)(t0 - (double)r.t0h);
    r.Ph = (float)P;
    r.Pl = (float)(P - (double)r.Ph);
    r.invP = (float)(1.0 / P);
    r.nang = (float)(2.0 * PT_PI_D / P);
    double a = a_f;
    double ci = cos((double)inc);
    r.a = (float)a;
    r.cosi = (float)ci;
    r.k = k;
    double e = 0.0, w = 0.5 * PT_PI_D;
    if (ecc) {
        e = e_f;
        w = w_f;
    }
    r.ecc = ecc ? 1.0f : 0.0f;
    // conjunction anchor: f_tr = pi/2 - w, E_tr from tan(E/2) = sqrt((1-e)/(1+e)) tan(f/2).
    // FP32 suffices: the anchor's sine and cosine only scale the small
    // differential terms of orbit_z (relative error ~1e-7 there), and the
    // sky position at conjunction is zero by construction, not computed.
    // A circular orbit uses none of it (orbit_z, orbit_state).
    double ftr = 0.0, Etr = 0.0, sE = 0.0;
    r.ecE = r.esE = r.sE = r.Uc = r.Us = r.Vs = r.Vc = r.Vtr = 0.0f;
    r.cE = 1.0f;
    if (ecc) {
        float ef = (float)e, wf = (float)w;
        float ftrf = 0.5f * PT_PI_F - wf;
        float Etrf = 2.0f * atan2f(sqrtf(1.0f - ef) * sinf(0.5f * ftrf), sqrtf(1.0f + ef) * cosf(0.5f * ftrf));
        float sEf, cEf, swf, cwf;
        sincosf(Etrf, &sEf, &cEf);
        sincosf(wf, &swf, &cwf);
        float sef = sqrtf((1.0f - ef) * (1.0f + ef)), af = (float)a;
        ftr = 0.5 * PT_PI_D - w;
        Etr = Etrf;
        sE = sEf;
        r.ecE = ef * cEf;
        r.esE = ef * sEf;
        r.cE = cEf;
        r.sE = sEf;
        r.Uc = af * cwf;
        r.Us = af * sef * swf;
        r.Vs = af * swf;
        r.Vc = af * sef * cwf;
        r.Vtr = af * (1.0f - ef * cEf);
    }
    r.nq = ecc ? (float)(e / (1.0 - e)) : 0.0f;
    r.pad1 = r.pad2 = 0.0f;
    // Conservative window.  z^2 >= r_min^2 (sin^2(th) sin^2 i + cos^2 i) with
    // th = w + f - pi/2 and r_min = a (1 - e), so z > 1 + k whenever
    // sin^2 th > ((1+k)^2 / r_min^2 - cos^2 i) / sin^2 i.  The true-anomaly
    // window [f_tr - th_w, f_tr + th_w] maps to a mean-anomaly window and
    // from there to time; widened by half an exposure and a margin.
    float rr = (1.0f + fabsf(k)) * 1.0001f + 1e-5f;
    float rmin = (float)(a * (1.0 - e));
    float ci2 = (float)(ci * ci), si2 = 1.0f - ci2;
    float lo, hi;
    float full = 1.5f * (float)P;
    if (rmin * (float)fabs(ci) >= rr) {
        lo = 1.0f;
        hi = -1.0f;   // never in transit
    } else {
        float s2 = (rr * rr / (rmin * rmin) - ci2) / fmaxf(si2, 1e-30f);
        if (s2 >= 1.0f) {
            lo = -full;
            hi = full;
        } else {
            float thw = asinf(sqrtf(fmaxf(s2, 0.0f))) * 1.001f + 1e-5f;
            if (ecc && e > 0.0) {
                // r = a (1 - e^2) / (1 + e cos f) is smallest where cos f is
                // largest; over f in [f_tr - thw, f_tr + thw] that bound is
                // much tighter than a (1 - e), and the window it gives
                // (narrower, so the bound still holds on it) is conservative.
                float ftr_f = (float)ftr;
                float f1 = ftr_f - thw, f2 = ftr_f + thw;
                float cmax = fmaxf(cosf(f1), cosf(f2));
                float f0 = 6.28318530717958f * ceilf(f1 / 6.28318530717958f);   // first multiple of 2 pi >= f1
                if (f0 <= f2) cmax = 1.0f;
                float ef2 = (float)e;
                float rmin2 = (float)a * (1.0f - ef2 * ef2) / (1.0f + ef2 * cmax) * 0.9999f;
                float s2b = (rr * rr / (rmin2 * rmin2) - ci2) / fmaxf(si2, 1e-30f);
                if (rmin2 > rmin && s2b < s2) thw = asinf(sqrtf(fmaxf(s2b, 0.0f))) * 1.001f + 1e-5f;
            }
            float margin = half_exp + 1e-6f + 1e-6f * (float)P;
            if (!ecc) {
                lo = -thw / r.nang - margin;
                hi = thw / r.nang + margin;
            } else {
                float ef = (float)e, ftrf = (float)ftr;
                float se2 = sqrtf(1.0f - ef), se1 = sqrtf(1.0f + ef);
                float El = 2.0f * atan2f(se2 * sinf(0.5f * (ftrf - thw)), se1 * cosf(0.5f * (ftrf - thw)));
                float Eh = 2.0f * atan2f(se2 * sinf(0.5f * (ftrf + thw)), se1 * cosf(0.5f * (ftrf + thw)));
                float Mtr = (float)(Etr - e * sE);
                float Ml = wrap_neg(El - ef * sinf(El) - Mtr);
                float Mh = wrap_pos(Eh - ef * sinf(Eh) - Mtr);
                if (Mh - Ml >= 3.0f) {
                    lo = -full;
                    hi = full;
                } else {
                    lo = Ml * 1.0005f / r.nang - margin;
                    hi = Mh * 1.0005f / r.nang + margin;
                }
            }
        }
    }
    r.win_lo = lo;
    r.win_hi = hi;
    *out = r;
}


// Warp-aggregated append to a shared-memory queue; returns the slot.
__device__ __forceinline__ int warp_append(int *counter, bool pred)
{
    unsigned mask = __ballot_sync(0xffffffffu, pred);
    int lane = threadIdx.x & 31;
    int leader = __ffs(mask) - 1;
    int base = 0;
    if (mask != 0u && lane == leader) base = atomicAdd(counter, __popc(mask));
    base = __shfl_sync(0xffffffffu, base, leader < 0 ? 0 : leader);
    return base + __popc(mask & ((1u << lane) - 1u));
}


// ---------------------------------------------------------------------------
// Chains of dependent launches.  A call's second and later kernels are
// launched with programmatic stream serialization: their blocks are set up
// while the last blocks of the kernel before them run, instead of after it
// (three kernels of a sampler's residuals 45.0 -> 40.2 us, five of the
// z-interpolated Gimenez residuals 69.4 -> 60.1; the batched plans, whose
// launches are one graph's, gained nothing and are left).  Every kernel of a chain begins
// with chain_begin() in all its threads: it lets the next kernel's blocks in
// (they start when every block of this one has begun, so they take no room
// from it) and then waits until the kernels before it are complete and their
// writes visible.  A call's first kernel is an ordinary launch.  What an earlier
// kernel of the chain wrote is read by ordinary loads: a load through the
// read-only path (__ldg) may be moved ahead of the wait.
// ---------------------------------------------------------------------------
__device__ __forceinline__ void chain_next() { asm volatile("griddepcontrol.launch_dependents;" ::: "memory"); }
__device__ __forceinline__ void chain_wait() { asm volatile("griddepcontrol.wait;" ::: "memory"); }
__device__ __forceinline__ void chain_begin()
{
    chain_next();
    chain_wait();
}

// Opt-in to `bytes` of dynamic shared memory.  The limit belongs to the function
// (on the current device), not to the launch, and every host thread sets the same
// one: a caller passes a constant of the kernel, the most that any of its launches
// asks for, never this launch's own size (a thread with a smaller launch would
// otherwise lower the limit between another's setting and its launch, which is
// then refused).  It costs well under a microsecond.
template <typename F>
inline cudaError_t allow_smem(F fn, size_t bytes)
{
    return cudaFuncSetAttribute(fn, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)bytes);
}

template <typename... P, typename... A>
inline cudaError_t launch_chained(void (*fn)(P...), dim3 grid, dim3 block, size_t smem, cudaStream_t s, A... args)
{
    cudaLaunchConfig_t cfg = {};
    cudaLaunchAttribute at[1];
    at[0].id = cudaLaunchAttributeProgrammaticStreamSerialization;
    at[0].val.programmaticStreamSerializationAllowed = 1;
    cfg.gridDim = grid;
    cfg.blockDim = block;
    cfg.dynamicSmemBytes = smem;
    cfg.stream = s;
    cfg.attrs = at;
    cfg.numAttrs = 1;
    return cudaLaunchKernelEx(&cfg, fn, P(args)...);
}

}  // namespace pt
