// cc_tau32.cuh -- the certified FP32 decision of the edge predicate tau(i,j) < h
// (arXiv:1407.7105 Eq. tauij): the decision itself, and the cheaper tests that
// certify a pair, or all pairs of two groups of bodies, apart.
// The header compiles for the host too, where the tests compare what it
// certifies with the predicate in 64 bits.
#pragma once
#include "cc_fp64.cuh"
#ifndef __CUDACC__
#include <math.h>
#endif

namespace cc {

struct TauParams {
    double G, eps2, eta_in, eta, h, near_tol;
    int eta_outside;
    int fault_test;  // failure-path test hooks of the tau kernels (cc_params.fault_test)
};

#ifdef __CUDA_ARCH__
CC_HD float nan_32() { return __int_as_float(0x7fffffff); }
CC_HD float rsqrt_32(float x) { return rsqrtf(x); }
CC_HD float log2_est(float x) { return __log2f(x); }
// reciprocal square root, PTX rsqrt.approx.ftz.f32 (relative error below
// 2^-22.9 for normal inputs; a denormal input is flushed to zero and gives
// +inf, which the pre-test's comparisons reject)
CC_HD float rsqrt_ftz(float x) { return rsqrt_est(x); }
// two packed FP32 values; the operations round each half as the scalar ones do
CC_HD uint64_t pack2(float a, float b)
{
    uint64_t v;
    asm("mov.b64 %0, {%1, %2};" : "=l"(v) : "f"(a), "f"(b));
    return v;
}
CC_HD void unpack2(uint64_t v, float &a, float &b)
{
    asm("mov.b64 {%0, %1}, %2;" : "=f"(a), "=f"(b) : "l"(v));
}
CC_HD uint64_t add2(uint64_t a, uint64_t b)
{
    uint64_t d;
    asm("add.rn.f32x2 %0, %1, %2;" : "=l"(d) : "l"(a), "l"(b));
    return d;
}
CC_HD uint64_t mul2(uint64_t a, uint64_t b)
{
    uint64_t d;
    asm("mul.rn.f32x2 %0, %1, %2;" : "=l"(d) : "l"(a), "l"(b));
    return d;
}
CC_HD uint64_t fma2(uint64_t a, uint64_t b, uint64_t c)
{
    uint64_t d;
    asm("fma.rn.f32x2 %0, %1, %2, %3;" : "=l"(d) : "l"(a), "l"(b), "l"(c));
    return d;
}
#else
// (the host's own; subnormals flushed where the instruction does)
inline float nan_32() { return u2f(0x7fffffffu); }
inline float rsqrt_32(float x) { return 1.0f / std::sqrt(x); }
inline float log2_est(float x) { return std::log2(x); }
inline float rsqrt_ftz(float x) { return rsqrt_est(std::fabs(x) < 1.17549435e-38f ? 0.0f * x : x); }
inline uint64_t pack2(float a, float b) { return (uint64_t)f2u(b) << 32 | f2u(a); }
inline void unpack2(uint64_t v, float &a, float &b)
{
    a = u2f((uint32_t)v);
    b = u2f((uint32_t)(v >> 32));
}
inline uint64_t add2(uint64_t a, uint64_t b)
{
    return pack2(u2f((uint32_t)a) + u2f((uint32_t)b), u2f((uint32_t)(a >> 32)) + u2f((uint32_t)(b >> 32)));
}
inline uint64_t mul2(uint64_t a, uint64_t b)
{
    return pack2(u2f((uint32_t)a) * u2f((uint32_t)b), u2f((uint32_t)(a >> 32)) * u2f((uint32_t)(b >> 32)));
}
inline uint64_t fma2(uint64_t a, uint64_t b, uint64_t c)
{
    return pack2(fma_f(u2f((uint32_t)a), u2f((uint32_t)b), u2f((uint32_t)c)),
                 fma_f(u2f((uint32_t)(a >> 32)), u2f((uint32_t)(b >> 32)), u2f((uint32_t)(c >> 32))));
}
#endif

// ------------------------------------------------------------ tau, FP32 certified
// Error model (u = 2^-24; +,-,*,fma round to nearest: u each; rsqrtf within
// 2 ulp, budgeted 8u; every bound below is budgeted generously):
//   |dx~ - dx| <= er r,  er = 2.05u + 11u^2 X / r      (float-float difference)
//   |dv~ - dv| <= ev |dv|, ev = 2.05u + 11u^2 V / |dv|
//   rinv = rsqrt(r2), s1 = rsqrt(r mu), s2 = rsqrt(v2)
//   T_ff = eta r2 s1          (= eta sqrt(r^3/mu)),      rel. error <= 40u + 3er
//   T_fb = eta r s2           (= eta r/|dv|),            rel. error <= 40u + 3er + 3ev
//   dT_ff = 1.5 eta rv s1,  dT_fb = eta rv s2 rinv (1 + mu s2^2 rinv)
//   rv = dx.dv has no relative bound (cancellation): |drv| <= (er+ev+4u) r |dv|,
//   so |d dT| <= 32u|dT_ff| + 1.5 eta s1 |drv|   (ff)
//              80u|dT_fb| + eta s2 rinv (1 + mu s2^2 rinv) |drv|   (fb)
//   D = 1 - min(dT,1)/2 >= 1/2,  |dD| <= |d dT|/2 + 2u D
// tau_x = T_x / D_x < h is certain when T~(1+eT)(1+s) < h (D~ - dD), and
// certainly false when T~(1-eT)(1-s) >= h (D~ + dD); the slack s = 2e-6
// covers the FP32 evaluation of the bounds and the FP64 predicate's own
// rounding.  Any NaN/Inf fails both tests: the pair is undecided.
//
// Range.  The model holds while no quantity overflows and none that carries
// the result loses bits below the normal floats.  So a pair stays undecided
// unless r^2 >= TAU_TINY, mu >= TAU_MU_MIN and r mu is finite; its flyby term
// is used from |dv|^2 >= TAU_TINY on; and eta/h is NaN, which leaves every pair
// undecided, unless the constants lie in the ranges that mixed_etah asks for.
// Then, with 1/r <= 1e15, s2 <= 1e15 and s1 <= 3.2e18:
//   an infinite r^2 or |dv|^2 makes its root's product NaN; what else overflows
//   (rv, mu/v^2) makes dD infinite or NaN, and its term proves nothing;
//   a term that underflows was below 2^-126 beside a sum above 1e-30, and the
//   float-float roundings of 2^-149 are far below u r and u |dv|;
//   T/h, a product left to right, is too small only when the true one is below
//   1e-19 (D - dD is not: dD covers u D).  It may overflow early: T_ff is then
//   above a finite D all the same (etah r^2 >= 3.4e38 > 0.75 eta |rv|, whose
//   double did not overflow), an infinite T_fb proves nothing (tau_decide_at);
//   below |dv|^2 = TAU_TINY |dv| counts as 1e-15, so that drv holds all of c_v (an
//   FP32 difference of zero may hide one of that size).
// With G <= 1e14 TAU_MU_MIN is above tau_mu_floor.  A pair that this leaves undecided is looked
// at once more in units of its own (tau_wide).
constexpr float U32 = 5.9604645e-8f;  // 2^-24
constexpr float SLACK = 2e-6f;
constexpr float TAU_TINY = 1e-30f, TAU_HUGE = 1e37f, TAU_MU_MIN = 1e-22f;

// eta and eta/h in float (the decision compares T/h with D); c_x = 11 u^2 X
// and c_v = 11 u^2 V carry the float-float rounding of the differences
struct MixedTauParams {
    float eta, etah, eps2, G;
    float hq;  // eta/etah (h, or h/eta when eta multiplies the min): the pre-test's q = hq |dv|/r
};
// the tau kernel's: with tau_pair_bounds' constants (c^2, log2 T^2 and log2 V of
// its bounds; pb_c2 < 0: they are off)
struct MixedTauBounds : MixedTauParams {
    float pb_c2, pb_lt, pb_lv;
};

// eta/h in float: NaN, which settles no pair in any test of this file, when a
// constant is outside the range that they hold in
CC_HD float mixed_etah(double eta_in, double eta, int eta_outside, double h, double G, double eps2)
{
    const float etah = (float)(eta_outside ? eta_in * eta / h : eta_in / h);
    const float e = (float)eta_in, g = (float)G, s = (float)eps2;
    const bool in = etah >= 1e-30f && etah <= 1e30f && e >= 1e-5f && e <= 1e3f && g >= 1e-30f && g <= 1e14f && s <= TAU_HUGE;
    return in ? etah : nan_32();
}

// mu from which its float is good to the model's u (a mass below the normal floats
// is off by up to 2^-150).  The tests that only need mu from above take no less.
CC_HD float tau_mu_floor(const MixedTauParams &Q) { return 1e-36f * fmaxf(1.f, Q.G); }

// The h-independent part of the decision: everything except T/h.  The
// decision at a threshold h then costs two products and four comparisons,
// and since eta/h doubles exactly when h halves, T/h at h 2^-m is T/h at h
// times 2^m bit for bit: decide(prep, etah * 2^m) is the decision the full
// evaluation would take at h 2^-m for the same state.
struct TauPrep32 {
    float r2, s1, r, s2;         // Tff/h = (etah r2) s1, Tfb/h = (etah r) s2
    float ffA, ffB, ffLo, ffHi;  // ff edge certain: Tff ffA < ffLo; no edge certain: Tff ffB >= ffHi
    float fbA, fbB, fbLo, fbHi;  // the same for the flyby term
    bool fb;                     // flyby term usable (else only a certain ff edge decides)
};

CC_HD TauPrep32 tau_prep_fp32(float dx0, float dx1, float dx2, float dv0, float dv1, float dv2,
                                                   float mu, float c_x, float c_v, const MixedTauParams &Q)
{
    TauPrep32 t;
    const float A = 1.f + SLACK, B = 1.f - SLACK;
    const float r2 = fmaf(dx2, dx2, fmaf(dx1, dx1, fmaf(dx0, dx0, Q.eps2)));
    const float v2 = fmaf(dv2, dv2, fmaf(dv1, dv1, dv0 * dv0));
    const float rv = fmaf(dx2, dv2, fmaf(dx1, dv1, dx0 * dv0));
    const float rinv = rsqrt_32(r2);
    const float r = r2 * rinv;
    const float rm = r * mu;
    const float s1 = rsqrt_32(rm);
    const bool in = r2 >= TAU_TINY && mu >= TAU_MU_MIN && rm <= 3.4e38f;  // (NaN is out)
    const float er = fmaf(c_x, rinv, 2.05f * U32);
    const float w2 = fmaxf(v2, TAU_TINY), s2 = rsqrt_32(w2);
    const float vn = w2 * s2;  // |dv|
    const float ev = fmaf(c_v, s2, 2.05f * U32);
    const float drv = (er + ev + 4.f * U32) * (r * vn);
    // free fall: T/h = (eta/h) r2 s1, dT/dt = 1.5 eta rv s1
    const float dTff = 1.5f * Q.eta * rv * s1;
    const float Dff = fmaf(-0.5f, fminf(dTff, 1.f), 1.f);
    const float dDff = fmaf(0.5f, fmaf(32.f * U32, fabsf(dTff), 1.5f * Q.eta * s1 * drv), 2.f * U32 * Dff);
    const float eff = fmaf(3.f, er, 40.f * U32);
    t.r2 = in ? r2 : nan_32();  // out of range: T_ff/h is NaN, T_fb not used
    t.s1 = s1;
    t.r = r;
    t.s2 = s2;
    t.ffA = fmaf(eff, A, A);
    t.ffB = fmaf(-eff, B, B);
    t.ffLo = Dff - dDff;
    t.ffHi = Dff + dDff;
    // an exactly zero (or unresolved) FP32 velocity difference may hide a
    // tiny nonzero FP64 one, whose flyby term can be small: only a certain
    // free-fall edge decides such a pair
    t.fb = in && v2 >= TAU_TINY && !(vn < 6.f * c_v);
    // flyby: T/h = (eta/h) r s2, dT/dt = eta rv s2 rinv (1 + mu s2^2 rinv)
    const float g = fmaf(mu * s2 * s2, rinv, 1.f);
    const float k = s2 * rinv * g;
    const float dTfb = Q.eta * rv * k;
    const float Dfb = fmaf(-0.5f, fminf(dTfb, 1.f), 1.f);
    const float dDfb = fmaf(0.5f, fmaf(80.f * U32, fabsf(dTfb), Q.eta * k * drv), 2.f * U32 * Dfb);
    const float efb = fmaf(3.f, er + ev, 40.f * U32);
    t.fbA = fmaf(efb, A, A);
    t.fbB = fmaf(-efb, B, B);
    t.fbLo = Dfb - dDfb;
    t.fbHi = Dfb + dDfb;
    return t;
}

// returns 1 = edge certain, 0 = no edge certain, -1 = undecided; etah =
// eta/h in float
CC_HD int tau_decide_at(const TauPrep32 &t, float etah)
{
    const float Tff = etah * t.r2 * t.s1;
    const bool ff_yes = Tff * t.ffA < t.ffLo;
    if (!t.fb) return ff_yes ? 1 : -1;
    const bool ff_no = Tff * t.ffB > t.ffHi;  // (not when both are infinite)
    const float Tfb = etah * t.r * t.s2;
    const bool fb_yes = Tfb * t.fbA < t.fbLo;
    const bool fb_no = Tfb * t.fbB > t.fbHi;
    if (ff_yes || fb_yes) return 1;
    if (ff_no && fb_no && Tfb <= 3.4e38f) return 0;
    return -1;
}

// Units of a pair's own: powers of two (exact) 2^a for lengths and 2^v for speeds
// that bring r into [1, 4) and mu and |dv| around it: with q = log2 of mu/(r |dv|^2),
// whatever the units, |dv|' is near 2^(-q/4) and mu' near 2^(q/2).  a, b, c: the
// exponents of r, |dv| and mu.
CC_HD int tau_speed_unit(int a, int b, int c, bool still, int &q)
{
    q = still ? 0 : c - a - 2 * b;
    return still ? (c - a) / 2 : b + q / 4;
}
CC_HD int exp_of_f(float x) { return (int)((f2u(x) >> 23) & 0xffu) - 127; }  // x > 0; subnormals: below any other
CC_HD float two_to_f(int k) { return u2f((uint32_t)(127 + k) << 23); }

// The decision for one pair in units of its own, from float differences (c_x, c_v
// as in tau_prep_fp32): what the floats hold, whatever the caller's units, is in
// the range of the model, but for mu/(r |dv|^2) outside 2^+-140.  For the pairs
// that the tau kernel's certificates leave open; ~30 operations more a pair.
CC_HD int tau_decide_own(const float d[6], float mu, float c_x, float c_v, const MixedTauParams &Q)
{
    const float big_x = fmaxf(fabsf(d[0]), fmaxf(fabsf(d[1]), fabsf(d[2])));
    const float big_v = fmaxf(fabsf(d[3]), fmaxf(fabsf(d[4]), fabsf(d[5])));
    const int ax = exp_of_f(big_x), ae = Q.eps2 > 0.f ? (exp_of_f(Q.eps2) + 1) >> 1 : -127, a = ax > ae ? ax : ae;
    const int b = exp_of_f(big_v), c = exp_of_f(mu);
    const bool still = big_v == 0.f;
    int q;
    const int v = tau_speed_unit(a, b, c, still, q), te = a - v;
    // (100: the float-float roundings of 2^-149 stay far below u r and u |dv|; an
    // eps^2 near or below the least float, which mixed_tau_params keeps above zero,
    // is nothing beside r^2 >= 2^-90)
    const bool in = a >= -100 && a <= 100 && v >= -100 && v <= 100 && te >= -120 && te <= 120 && q >= -140 &&
                    q <= 140 && (still || b >= -100) && mu >= tau_mu_floor(Q) && mu <= 3.4e38f &&
                    (Q.eps2 == 0.f || Q.eps2 >= TAU_TINY || a >= -45);
    if (!in) return -1;
    const float X = two_to_f(-a), V = two_to_f(-v);
    MixedTauParams U = Q;
    U.etah = Q.etah * two_to_f(te);
    U.eps2 = Q.eps2 * X * X;
    const float m = u2f((f2u(mu) & 0x7fffffu) | ((uint32_t)(127 + c - a - 2 * v) << 23));
    if (!(U.etah >= 1e-30f && U.etah <= 1e30f)) return -1;
    return tau_decide_at(tau_prep_fp32(d[0] * X, d[1] * X, d[2] * X, d[3] * V, d[4] * V, d[5] * V, m, c_x * X, c_v * V, U),
                         U.etah);
}

// The same from a pair's 64-bit differences, for pairs that the decision left
// open: for the range of the floats, or because the float pairs do not resolve a
// difference far from the origin (near-threshold pairs stay open as before).  For
// pairs whose quantities the predicate's own 64-bit operations take without
// overflow or underflow.
struct TauWide {
    TauPrep32 t;
    float etah;  // eta/h in these units, for the first threshold
    bool in;     // else every pair is open
    bool still;  // |dv|^2 is zero in 64 bits: the predicate has no flyby term
};

// the exponent of a positive finite x; zero and subnormals: below any other
CC_HD int exp_of(double x) { return (int)((d2u(x) >> 52) & 0x7ffu) - 1023; }
CC_HD double two_to(int k) { return u2d((uint64_t)(1023 + k) << 52); }

CC_HD TauWide tau_wide(const double dx[3], const double dv[3], double mi, double mj, const TauParams &P, double h)
{
    TauWide w;
    const double mu = P.G * (mi + mj), big_x = fmax(fmax(fabs(dx[0]), fabs(dx[1])), fmax(fabs(dx[2]), sqrt(P.eps2)));
    const double big_v = fmax(fmax(fabs(dv[0]), fabs(dv[1])), fabs(dv[2]));
    const int a = exp_of(big_x), c = exp_of(mu), b = exp_of(big_v);
    w.still = big_v == 0.0;
    int q;
    const int vb = tau_speed_unit(a, b, c, w.still, q), te = a - vb;  // the unit of time: 2^te
    const double e = (P.eta_outside ? P.eta_in * P.eta / h : P.eta_in / h) * two_to(te < -900 ? -900 : te > 900 ? 900 : te);
    w.in = a >= -250 && a <= 250 && c >= -250 && c <= 250 && (w.still || (b >= -250 && b <= 250)) && q >= -140 && q <= 140 &&
           e >= 1e-30 && e <= 1e30 && P.eta_in >= 1e-5 && P.eta_in <= 1e3 && mi > 0.0 && mj > 0.0;
    if (!w.in) return w;
    const double X = two_to(-a), V = two_to(-vb);
    MixedTauParams Q;
    Q.eta = (float)P.eta_in;
    Q.etah = w.etah = (float)e;
    Q.eps2 = (float)(P.eps2 * X * X);
    Q.G = 0.f;
    Q.hq = 0.f;
    w.t = tau_prep_fp32((float)(dx[0] * X), (float)(dx[1] * X), (float)(dx[2] * X), (float)(dv[0] * V),
                        (float)(dv[1] * V), (float)(dv[2] * V), (float)(mu * X * V * V), 0.f, 0.f, Q);
    return w;
}

// the decision of tau_decide_at (etah: w.etah 2^m for the threshold h 2^-m)
CC_HD int tau_decide_wide(const TauWide &w, float etah)
{
    if (!w.in) return -1;
    if (w.still) {
        const float Tff = etah * w.t.r2 * w.t.s1;
        return Tff * w.t.ffA < w.t.ffLo ? 1 : Tff * w.t.ffB > w.t.ffHi ? 0 : -1;
    }
    return tau_decide_at(w.t, etah);
}

// A sufficient test for "no edge" that skips the certified evaluation for
// the great majority of pairs (those whose tau is well above h).  With T =
// T_ff or T_fb and D = 1 - min(dT/dt, 1)/2, tau_x = T/D and D <= 1 + |dT/dt|/2:
//   free fall: |dT_ff/dt| = 1.5 T_ff |rv|/r^2 <= 1.5 T_ff |dv|/r, so
//     tau_ff >= h  if  (T_ff/h) (1 - 0.75 q) >= 1,  q = h|dv|/r (q < 4/3);
//   flyby:     |dT_fb/dt| <= eta (1 + mu/(r v^2))  (T_fb = eta r/|dv|), so
//     tau_fb >= h  if  T_fb/h >= 1 + eta (1 + mu/(r v^2))/2.
// (eta is the factor inside T: Q.eta; hq = h/eta_in, the same as
// eta/etah in both readings of the eta placement.)  The differences may be
// formed from the rounded high parts alone: then |dx~ - dx| <= u r + c_x
// + 3.5 u r with c_x = 7 u max|x_i| (per component |x_j| <= |x_i| + r),
// likewise c_v for the velocities.  Once (c_x + 3.5 u r)/r and the velocity
// analogue are below 1e-4, every FP32 quantity used has relative
// error below 1e-3 (the error model above: 40u + 3(er + ev) plus the rsqrt
// budget), so a 2 % margin on each inequality makes the test rigorous; a
// pair it does not settle goes to the certified decision.  Out of the range
// above nothing is certified (r mu may be too large: then T_ff = 0), nor from a
// T that overflowed, which mu/(r v^2) may have done too.  (A larger mu makes the
// test stricter: mu from its floor on.)
CC_HD bool tau_quick_apart(float dx0, float dx1, float dx2, float dv0, float dv1, float dv2,
                                                float mu, float c_x, float c_v, const MixedTauParams &Q)
{
    const float r2 = fmaf(dx2, dx2, fmaf(dx1, dx1, fmaf(dx0, dx0, Q.eps2)));
    const float v2 = fmaf(dv2, dv2, fmaf(dv1, dv1, dv0 * dv0));
    const float rinv = rsqrt_ftz(r2);
    const float r = r2 * rinv;
    const float m = fmaxf(mu, tau_mu_floor(Q)), rm = r * m;
    const float s1 = rsqrt_ftz(rm);
    const float s2 = rsqrt_ftz(v2);   // inf for v2 = 0: rejected below
    const float vn = v2 * s2;         // |dv|
    const float Tff = Q.etah * r2 * s1;                  // T_ff / h
    const float q = Q.hq * vn * rinv;                    // h |dv| / r
    const float Tfb = Q.etah * r * s2;                   // T_fb / h
    const float g = m * rinv * s2 * s2;                  // mu / (r v^2)
    const float M = 1.02f;
    // (the bounds below leave 3.5u for a relative part of c_x/r, c_v/|dv|;
    // all conditions are evaluated: no short-circuit branches)
    const bool ok = (fminf(r2, v2) >= TAU_TINY) & (rm >= 2e-38f) & (fmaxf(r2, v2) <= TAU_HUGE) &
                    (fmaxf(Tff, Tfb) <= 3.4e38f) & (c_x * rinv <= 0.99e-4f) & (v2 > 0.f) & (c_v * s2 <= 0.99e-4f) & (0.75f * M * q < 1.f) &
                    (Tff * fmaf(-0.75f * M, q, 1.f) >= M) & (Tfb >= M * fmaf(0.5f * Q.eta, 1.f + g, 1.f));
    return ok;
}

// The same bounds over every pair of two groups of bodies at once.  A group
// is summarised by the boxes of its high parts (positions, velocities) and
// its largest G m.  Over pairs (i in A, j in B): r >= d = the boxes'
// distance (softened), |dv| <= vmax (the velocity boxes' widest relative
// speed), mu <= muA + muB.  Free fall: T_ff/h = etah sqrt(r^3/mu) grows with
// r and falls with mu, q = hq |dv|/r grows with |dv| and falls with r, so
// (T_ff/h)(1 - 0.75 q) >= 1 for every pair once it holds at (d, vmax,
// mu_max).  Flyby: with T_fb/h = etah r/v and |dT/dt| <= eta (1 + mu/(r
// v^2)), tau_fb/h >= f(r, v) = 2 etah r^2 v / ((2 + eta) r v^2 + eta mu),
// which grows with r and falls with mu; f >= 1 holds for v between the two
// roots v- < v+ of (2 + eta) d v^2 - 2 etah d^2 v + eta mu_max = 0.  Slow
// pairs fall below v- (approaching bodies with |dv| -> 0 have tau -> 0 in
// this form), so the groups are certified apart only for pairs with
// |dv| >= v-: the function returns true when every pair has tau_ff >= h
// and vmax <= v+, and sets vthr2 so that a pair whose high-part velocity
// difference has |dv~|^2 >= vthr2 is certified apart (vthr adds 16 u max|v|
// for the high parts' rounding and that of their difference: at most
// sqrt(3) (2 u max|v| + u |dv~|) <= 9.5 u max|v|).  pad_x, pad_v bound |x - x_hi| + |x' - x'_hi|
// over the two groups (likewise v); the 2 % margin M absorbs the FP32
// rounding of these few operations.
struct GroupBox {
    float xlo[3], xhi[3], vlo[3], vhi[3];
    float gm;    // max G m of the group (high part)
    float amax;  // max |x_hi| component
    float vabs;  // max |v_hi| component
};

CC_HD bool tau_groups_apart(const GroupBox &A, const GroupBox &B, const MixedTauParams &Q,
                                                 float &vthr2)
{
    const float M = 1.02f;
    const float pad_x = 4.f * U32 * fmaxf(A.amax, B.amax);
    const float pad_v = 4.f * U32 * fmaxf(A.vabs, B.vabs);
    float d2 = Q.eps2, w2 = 0.f;
#pragma unroll
    for (int k = 0; k < 3; ++k) {
        const float g = fmaxf(0.f, fmaxf(B.xlo[k] - A.xhi[k], A.xlo[k] - B.xhi[k]) - pad_x);
        const float w = fmaxf(0.f, fmaxf(B.vhi[k] - A.vlo[k], A.vhi[k] - B.vlo[k])) + pad_v;
        d2 = fmaf(g, g, d2);
        w2 = fmaf(w, w, w2);
    }
    const float d = sqrtf(d2), vmax = fmaxf(sqrtf(w2), 1e-18f);  // (squares below the floats: at most that)
    const float mu = fmaxf((A.gm + B.gm) * 1.0001f, tau_mu_floor(Q));
    if (!(d2 >= TAU_TINY) || !(d2 <= TAU_HUGE)) return false;
    // free fall at (d, vmax, mu_max)
    const float X = Q.etah * d * sqrtf(d / mu);
    const float q = Q.hq * vmax / d;
    if (!(X * (1.f - 0.75f * M * q) >= M) || !(X <= TAU_HUGE)) return false;
    // flyby: the roots of v^2 - 2 b v + c with the margin M on f >= 1 (b is a
    // speed: its square is in range where the speeds' are)
    const float e = Q.etah * d2, b = e / (M * (2.f + Q.eta) * d), c = Q.eta * mu / ((2.f + Q.eta) * d);
    const float disc = b * b - c;
    if (!(e >= TAU_TINY) || !(disc >= TAU_TINY) || !(disc <= TAU_HUGE)) return false;
    const float vp = b + sqrtf(disc);
    const float vm = c / vp;
    if (!(vmax <= vp * 0.9999f)) return false;
    const float vt = fmaxf(vm * 1.0001f + 4.f * pad_v, 1e-15f);
    vthr2 = vt * vt;
    return true;
}

// The same two bounds for single pairs of the groups, as three comparisons on
// r~^2 and |dv~|^2 (no square root, no division): with T_ff/h = etah
// sqrt(r^3/mu), f(r, v) as above and mu <= mu_max,
//   (3) r >= c v,  c = M (2 + eta) / (2 etah (1 - D)):  the first term of the
//       flyby's denominator takes the share 1 - D of its numerator, and q =
//       hq v/r <= hq/c;
//   (1) r >= r_min, r_min^3 = mu_max T^2, T = M/(etah (1 - 0.75 M hq/c)):
//       free fall at that q;
//   (2) v >= v_thr = V mu_max/r_min^2, V = M eta/(2 etah D): the flyby's second
//       term takes the share D.
// M = 1.02 covers the FP32 rounding and the high parts': r_min >= 1.02e3 c_x
// and v_thr >= 1.02e3 c_v (c_x = 7.1 u max|x_i|, c_v likewise) put the
// relative error of r~ and v~ below 1e-3 + 4.5u, of r^2 v below 4e-3.
// The kernel forms p = r~^2 - r_min^2 and w = v~^2 - v_thr^2 by starting
// their sums at -r_min^2 (+ eps^2) and -v_thr^2, and asks for w >= 0 and p -
// c^2 w >= 0: that is (3) with r_min^2 - c^2 v_thr^2 to spare (r_min is
// raised until it is not negative), and it implies (1).  Returns false when
// the bounds cannot be used (the caller then leaves every pair open); the
// caller has seen that all |x|, |v| are below TAU_WILD, so no sum overflows
// (3 (2 TAU_WILD)^2 < 3.4e38: parsecs in SI and CGS units are inside).
constexpr float TAU_WILD = 5e18f;
// whether a body's high parts and G m are inside what the bounds allow for
// (NaN is not)
CC_HD bool tau_in_box(const float s[6], float gm)
{
    bool in = gm >= 0.f && gm < 1e36f;
    for (int k = 0; k < 6; ++k) in = in && fabsf(s[k]) < TAU_WILD;
    return in;
}

struct PairBounds {
    float p0, w0;  // eps^2 - r_min^2, -v_thr^2
};

CC_HD bool tau_pair_bounds(float amax, float vabs, float mu_max, const MixedTauBounds &Q,
                                                PairBounds &b)
{
    // r_min and v_thr by exp2 of sums of logarithms, which no unit takes out of
    // the floats' range; their error (below 1e-4) is far inside the 5e-4
    const float lm = log2_est(fmaxf(mu_max * 1.0001f, tau_mu_floor(Q)));
    float rmin = 1.0005f * exp2f((lm + Q.pb_lt) * (1.f / 3.f));
    rmin = fmaxf(rmin, fmaxf(1.02e3f * 7.1f * U32 * amax, 1e-15f));
    float vt = 1.0005f * exp2f(lm + Q.pb_lv - 2.f * log2_est(rmin));
    vt = fmaxf(vt, fmaxf(1.02e3f * 7.1f * U32 * vabs, 1e-15f));
    const float w2 = vt * vt, p2 = fmaxf(rmin * rmin, 1.0001f * Q.pb_c2 * w2);
    b.p0 = Q.eps2 - p2;
    b.w0 = -w2;
    return Q.pb_c2 >= 0.f && w2 < TAU_HUGE && p2 < TAU_HUGE;
}

// those sums for two columns of a row at a time (the packed differences of
// their high parts): the sign bit of a half is set when its pair stays open
CC_HD uint64_t tau_speed_open(uint64_t du, uint64_t dv, uint64_t dw, uint64_t w0)
{
    return fma2(dw, dw, fma2(dv, dv, fma2(du, du, w0)));
}
CC_HD uint64_t tau_pair_open(uint64_t dx, uint64_t dy, uint64_t dz, uint64_t du, uint64_t dv, uint64_t dw, uint64_t p0,
                             uint64_t w0, uint64_t nc2 /* -c^2 twice */)
{
    const uint64_t pp = fma2(dz, dz, fma2(dy, dy, fma2(dx, dx, p0)));
    const uint64_t ww = tau_speed_open(du, dv, dw, w0);
    return fma2(ww, nc2, pp) | ww;
}

// The same with (2) taken at each pair's own separation: v >= V mu_max/r^2 as
// (a p)^2 w >= a^2 (V mu_max)^2 with p = r~^2 - r_min^2 and w = v~^2 - v_fl^2, v_fl the
// least speed that the high parts resolve (1.02e3 c_v).  p <= r^2 and w <= v^2, so it
// implies (2) with the margin of V, and w >= 0; (3) and (1) as before, with v_fl in
// v_thr's place.  In a cold system v_thr, which is V mu_max/r_min^2, is above most
// speeds at separations far above r_min.  a, a power of two, keeps a p below 2^50 and
// (a p)^2 w below 2^100 whatever the units; a product that underflows leaves its
// pair open.  Returns false when the threshold is out of the floats' range.
struct PairFar {
    float p0, w0, a, k;  // eps^2 - r_min^2, -v_fl^2, a, -a^2 (V mu_max)^2
};

// xmax: both groups' largest |x_hi| component; wmax: their widest relative speed per
// component (of the high parts)
CC_HD bool tau_pair_far(float amax, float vabs, float xmax, float wmax, float mu_max, const MixedTauBounds &Q, PairFar &f)
{
    // (3.6 = log2 12: p <= 12 xmax^2 + eps^2, w <= 12 wmax^2)
    const float lm = log2_est(fmaxf(mu_max * 1.0001f, tau_mu_floor(Q)));
    float rmin = 1.0005f * exp2f((lm + Q.pb_lt) * (1.f / 3.f));
    rmin = fmaxf(rmin, fmaxf(1.02e3f * 7.1f * U32 * amax, 1e-15f));
    const float vf = fmaxf(1.02e3f * 7.1f * U32 * vabs, 1e-15f), w2 = vf * vf;
    const float p2 = fmaxf(rmin * rmin, 1.0001f * Q.pb_c2 * w2);
    const float lp = fmaxf(2.f * log2_est(xmax) + 3.6f, log2_est(Q.eps2)) + 1.f, lw = 2.f * log2_est(wmax) + 3.6f;
    const float la = floorf(fminf(50.f, 50.f - 0.5f * lw) - lp), lk = 2.f * (lm + Q.pb_lv + la);
    f.p0 = Q.eps2 - p2;
    f.w0 = -w2;
    f.a = exp2f(la);
    f.k = -1.002f * exp2f(lk);
    return Q.pb_c2 >= 0.f && p2 < TAU_HUGE && w2 < TAU_HUGE && fabsf(la) <= 120.f && lk >= fmaxf(lw, 0.f) - 110.f &&
           lk <= 110.f;
}
CC_HD uint64_t tau_far_open(uint64_t dx, uint64_t dy, uint64_t dz, uint64_t du, uint64_t dv, uint64_t dw, uint64_t p0,
                            uint64_t w0, uint64_t nc2, uint64_t a, uint64_t k)
{
    const uint64_t pp = fma2(dz, dz, fma2(dy, dy, fma2(dx, dx, p0)));
    const uint64_t ww = tau_speed_open(du, dv, dw, w0), t = mul2(pp, a);
    return fma2(ww, nc2, pp) | fma2(mul2(t, t), ww, k);
}

// the widest relative speed between two groups, per component from their boxes
CC_HD float tau_speed_span(const GroupBox &A, const GroupBox &B)
{
    float w = 0.f;
#pragma unroll
    for (int k = 0; k < 3; ++k) w = fmaxf(w, fmaxf(B.vhi[k] - A.vlo[k], A.vhi[k] - B.vlo[k]));
    return w;
}

// the FP32 constants of a split at threshold P.h
inline MixedTauBounds mixed_tau_params(const TauParams &P)
{
    MixedTauBounds Q;
    const double etah = P.eta_outside ? P.eta_in * P.eta / P.h : P.eta_in / P.h;
    const double hq = P.eta_outside ? P.h / P.eta : P.h;  // h/eta_in in the units of T: eta_in/etah
    Q.eta = (float)P.eta_in;
    Q.etah = mixed_etah(P.eta_in, P.eta, P.eta_outside, P.h, P.G, P.eps2);
    Q.eps2 = P.eps2 > 0.0 ? fmaxf((float)P.eps2, 1e-37f) : 0.f;
    Q.G = (float)P.G;
    Q.hq = (float)hq;
    // D: a 3 % tighter (3) at the usual eta; more where eta is not small
    const double M = 1.02, D = fmax(1.0 / 32, 0.75 * P.eta_in / (2.0 + P.eta_in));
    const double c = M * (2.0 + P.eta_in) / (2.0 * etah * (1.0 - D));
    const double q = hq / c, T = M / (etah * (1.0 - 0.75 * M * q));
    Q.pb_c2 = (float)(c * c * 1.0001);
    Q.pb_lt = (float)(2.0 * log2(T));
    Q.pb_lv = (float)log2(M * P.eta_in / (2.0 * etah * D));
    // (q >= 4/(3M) has no free-fall bound; constants outside the float range)
    if (!(Q.etah > 0.f) || !(0.75 * M * q < 0.95) || !(Q.pb_c2 > 1e-36f) || !(Q.pb_c2 < 1e30f)) Q.pb_c2 = -1.f;
    return Q;
}

}  // namespace cc
