// cc_device.cuh -- device functions shared by several kernels of libcc.so:
// float-float splits, edge depths, compensated summation, and the universal-
// variable two-body flow of the CC_KEPLER variant (arXiv:1407.7105 Sec. 3.2).
// (The certified FP32 decision of the edge predicate is in cc_tau32.cuh.)
#pragma once
#include "cc_fp64.cuh"
#include "cc_internal.cuh"
#include "cc_tau32.cuh"

namespace cc {

// 2^k as a float (0 <= k <= 127); 2^-k as a double (0 <= k <= 1022)
__device__ __forceinline__ float pow2f(int k) { return __int_as_float((127 + k) << 23); }
__device__ __forceinline__ double pow2m(int k) { return __longlong_as_double((long long)(1023 - k) << 52); }

// x 2^-k for a normal x whose result stays normal: an exponent-field
// subtraction (exact, and no FP64 instruction)
__device__ __forceinline__ double scale2m(double x, int k)
{
    return __longlong_as_double(__double_as_longlong(x) - ((long long)k << 52));
}

// The first m >= 0 with h 2^-m <= tau (the first threshold of the sequence
// h, h/2, h/4, ... at which tau < threshold fails), at most `levels`.  h is
// positive and normal; the comparison is exact: (exponent, significand) of
// h 2^-m against those of tau.  NaN tau: 0 (the predicate is false).
__device__ __forceinline__ int first_level_at_or_below(double tau, double h, int levels)
{
    if (!(tau < h)) return 0;
    if (!(tau >= 2.2250738585072014e-308)) return levels;  // 0, negative or subnormal: below every threshold
    const long long bt = __double_as_longlong(tau), bh = __double_as_longlong(h);
    const int et = (int)(bt >> 52), eh = (int)(bh >> 52);
    const long long mt = bt & 0xFFFFFFFFFFFFFll, mh = bh & 0xFFFFFFFFFFFFFll;
    const int m = eh - et + (mh <= mt ? 0 : 1);
    return m < levels ? m : levels;
}

// The first m in [m0, levels) at which the wide decision says no edge at
// h 2^-m; `levels` if every one is an edge; -1 when it leaves one open (or
// there are more than a hundred: 2^m is a float).
__device__ __forceinline__ int tau_wide_level(const TauWide &w, int m0, int levels)
{
    for (int m = m0; m < levels; ++m) {
        if (m > 100) return -1;
        const int dec = tau_decide_wide(w, w.etah * pow2f(m));
        if (dec < 0) return -1;
        if (dec == 0) return m;
    }
    return levels;
}

// What the FP32 decision left open at h 2^-m0: the first of the thresholds up
// to h 2^-levels that the pair is no edge at (e), from the decision in the pair's
// own units, else (e = -1) the FP64 tau.
struct TauOpen {
    double tau;
    int e;
};
__device__ __forceinline__ TauOpen tau_open(double dx0, double dx1, double dx2, double dv0, double dv1, double dv2,
                                            double mi, double mj, const TauParams &P, double h, int m0, int levels)
{
    const double dx[3] = {dx0, dx1, dx2}, dv[3] = {dv0, dv1, dv2};
    TauOpen o;
    o.tau = 0.0;
    o.e = tau_wide_level(tau_wide(dx, dv, mi, mj, P, h), m0, levels);
    if (o.e < 0) o.tau = tau_fp64(dx0, dx1, dx2, dv0, dv1, dv2, mi, mj, P);
    return o;
}

// Float-float split of a double: hi = fl32(x) (round to nearest even),
// lo = fl32(x - hi).  For |x| in [2^-74, 2^127) it is computed with integer
// operations and int->float conversions (the significand rounded to 24
// bits by integer arithmetic, the remainder converted exactly-then-rounded),
// giving the same two floats as the FP64 route at a fraction of its cost on
// a part whose FP64 pipe is 1/58 of the FP32 rate; outside that range it
// takes the FP64 route.
__device__ __forceinline__ void ff_split(double x, float &hi, float &lo)
{
    const unsigned long long b = (unsigned long long)__double_as_longlong(x);
    const int e = (int)((b >> 52) & 0x7FFull);
    if (e < 949 || e > 1150) {
        hi = __double2float_rn(x);
        lo = __double2float_rn(x - (double)hi);
        return;
    }
    const long long F = (long long)((b & 0xFFFFFFFFFFFFFull) | 0x10000000000000ull);  // 53-bit significand
    const long long Fr = (F + 0x0FFFFFFFll + ((F >> 29) & 1ll)) >> 29;             // 24 bits, nearest even
    const int d = (int)(F - (Fr << 29));                                           // |d| <= 2^28
    const float s_hi = __int_as_float((e - 1046 + 127) << 23);                     // 2^(e-1046)
    const float s_lo = __int_as_float((e - 1075 + 127) << 23);                     // 2^(e-1075)
    const float h = __int2float_rn((int)Fr) * s_hi;
    const float l = __int2float_rn(d) * s_lo;
    const bool neg = (b >> 63) != 0ull;
    hi = neg ? -h : h;
    lo = neg ? -l : l;
}

// fl32(x) = round-to-nearest-even double -> float, by integer arithmetic for
// results in the normal float range (same value as __double2float_rn); the
// conversion instruction costs ~180 cycles per warp on GB300.
__device__ __forceinline__ float fl32(double x)
{
    const unsigned long long b = (unsigned long long)__double_as_longlong(x);
    const int e = (int)((b >> 52) & 0x7FFull);
    if (e < 1023 - 126 || e > 1023 + 126) return __double2float_rn(x);
    const unsigned long long mag = b & 0x7FFFFFFFFFFFFFFFull;
    const unsigned long long r = mag + 0x0FFFFFFFull + ((mag >> 29) & 1ull);  // drop 29 bits, nearest even
    const unsigned int fb = (unsigned int)((r >> 29) - (896ull << 23)) | ((unsigned int)(b >> 32) & 0x80000000u);
    return __uint_as_float(fb);
}

// f2d(f) = the exact double of a float, by integer arithmetic for normal
// floats and zeros (the conversion instruction costs ~140 cycles per warp)
__device__ __forceinline__ double f2d(float f)
{
    const unsigned int u = __float_as_uint(f);
    const unsigned int ex = (u >> 23) & 0xFFu;
    if ((u & 0x7FFFFFFFu) == 0u) return __longlong_as_double((long long)((unsigned long long)u << 32));
    if (ex == 0u || ex == 255u) return (double)f;
    const unsigned long long b = ((unsigned long long)(u & 0x80000000u) << 32) |
                                 ((unsigned long long)(ex + 896u) << 52) |
                                 ((unsigned long long)(u & 0x7FFFFFu) << 29);
    return __longlong_as_double((long long)b);
}

// one edge record at an atomically reserved slot (dropped past cap; the
// count still tells the host the list is incomplete)
__device__ __forceinline__ bool record_edge(const EdgeList &E, int a, int b, int e, double tau)
{
    const unsigned long long q = atomicAdd(E.count, 1ull);
    if ((long long)q >= E.cap) return false;
    {
        EdgeRec r;
        r.a = a;
        r.b = b;
        r.e = e;
        r.pad = 0;
        r.tau = tau;
        E.rec[q] = r;
    }
    return true;
}

// Kahan-compensated accumulation: s + (-c) carries the running sum
__device__ __forceinline__ void kahan_add(float &s, float &c, float x)
{
    const float y = x - c;
    const float t = s + y;
    c = (t - s) - y;
    s = t;
}

// ------------------------------------------------------------ Kepler
// Stumpff functions c2(z) = (1 - cos sqrt z)/z, c3(z) = (sqrt z - sin sqrt z)/z^{3/2}
// (hyperbolic continuation for z < 0), by their Taylor series near 0.
__device__ __forceinline__ void stumpff(double z, double &c2, double &c3)
{
    if (fabs(z) < 0.1) {
        // c2 = sum (-z)^k/(2k+2)!, c3 = sum (-z)^k/(2k+3)!
        double t2 = 0.5, t3 = 1.0 / 6.0;
        c2 = 0.0;
        c3 = 0.0;
#pragma unroll
        for (int k = 0; k < 10; ++k) {
            c2 += t2;
            c3 += t3;
            t2 *= div_const(-z, (2.0 * k + 3.0) * (2.0 * k + 4.0));
            t3 *= div_const(-z, (2.0 * k + 4.0) * (2.0 * k + 5.0));
        }
    } else if (z > 0.0) {
        const double s = sqrt(z);
        double sn, cs;
        sincos(s, &sn, &cs);
        c2 = (1.0 - cs) / z;
        c3 = (s - sn) / (z * s);
    } else {
        const double s = sqrt(-z);
        c2 = (cosh(s) - 1.0) / (-z);
        c3 = (sinh(s) - s) / (-z * s);
    }
}

// The same functions in FP32 (the starter of the iteration below), every
// operation an explicit IEEE one so that every translation unit computes
// the same starter (a contracted multiply-add would move it by an ulp, and
// the FP64 iteration's stopping point with it)
__device__ __forceinline__ void stumpff_f(float z, float &c2, float &c3)
{
    if (fabsf(z) < 0.1f) {
        float t2 = 0.5f, t3 = 1.0f / 6.0f;
        c2 = 0.0f;
        c3 = 0.0f;
        auto term = [&](float f2, float f3) {
            c2 = __fadd_rn(c2, t2);
            c3 = __fadd_rn(c3, t3);
            t2 = __fmul_rn(t2, f2);
            t3 = __fmul_rn(t3, f3);
        };
        term(div_const_f<12>(-z), div_const_f<20>(-z));
        term(div_const_f<30>(-z), div_const_f<42>(-z));
        term(div_const_f<56>(-z), div_const_f<72>(-z));
        term(div_const_f<90>(-z), div_const_f<110>(-z));
        term(div_const_f<132>(-z), div_const_f<156>(-z));
        term(0.0f, 0.0f);
    } else if (z > 0.0f) {
        const float s = __fsqrt_rn(z);
        float sn, cs;
        sincosf(s, &sn, &cs);
        c2 = __fdiv_rn(__fsub_rn(1.0f, cs), z);
        c3 = __fdiv_rn(__fsub_rn(s, sn), __fmul_rn(z, s));
    } else {
        const float s = __fsqrt_rn(-z);
        c2 = __fdiv_rn(__fsub_rn(coshf(s), 1.0f), -z);
        c3 = __fdiv_rn(__fsub_rn(sinhf(s), s), __fmul_rn(-z, s));
    }
}

// The universal Kepler equation's left side (less its t = sqrt(mu) dt); it grows
// with chi, its derivative being the separation.
__device__ __forceinline__ double kepler_eq(double chi, double alpha, double a1, double a2, double r0n, double t)
{
    const double x2 = chi * chi;
    double c2, c3;
    stumpff(alpha * x2, c2, c3);
    return a1 * x2 * c2 + a2 * x2 * chi * c3 + r0n * chi - t;
}

// Its root between two neighbouring doubles by bisection, for the orbits that the
// iteration of kepler_universal does not bring to its criterion: from a start far
// from the root near a tight pericentre (1 - e below 1e-3) it creeps, at a few
// thousandths of the way a step, and where the derivative is small it runs round a
// cycle of doubles about the root.  2.5e-7 of the solves of a cluster of binaries,
// one state of 32768 bodies in a hundred.  An equation that overflows (or is NaN)
// counts as beyond the root.
static __device__ __noinline__ bool kepler_bisect(double alpha, double a1, double a2, double r0n, double t, double &chi)
{
    const double s = t < 0.0 ? -1.0 : 1.0;
    double lo = 0.0, hi = s * fmin(fabs(t) / r0n, 1e300);
    for (int it = 0; s * kepler_eq(hi, alpha, a1, a2, r0n, t) < 0.0; ++it) {
        if (it == 2000) return false;
        lo = hi;
        hi *= 2.0;
    }
    for (int it = 0; it < 2000; ++it) {
        const double mid = lo + 0.5 * (hi - lo);
        if (mid == lo || mid == hi) break;
        if (s * kepler_eq(mid, alpha, a1, a2, r0n, t) < 0.0) lo = mid; else hi = mid;
    }
    const double fl = fabs(kepler_eq(lo, alpha, a1, a2, r0n, t)), fh = fabs(kepler_eq(hi, alpha, a1, a2, r0n, t));
    chi = fl < fh ? lo : hi;
    return isfinite(fmin(fl, fh));
}

// Advance the relative orbit (r0, v0) under mu by dt; returns false when
// the iteration does not converge.  The Laguerre-Conway iteration runs in
// FP32 first (a GB300 FP64 instruction costs the pipe ~64 cycles, an FP32
// one ~4) until its step falls to a few FP32 ulps of chi; the FP64
// iteration then converges from there in one or two steps to the same
// FP64 criterion (and starts from the usual guess if the FP32 pass did not
// settle).  A few orbits in a thousand never bring the FP32 step below that
// criterion: near a tight pericentre its rounding is larger, and the
// iteration runs round a short cycle of floats.  It is a function of one float
// alone, so the first repeated value shows the cycle, and that no step in it
// will settle: it ends there instead of after 60 steps (a warp, and a launch,
// wait for their slowest orbit).  32768 bodies, half of them in binaries: the
// Kepler launches of a step 6.6 -> 5.0 ms, the batched kernel, whose components
// run solves one after another, 46 -> 33 ms with this and the series'
// divisions (div_const), the same bits.
__device__ __forceinline__ bool kepler_universal(const double r0[3], const double v0[3], double mu, double dt, double r1[3],
                                 double v1[3])
{
    const double r0n = sqrt(r0[0] * r0[0] + r0[1] * r0[1] + r0[2] * r0[2]);
    const double v0s = v0[0] * v0[0] + v0[1] * v0[1] + v0[2] * v0[2];
    const double sig = r0[0] * v0[0] + r0[1] * v0[1] + r0[2] * v0[2];
    const double smu = sqrt(mu);
    const double alpha = 2.0 / r0n - v0s / mu;
    if (!(r0n > 0.0) || !(mu > 0.0) || !isfinite(alpha)) return false;
    // whole periods of a bound orbit are the identity: reduce dt
    if (alpha > 0.0) {
        const double P = 2.0 * CUDART_PI * sqrt(1.0 / (mu * alpha * alpha * alpha));
        if (fabs(dt) > P) dt = dt - P * trunc(dt / P);
    }
    const double a1 = sig / smu, a2 = 1.0 - alpha * r0n;
    double chi = (alpha > 0.0) ? smu * alpha * dt : smu * dt / r0n;
    if (alpha > 0.0 && fabs(alpha * r0n) < 1e-3) chi = smu * dt / r0n;
    {
        const float af = (float)alpha, a1f = (float)a1, a2f = (float)a2, r0f = (float)r0n;
        const float tf = (float)(smu * dt);
        float xf = (float)chi;
        bool ok32 = false;
        // (compared with the value kept at the last power of two: a cycle is
        // seen at the latest one turn after it is inside one)
        float kept = CUDART_NAN_F;
        for (int it = 0; it < 60; ++it) {
            const float x2 = __fmul_rn(xf, xf), z = __fmul_rn(af, x2);
            float c2f, c3f;
            stumpff_f(z, c2f, c3f);
            const float zc3 = __fsub_rn(1.0f, __fmul_rn(z, c3f)), zc2 = __fsub_rn(1.0f, __fmul_rn(z, c2f));
            const float F = __fsub_rn(__fadd_rn(__fadd_rn(__fmul_rn(__fmul_rn(a1f, x2), c2f),
                                                          __fmul_rn(__fmul_rn(__fmul_rn(a2f, x2), xf), c3f)),
                                                __fmul_rn(r0f, xf)),
                                      tf);
            const float G1 = __fadd_rn(__fadd_rn(__fmul_rn(__fmul_rn(a1f, xf), zc3), __fmul_rn(__fmul_rn(a2f, x2), c2f)),
                                       r0f);
            const float G2 = __fadd_rn(__fmul_rn(a1f, zc2), __fmul_rn(__fmul_rn(a2f, xf), zc3));
            const float disc = __fsqrt_rn(fabsf(__fsub_rn(__fmul_rn(__fmul_rn(16.0f, G1), G1),
                                                          __fmul_rn(__fmul_rn(20.0f, F), G2))));
            const float den = __fadd_rn(G1, copysignf(disc, G1));
            const float d = (den != 0.0f) ? __fdiv_rn(__fmul_rn(5.0f, F), den) : __fdiv_rn(F, G1);
            xf = __fsub_rn(xf, d);
            if (!isfinite(xf)) break;
            if (fabsf(d) <= 4e-7f * fabsf(xf)) {
                ok32 = true;
                break;
            }
            if (xf == kept) break;
            if ((it & (it + 1)) == 0) kept = xf;
        }
        if (ok32) chi = (double)xf;
    }
    double c2 = 0.5, c3 = 1.0 / 6.0, F1 = r0n;
    bool conv = false;
    long long kept64 = -1;  // (a NaN's bits; as in FP32, a repeated chi shows a cycle)
    // Laguerre-Conway iteration (order n = 5) on the universal Kepler equation
    for (int it = 0; it < 200; ++it) {
        const double x2 = chi * chi, z = alpha * x2;
        stumpff(z, c2, c3);
        const double F = a1 * x2 * c2 + a2 * x2 * chi * c3 + r0n * chi - smu * dt;
        F1 = a1 * chi * (1.0 - z * c3) + a2 * x2 * c2 + r0n;
        const double F2 = a1 * (1.0 - z * c2) + a2 * chi * (1.0 - z * c3);
        const double disc = sqrt(fabs(16.0 * F1 * F1 - 20.0 * F * F2));
        const double den = F1 + copysign(disc, F1);
        const double d = (den != 0.0) ? 5.0 * F / den : F / F1;
        chi -= d;
        if (fabs(d) <= 1e-15 * fmax(1.0, fabs(chi))) {
            conv = true;
            break;
        }
        const long long b = __double_as_longlong(chi);
        if (b == kept64) break;
        if ((it & (it + 1)) == 0) kept64 = b;
    }
    bool moved = true;
    if (!conv) {
        if (!kepler_bisect(alpha, a1, a2, r0n, smu * dt, chi)) return false;
    } else {
        // one Newton polish at the converged point
        const double x2 = chi * chi, z = alpha * x2;
        stumpff(z, c2, c3);
        const double F = a1 * x2 * c2 + a2 * x2 * chi * c3 + r0n * chi - smu * dt;
        F1 = a1 * chi * (1.0 - z * c3) + a2 * x2 * c2 + r0n;
        const double last = chi;
        chi -= F / F1;
        moved = chi != last;
    }
    const double x2 = chi * chi, z = alpha * x2;
    if (moved) stumpff(z, c2, c3);
    const double f = 1.0 - x2 * c2 / r0n;
    const double g = dt - x2 * chi * c3 / smu;
    for (int k = 0; k < 3; ++k) r1[k] = f * r0[k] + g * v0[k];
    const double r = sqrt(r1[0] * r1[0] + r1[1] * r1[1] + r1[2] * r1[2]);
    const double fd = smu / (r * r0n) * chi * (z * c3 - 1.0);
    const double gd = 1.0 - x2 * c2 / r;
    for (int k = 0; k < 3; ++k) v1[k] = fd * r0[k] + gd * v0[k];
    return isfinite(r);
}

// Two-body flow of particles a and b over dt (Eq. kepler, eps = 0): the
// centre of mass moves uniformly, the relative orbit r = x_a - x_b follows
// kepler_universal.  xa.. are updated in place; false if unconverged.
__device__ __forceinline__ bool kepler_pair(double ma, double mb, double xa[3], double xb[3], double va[3],
                                            double vb[3], double G, double dt)
{
    const double M = ma + mb;
    double r0[3], v0[3], xc[3], vc[3], r1[3], v1[3];
    for (int k = 0; k < 3; ++k) {
        xc[k] = (ma * xa[k] + mb * xb[k]) / M;
        vc[k] = (ma * va[k] + mb * vb[k]) / M;
        r0[k] = xa[k] - xb[k];
        v0[k] = va[k] - vb[k];
    }
    if (!kepler_universal(r0, v0, G * M, dt, r1, v1)) return false;
    for (int k = 0; k < 3; ++k) {
        const double xcn = xc[k] + vc[k] * dt;
        xa[k] = xcn + (mb / M) * r1[k];
        xb[k] = xcn - (ma / M) * r1[k];
        va[k] = vc[k] + (mb / M) * v1[k];
        vb[k] = vc[k] - (ma / M) * v1[k];
    }
    return true;
}

// Row ti and column offset of triangular tile t (tiles (ti, tj), tj >= ti,
// numbered row by row; row ti starts at ti nt - ti (ti - 1) / 2): the root of
// the quadratic in single precision, then exact integer corrections.
__device__ __forceinline__ int tri_tile_row(int &t, int nt)
{
    auto off = [nt](int x) { return x * nt - (x * (x - 1)) / 2; };
    const float b = 2.f * (float)nt + 1.f;
    int ti = (int)(0.5f * (b - sqrtf(fmaxf(b * b - 8.f * (float)t, 0.f))));
    ti = max(0, min(ti, nt - 1));
    while (ti > 0 && off(ti) > t) --ti;
    while (ti + 1 < nt && off(ti + 1) <= t) ++ti;
    t -= off(ti);
    return ti;
}

}  // namespace cc
