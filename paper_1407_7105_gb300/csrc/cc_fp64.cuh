// cc_fp64.cuh -- correctly rounded FP64 products and r^-3 off the FP64 pipe.
//
// A GB300 SM issues one FP64 warp instruction per scheduler every 64 cycles
// and leaves its integer and FP32 pipes idle meanwhile.  The pair forces of
// the FP64 form are bound by exactly that, so their multiplications and the
// reciprocal cube of the distance are computed here with 32-bit integer
// products and FP32 approximations, to the same bits as the IEEE operations
// (round to nearest, ties to even):
//   mul_rn, sqr_rn : a b and a a by 32 x 32 -> 64-bit products of the
//                    significands;
//   rinv3_rn       : rn(1 / rn(x rn(sqrt x))), each of the two roundings by
//                    an FP32 estimate good to ~2^-45, one exact FP64 residual
//                    (a fused multiply-add, as in Markstein's proofs for
//                    division and square root by Newton steps), the
//                    correction in units of the last place, and an integer
//                    rounding of it; a correction too close to a tie for its
//                    error is reported, and the caller takes the IEEE path;
//   rsqrt_near     : x^-1/2 to 0.51 units of the last place by the same steps,
//                    for sums that ask for no particular bits.
// The callers see to the ranges (fast_range): no operand or result is
// subnormal, infinite or NaN here; zero operands of mul_rn and sqr_rn are.
// The header compiles for the host too, where the tests compare every
// function with the machine's own arithmetic.
#pragma once
#include <stdint.h>
#ifdef __CUDACC__
#define CC_HD __host__ __device__ __forceinline__
#else
#define CC_HD inline
#endif
#ifndef __CUDA_ARCH__
#include <cmath>
#include <cstring>
#endif

namespace cc {

#ifdef __CUDA_ARCH__
CC_HD uint64_t d2u(double x) { return (uint64_t)__double_as_longlong(x); }
CC_HD double u2d(uint64_t b) { return __longlong_as_double((long long)b); }
CC_HD uint32_t f2u(float x) { return __float_as_uint(x); }
CC_HD float u2f(uint32_t b) { return __uint_as_float(b); }
CC_HD float rsqrt_est(float x)
{
    float y;
    asm("rsqrt.approx.ftz.f32 %0, %1;" : "=f"(y) : "f"(x));
    return y;
}
CC_HD float rcp_est(float x)
{
    float y;
    asm("rcp.approx.ftz.f32 %0, %1;" : "=f"(y) : "f"(x));
    return y;
}
CC_HD int32_t rint_i(float x) { return __float2int_rn(x); }
CC_HD float fma_f(float a, float b, float c) { return fmaf(a, b, c); }
CC_HD double fma_d(double a, double b, double c) { return __fma_rn(a, b, c); }
CC_HD uint32_t shl_f(uint32_t hi, uint32_t lo, uint32_t s) { return __funnelshift_l(lo, hi, s); }
#else
template <class A, class B>
inline A bits_as(B b)
{
    A a;
    static_assert(sizeof(A) == sizeof(B), "bits");
    std::memcpy(&a, &b, sizeof a);
    return a;
}
inline uint64_t d2u(double x) { return bits_as<uint64_t>(x); }
inline double u2d(uint64_t b) { return bits_as<double>(b); }
inline uint32_t f2u(float x) { return bits_as<uint32_t>(x); }
inline float u2f(uint32_t b) { return bits_as<float>(b); }
// (the tests move the estimates by the hardware's error bounds, 2^-22.9 and 2^-23)
extern float est_shift;
inline float rsqrt_est(float x) { return (1.0f / std::sqrt(x)) * (1.0f + est_shift); }
inline float rcp_est(float x) { return (1.0f / x) * (1.0f + est_shift); }
inline int32_t rint_i(float x) { return (int32_t)std::lrintf(x); }
inline float fma_f(float a, float b, float c) { return std::fma(a, b, c); }
inline double fma_d(double a, double b, double c) { return std::fma(a, b, c); }
inline uint32_t shl_f(uint32_t hi, uint32_t lo, uint32_t s) { return (uint32_t)(((((uint64_t)hi << 32) | lo) << s) >> 32); }
#endif

// The rounded product from the significands' exact product p3 2^64 + t 2^32 +
// z (p3 in [2^40, 2^42)) and the exponent fields' sum (in the high words'
// place, biased twice): 53 bits kept, the rest rounded by a carry.
CC_HD uint64_t mul_round(uint64_t p3, uint32_t t, uint32_t z, uint32_t ex)
{
    const uint32_t h = (uint32_t)(p3 >> 32), l = (uint32_t)p3, big = h >> 9, s = 12u - big;
    const uint32_t mh = shl_f(h, l, s), ml = shl_f(l, t, s);
    const uint32_t rem = (t << s) | (z != 0u ? 1u : 0u);  // sticky
    const uint64_t up = ((uint64_t)rem + 0x7fffffffu + (ml & 1u)) >> 32;
    // (the significand's leading bit, and a carry out of it, step the exponent)
    return (((uint64_t)(mh + ex - (1024u << 20) + (big << 20)) << 32) | ml) + up;
}

CC_HD uint64_t mul_rn(uint64_t a, uint64_t b)
{
    const uint32_t a1 = (uint32_t)(a >> 32), b1 = (uint32_t)(b >> 32);
    const uint32_t ah = (a1 & 0xfffffu) | 0x100000u, al = (uint32_t)a;
    const uint32_t bh = (b1 & 0xfffffu) | 0x100000u, bl = (uint32_t)b;
    const uint64_t p0 = (uint64_t)al * bl;
    const uint64_t p1 = (uint64_t)ah * bl + (p0 >> 32);
    const uint64_t p2 = (uint64_t)al * bh + (uint32_t)p1;
    const uint64_t p3 = (uint64_t)ah * bh + (p1 >> 32) + (p2 >> 32);
    const uint32_t ea = a1 & 0x7ff00000u, eb = b1 & 0x7ff00000u;
    const uint64_t r = mul_round(p3, (uint32_t)p2, (uint32_t)p0, ea + eb);
    const uint64_t sign = (uint64_t)((a1 ^ b1) & 0x80000000u) << 32;
    return (ea == 0u || eb == 0u ? 0ull : r) | sign;
}

CC_HD uint64_t sqr_rn(uint64_t a)
{
    const uint32_t a1 = (uint32_t)(a >> 32);
    const uint32_t ah = (a1 & 0xfffffu) | 0x100000u, al = (uint32_t)a;
    const uint64_t p0 = (uint64_t)al * al;
    const uint64_t c = (((uint64_t)ah * al) << 1) + (p0 >> 32);
    const uint64_t p3 = (uint64_t)ah * ah + (c >> 32);
    const uint32_t ea = a1 & 0x7ff00000u;
    const uint64_t r = mul_round(p3, (uint32_t)c, (uint32_t)p0, 2u * ea);
    return ea == 0u ? 0ull : r;
}

// exponent field within 2^-200 .. 2^200 (what fast_range asks of a nonzero value)
CC_HD bool exp_fast(uint64_t x)
{
    return ((uint32_t)(x >> 52) & 0x7ffu) - 823u <= 400u;
}
// a difference the functions here may take: zero, or within 2^-200 .. 2^200
// (asked of the two words apart: a test of the whole would be turned into an
// FP64 comparison)
CC_HD bool fast_range(uint64_t x)
{
    return exp_fast(x) || (((uint32_t)(x >> 32) & 0x7fffffffu) | (uint32_t)x) == 0u;
}

// the low 29 bits of a significand in units of 2^-46 (times 2^p), as a float
CC_HD float low_part(uint32_t lo, uint32_t p)
{
    const uint32_t base = (104u + p) << 23;
    return u2f(base | ((lo & 0x1fffffffu) >> 6)) - u2f(base);
}

// a float estimate of a residual's value, truncated; exponent in the float
// range, or zero (seen in the high word: a residual here is above 2^-200)
CC_HD float trunc_f(uint64_t x)
{
    const uint32_t h = (uint32_t)(x >> 32);
    const uint32_t m = (((h & 0x7fffffffu) - (896u << 20)) << 3) | ((uint32_t)x >> 29);
    return u2f((h & 0x7fffffffu) == 0u ? 0u : m | (h & 0x80000000u));
}

// nearest integer to |c| < 2^21 and whether c is within 2^-13 of a tie (its
// error bound below is 2^-14)
CC_HD int32_t round_units(float c, bool &open)
{
    const float t = c + 12582912.0f;
    const float fr = c - (t - 12582912.0f);
    open = open || !((fr < 0.0f ? -fr : fr) <= 0.5f - 1.220703125e-4f);
    return (int32_t)(f2u(t) - 0x4b400000u);
}

// rn(1 / rn(x rn(sqrt x))) for x > 0 with exp_fast(x); open: a rounding was
// too close to call, the result is not to be used.
CC_HD uint64_t rinv3_rn(uint64_t x, bool &open)
{
    const uint32_t h = (uint32_t)(x >> 32), lo = (uint32_t)x;
    const int32_t E = (int32_t)(h >> 20) - 1023;
    const uint32_t p = (uint32_t)E & 1u;
    // x = m 2^(2k), m = m_h + m_l in [1, 4)
    const uint64_t m = ((uint64_t)((h & 0xfffffu) | ((1023u + p) << 20)) << 32) | lo;
    const float mh = u2f(((h & 0xfffffu) << 3 | lo >> 29) + ((127u + p) << 23)), ml = low_part(lo, p);
    // y = m^-1/2 to 2^-23.5, then S0 = sqrt(m) to 2^-45 from the FP32 residual
    const float y0 = rsqrt_est(mh);
    const float y = fma_f(y0, fma_f(-(mh * y0), 0.5f * y0, 0.5f), y0);
    const float t = mh * y, sh = t > 1.0f ? t : 1.0f;
    const float sl = (fma_f(-sh, sh, mh) + ml) * (0.5f * y);
    const uint64_t S0 = 0x3ff0000000000000ull + ((uint64_t)(f2u(sh) - 0x3f800000u) << 29) +
                        (uint64_t)(int64_t)rint_i(sl * 4503599627370496.0f);
    // sqrt(m) - S0 = (m - S0^2) / (2 S0) in units of 2^-52
    const double s0 = u2d(S0);
    const float es = trunc_f(d2u(fma_d(-s0, s0, u2d(m))));
    const uint64_t S = S0 + (uint64_t)(int64_t)round_units(es * (y * 2251799813685248.0f), open);
    // C = rn(m S) = C' 2^f, 1/C' by the same steps
    const uint64_t C = mul_rn(m, S);
    const uint32_t ch = (uint32_t)(C >> 32), cl = (uint32_t)C;
    const int32_t f = (int32_t)(ch >> 20) - 1023;
    const uint64_t C1 = ((uint64_t)((ch & 0xfffffu) | 0x3ff00000u) << 32) | cl;
    const float gh = u2f(((ch & 0xfffffu) << 3 | cl >> 29) + (127u << 23)), gl = low_part(cl, 0u);
    float qh = rcp_est(gh);
    qh = qh < 0.5f ? 0.5f : (qh > 0.99999994f ? 0.99999994f : qh);
    const float e = fma_f(-gl, qh, fma_f(-gh, qh, 1.0f));
    const float ql = qh * fma_f(e, e, e);
    const uint64_t Q0 = 0x3fe0000000000000ull + ((uint64_t)(f2u(qh) - 0x3f000000u) << 29) +
                        (uint64_t)((int64_t)rint_i(ql * 4503599627370496.0f) * 2);
    const float eq = trunc_f(d2u(fma_d(-u2d(C1), u2d(Q0), 1.0)));
    const uint64_t Q = Q0 + (uint64_t)(int64_t)round_units(eq * (qh * 9007199254740992.0f), open);
    // x = m 2^(2k): C 2^(3k), so the result is Q 2^-(f + 3k)
    const int32_t k = (E - (int32_t)p) >> 1;
    return Q - ((uint64_t)(int64_t)(f + 3 * k) << 52);
}

// a b for positive normal operands, cut off after 53 bits; rem = the next 32
CC_HD uint64_t mul_cut(uint64_t a, uint64_t b, uint32_t &rem)
{
    const uint32_t a1 = (uint32_t)(a >> 32), b1 = (uint32_t)(b >> 32);
    const uint32_t ah = (a1 & 0xfffffu) | 0x100000u, al = (uint32_t)a;
    const uint32_t bh = (b1 & 0xfffffu) | 0x100000u, bl = (uint32_t)b;
    const uint64_t p1 = (uint64_t)ah * bl + (((uint64_t)al * bl) >> 32);
    const uint64_t p2 = (uint64_t)al * bh + (uint32_t)p1;
    const uint64_t p3 = (uint64_t)ah * bh + (p1 >> 32) + (p2 >> 32);
    const uint32_t h = (uint32_t)(p3 >> 32), l = (uint32_t)p3, t = (uint32_t)p2, big = h >> 9, s = 12u - big;
    rem = t << s;
    const uint32_t ex = (a1 & 0x7ff00000u) + (b1 & 0x7ff00000u) - (1024u << 20) + (big << 20);
    return ((uint64_t)(shl_f(h, l, s) + ex) << 32) | shl_f(l, t, s);
}

// x^-1/2 for x > 0 with exp_fast(x), within 0.51 ulp
CC_HD uint64_t rsqrt_near(uint64_t x)
{
    const uint32_t h = (uint32_t)(x >> 32), lo = (uint32_t)x;
    const int32_t E = (int32_t)(h >> 20) - 1023;
    const uint32_t p = (uint32_t)E & 1u;
    const uint64_t m = ((uint64_t)((h & 0xfffffu) | ((1023u + p) << 20)) << 32) | lo;  // [1, 4)
    const float mh = u2f(((h & 0xfffffu) << 3 | lo >> 29) + ((127u + p) << 23)), ml = low_part(lo, p);
    // y to 2^-22 in [1/2, 1), its FP32 residual e = 1 - m y^2, Z0 to 2^-44
    float y = rsqrt_est(mh);
    y = y < 0.5f ? 0.5f : (y > 0.99999994f ? 0.99999994f : y);
    const float t = mh * y, tl = fma_f(mh, y, -t) + ml * y;
    const float e = fma_f(-tl, y, fma_f(-t, y, 1.0f));
    const float zl = y * e * fma_f(0.375f, e, 0.5f);
    const uint64_t Z0 = 0x3fe0000000000000ull + ((uint64_t)(f2u(y) - 0x3f000000u) << 29) +
                        (uint64_t)((int64_t)rint_i(zl * 4503599627370496.0f) * 2);
    // the residual 1 - m Z0^2 (the product's first 53 bits by an FP64
    // instruction, the rest of it in FP32), its correction in units of 2^-53
    const double z0 = u2d(Z0);
    uint32_t rem;
    const uint64_t u = mul_cut(m, Z0, rem);
    // (2^-84 times the product's exponent: rem counts 2^-32 of its last place)
    const float ul = (float)rem * u2f((uint32_t)((u >> 52) - 1023u + 43u) << 23);
    const float r = trunc_f(d2u(fma_d(-u2d(u), z0, 1.0))) - ul * y;
    const uint64_t Z = Z0 + (uint64_t)(int64_t)rint_i(r * (y * 4503599627370496.0f));
    return Z - ((uint64_t)(int64_t)((E - (int32_t)p) >> 1) << 52);
}

// x / C for a small whole constant, the division's bits in three operations:
// quotient by the rounded reciprocal, exact residual, correction (Markstein's
// theorem for a correctly rounded reciprocal; C's significand is not all ones)
// Explicit operations: what the compiler contracts around them stays as it is.
CC_HD double div_const(double x, double c)
{
#ifdef __CUDA_ARCH__
    const double y = 1.0 / c, q = __dmul_rn(x, y);
#else
    const double y = 1.0 / c, q = x * y;
#endif
    return fma_d(fma_d(-q, c, x), y, q);
}
template <int C>
CC_HD float div_const_f(float x)
{
    constexpr float y = 1.0f / C;
    const float q = x * y;
    return fma_f(fma_f(-q, (float)C, x), y, q);
}

#ifdef __CUDACC__
// a + b as a fused multiply-add with a one that the compiler cannot see: the
// same bits (a times one is exact), and a DFMA holds the pipe 64 cycles a warp
// where a DADD or DMUL holds it 77 (each measured alone on it; a product is
// __fma_rn with a minus zero, whose sum keeps every value and sign)
__device__ __forceinline__ double add_fma(double a, double b, double one) { return __fma_rn(a, one, b); }

// rn(1 / rn(r2 rn(sqrt r2))) by the IEEE instructions: what rinv3_rn is, and
// the way out where it does not apply
static __device__ __noinline__ double rinv3_ieee(double r2) { return __drcp_rn(__dmul_rn(r2, __dsqrt_rn(r2))); }

// r^-3 of a pair's difference (the squares summed in order, softened): the
// kick's operations, with the products and r^-3 off the FP64 pipe where their
// ranges allow.  Returns false when the force's products have to be IEEE ones.
__device__ __forceinline__ bool pair_rinv3(double dx0, double dx1, double dx2, double eps2, bool soft, double one,
                                           double &v)
{
    const uint64_t d0 = d2u(dx0), d1 = d2u(dx1), d2 = d2u(dx2);
    bool fast = fast_range(d0) && fast_range(d1) && fast_range(d2);
    if (fast) {
        double r2 = add_fma(add_fma(u2d(sqr_rn(d0)), u2d(sqr_rn(d1)), one), u2d(sqr_rn(d2)), one);
        if (soft) r2 = add_fma(r2, eps2, one);
        bool open = !exp_fast(d2u(r2));
        v = u2d(rinv3_rn(d2u(r2), open));
        if (open) {
            v = rinv3_ieee(r2);
            fast = exp_fast(d2u(r2));
        }
    } else {
        v = rinv3_ieee(
            __dadd_rn(__dadd_rn(__dadd_rn(__dmul_rn(dx0, dx0), __dmul_rn(dx1, dx1)), __dmul_rn(dx2, dx2)), eps2));
    }
    return fast;
}

#endif

}  // namespace cc
