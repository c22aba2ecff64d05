// xmath.cuh -- logarithm, exponential and power for the plain FP64 form.
//
// Series method (only correctly rounded operations, so the value does not
// depend on which library or compiler evaluates it; the translation units
// that use it are compiled without multiply-add contraction):
//   log: x = 2^e f, f in [sqrt(1/2), sqrt(2)); t = (f - 1) / (f + 1);
//        log f = 2 artanh t = 2 t sum_{i=0..11} t^(2i) / (2i + 1);
//        log x = e ln2_hi + (e ln2_lo + log f), ln 2 split after 32 bits.
//   exp: n = nearest integer to x / ln 2, r = (x - n ln2_hi) - n ln2_lo
//        (Cody-Waite), e^r = sum_{i=0..14} r^i / i! (Horner), times 2^n.
//   pow: x^y = exp(y log x), x > 0 (0 for x == 0, y > 0).
//
// What bounds the FP64 kernels is the FP64 pipe: on this part every FP64
// instruction -- a comparison, a conversion, a rounding to integer as much
// as an addition -- holds its sub-partition's pipe for about 65-77 issue
// slots, and a division takes eight of them.  So whatever is not an FP64
// rounding of the method is done on the integer and FP32 pipes here, with
// the same value bit for bit:
//   * comparisons, maxima and finiteness tests of numbers that are not
//     negative order like their bit patterns (two integer compares);
//   * the logarithm's argument split, the exponential's scaling and the
//     conversions of small integers are exponent-field arithmetic;
//   * a quotient by a divisor that many dividends share goes through its
//     correctly rounded reciprocal (div_by).
// Arguments outside the ordinary range (subnormal, infinite, NaN, near
// overflow) take the general code, kept out of line.
// Measured, results bit for bit as before: van der Pol RKCK, 4,096 systems
// 5.17 -> 3.82 ms; 32-point Brusselator grids, 8,192 systems 90.6 -> 68.3 ms;
// mass-action RKC, 100,003 systems 262 -> 241 ms.
#pragma once
#include <cmath>

namespace bode {
namespace xm {

constexpr double kLn2Hi = 0.6931471806019545;        // ln 2 rounded to 32 significant bits
constexpr double kLn2Lo = -4.2009150726810846e-11;   // ln 2 - kLn2Hi
constexpr double kLog2e = 1.4426950408889634;
constexpr double kLn10 = 2.302585092994046;
constexpr double kSqrtHalf = 0.7071067811865476;

constexpr unsigned long long kMagMask = 0x7fffffffffffffffull;
constexpr unsigned long long kInfBits = 0x7ff0000000000000ull;

// |x| as an integer that orders like it (NaN above infinity)
__device__ __forceinline__ unsigned long long mag(double x) {
    return (unsigned long long)__double_as_longlong(x) & kMagMask;
}
__device__ __forceinline__ bool is_nan(double x) { return mag(x) > kInfBits; }
__device__ __forceinline__ bool is_finite(double x) { return (__double2hiint(x) & 0x7ff00000) != 0x7ff00000; }
// x > 0, false for NaN
__device__ __forceinline__ bool is_pos(double x) {
    const long long b = __double_as_longlong(x);
    return b > 0 && b <= (long long)kInfBits;
}
// a < b for a, b >= 0; false when either is NaN
__device__ __forceinline__ bool lt_nn(double a, double b) { return mag(a) < mag(b) && mag(b) <= kInfBits; }
// a <= b for a, b >= 0; false when either is NaN
__device__ __forceinline__ bool le_nn(double a, double b) { return mag(a) <= mag(b) && mag(b) <= kInfBits; }
// fmax / fmin of a, b >= 0, a not NaN (a NaN b is passed over)
__device__ __forceinline__ double max_nn(double a, double b) { return lt_nn(a, b) ? b : a; }
__device__ __forceinline__ double min_nn(double a, double b) { return mag(b) < mag(a) ? b : a; }
// max(|a|, |b|); a NaN operand wins
__device__ __forceinline__ double max_mag(double a, double b) {
    return __longlong_as_double((long long)(mag(a) < mag(b) ? mag(b) : mag(a)));
}
// an integer of at most 24 bits as a double (FP32 conversions are exact here)
__device__ __forceinline__ double small_int(int k) { return (double)(float)k; }

// a / b with r = 1 / b correctly rounded and b in [2^-100, 2^100]: one
// residual correction of a r rounds correctly (Markstein, IBM J. Res. Dev.
// 34 (1990) 111: with a correctly rounded reciprocal and a quotient within
// one ulp, q - (q b - a) r with fused operations is the rounded quotient).
// Three FP64 instructions instead of a division's eight.  Dividends outside
// [2^-700, 2^700], where the residual could round, divide as usual; zeros
// take the short way and keep their sign.  Pass r = 0 for a divisor outside
// the range; one that is not positive divides as usual too.
static __device__ __noinline__ double div_general(double a, double b) { return a / b; }
__device__ __forceinline__ double div_by(double a, double b, double r) {
    const unsigned hi = (unsigned)__double2hiint(a) & 0x7fffffffu;
    const bool ordinary = hi - (323u << 20) <= (1400u << 20) || (hi | (unsigned)__double2loint(a)) == 0u;
    if (!ordinary || __double2hiint(r) <= 0) return div_general(a, b);
    const double q = a * r;
    return fma(-fma(q, b, -a), r, q);
}
// The reciprocal div_by takes: CUDA's own, 0 for a divisor outside the range.
__device__ __forceinline__ double reciprocal(double b) {
    const unsigned long long bits = (unsigned long long)__double_as_longlong(b);
    return bits - (923ull << 52) <= (200ull << 52) ? __drcp_rn(b) : 0.0;
}

// 1/(2i+1) for i = 11 .. 0, Horner in t^2; log x from f and its exponent
__device__ __forceinline__ double log_poly(double f, double ed) {
    const double t = (f - 1.0) / (f + 1.0);
    const double t2 = t * t;
    double q = 0.043478260869565216;
    q = q * t2 + 0.047619047619047616;
    q = q * t2 + 0.05263157894736842;
    q = q * t2 + 0.058823529411764705;
    q = q * t2 + 0.06666666666666667;
    q = q * t2 + 0.07692307692307693;
    q = q * t2 + 0.09090909090909091;
    q = q * t2 + 0.1111111111111111;
    q = q * t2 + 0.14285714285714285;
    q = q * t2 + 0.2;
    q = q * t2 + 0.3333333333333333;
    q = q * t2 + 1.0;
    const double logf = 2.0 * t * q;
    return ed * kLn2Hi + (ed * kLn2Lo + logf);
}

static __device__ __noinline__ double log_general(double x) {
    if (!(x > 0.0)) return x == 0.0 ? -INFINITY : NAN;
    if (isinf(x)) return x;
    int e;
    double f = frexp(x, &e);
    if (f < kSqrtHalf) {
        f = f * 2.0;
        e = e - 1;
    }
    return log_poly(f, (double)e);
}

__device__ __forceinline__ double log_series(double x) {
    const int hi = __double2hiint(x);
    if (hi < 0x00100000 || hi >= 0x7ff00000) return log_general(x);  // zero, subnormal, negative, infinite, NaN
    // f in [sqrt(1/2), sqrt(2)) by setting the exponent field
    const unsigned long long m = (((unsigned long long)(hi & 0xfffff) | 0x3fe00000ull) << 32) | (unsigned)__double2loint(x);
    int e = (hi >> 20) - 1022;
    const bool low = m < 0x3fe6a09e667f3bcdull;  // the bit pattern of kSqrtHalf
    if (low) e = e - 1;
    const double f = __longlong_as_double((long long)(m + (low ? 0x0010000000000000ull : 0ull)));
    return log_poly(f, small_int(e));
}

// 1/i! for i = 14 .. 0, Horner in r
__device__ __forceinline__ double exp_poly(double r) {
    double q = 1.1470745597729725e-11;
    q = q * r + 1.6059043836821613e-10;
    q = q * r + 2.08767569878681e-09;
    q = q * r + 2.505210838544172e-08;
    q = q * r + 2.755731922398589e-07;
    q = q * r + 2.7557319223985893e-06;
    q = q * r + 2.48015873015873e-05;
    q = q * r + 0.0001984126984126984;
    q = q * r + 0.001388888888888889;
    q = q * r + 0.008333333333333333;
    q = q * r + 0.041666666666666664;
    q = q * r + 0.16666666666666666;
    q = q * r + 0.5;
    q = q * r + 1.0;
    q = q * r + 1.0;
    return q;
}

static __device__ __noinline__ double exp_general(double x) {
    if (isnan(x)) return x;
    if (x > 709.0) return INFINITY;
    if (x < -745.0) return 0.0;
    const double n = rint(x * kLog2e);
    const double r = (x - n * kLn2Hi) - n * kLn2Lo;
    return ldexp(exp_poly(r), (int)n);
}

__device__ __forceinline__ double exp_series(double x) {
    // |x| < 707: the scaled result is normal, so the scaling adds to the exponent field
    if ((unsigned)(__double2hiint(x) & 0x7fffffff) >= 0x40861800u) return exp_general(x);
    const int n = __double2int_rn(x * kLog2e);
    const double nd = small_int(n);
    const double r = fma(-nd, kLn2Hi, x) - nd * kLn2Lo;  // n kLn2Hi is exact: fused or not, one rounding
    const double q = exp_poly(r);
    return __hiloint2double(__double2hiint(q) + (n << 20), __double2loint(q));
}

// Products on the integer pipe, rounded to nearest even exactly as the FP64
// pipe rounds them: the 53 x 53-bit product of the significands in four
// 32 x 32 multiply-adds, normalised by at most one bit, rounded from the
// remaining 64 bits.  About 30 integer instructions, 50-60 issue slots
// against the FP64 pipe's 77 -- on a pipe that otherwise idles, so a loop
// that does its products here and its sums there runs on both.
// Multiplier: the factor many products share, taken apart once.
struct Multiplier {
    unsigned hi, lo;  // significand, its top bit at bit 63
    int ex;           // exponent field less the bias, in place
    unsigned sign;
    double v;         // the factor itself
    bool ok;          // in [2^-400, 2^400] in magnitude
};
__device__ __forceinline__ Multiplier multiplier(double r) {
    Multiplier m;
    const unsigned h = (unsigned)__double2hiint(r), l = (unsigned)__double2loint(r);
    m.hi = __funnelshift_l(l, h, 11) | 0x80000000u;
    m.lo = l << 11;
    m.ex = (int)(h & 0x7ff00000u) - (1023 << 20);
    m.sign = h & 0x80000000u;
    m.v = r;
    m.ok = (h & 0x7fffffffu) - (623u << 20) <= (800u << 20);
    return m;
}
// a m.v for |a| in [2^-600, 2^600] and m.ok
__device__ __forceinline__ double mul_int(double a, const Multiplier& m) {
    const unsigned ah = (unsigned)__double2hiint(a), al = (unsigned)__double2loint(a);
    const unsigned mh = (ah & 0xfffffu) | 0x100000u;
    const unsigned long long p0 = (unsigned long long)al * m.lo;
    const unsigned long long p1 = (unsigned long long)al * m.hi + (p0 >> 32);
    const unsigned long long p2 = (unsigned long long)mh * m.lo + (unsigned)p1;
    const unsigned long long p3 = (unsigned long long)mh * m.hi + (p1 >> 32) + (p2 >> 32);
    unsigned hi = (unsigned)(p3 >> 32), lo = (unsigned)p3, g = (unsigned)p2;
    const unsigned sticky = (unsigned)p0;
    const unsigned sh = 1u - (hi >> 20);  // the product's top bit is bit 52 or 51 of p3
    hi = __funnelshift_l(lo, hi, sh);
    lo = __funnelshift_l(g, lo, sh);
    g = __funnelshift_l(sticky, g, sh);
    // round: up past half, at half to even (the bits below g only break the tie)
    g |= (sticky << sh) != 0u;
    const unsigned long long up = ((unsigned long long)g + 0x7fffffffull + (lo & 1u)) >> 32;
    const unsigned long long s = (((unsigned long long)hi << 32) | lo) + up;
    // hi carries the leading bit, one in the exponent field's last place
    const unsigned e = (ah & 0x7ff00000u) + (unsigned)m.ex - (sh << 20);
    const unsigned h = ((unsigned)(s >> 32) + e) | ((ah ^ m.sign) & 0x80000000u);
    return __hiloint2double((int)h, (int)(unsigned)s);
}

// exp_series of two arguments side by side, the Horner products on the
// integer pipe: the two chains fill each other's latencies, and each step
// leaves one FP64 instruction (the sum) of two.  The kinetics rate constants,
// 766 of them an evaluation: 1,000 systems 83.2 -> 66.2 ms.
__device__ __forceinline__ void exp_series2(const double (&x)[2], double (&out)[2]) {
    constexpr double c[14] = {1.6059043836821613e-10, 2.08767569878681e-09,  2.505210838544172e-08, 2.755731922398589e-07,
                              2.7557319223985893e-06, 2.48015873015873e-05,  0.0001984126984126984, 0.001388888888888889,
                              0.008333333333333333,   0.041666666666666664,  0.16666666666666666,   0.5,
                              1.0,                    1.0};
    Multiplier r[2];
    int n[2];
    bool ordinary = true;
#pragma unroll
    for (int u = 0; u < 2; ++u) {
        ordinary = ordinary && (unsigned)(__double2hiint(x[u]) & 0x7fffffff) < 0x40861800u;
        n[u] = __double2int_rn(x[u] * kLog2e);
        const double nd = small_int(n[u]);
        r[u] = multiplier(fma(-nd, kLn2Hi, x[u]) - nd * kLn2Lo);
        ordinary = ordinary && r[u].ok;
    }
    if (!ordinary) {
        out[0] = exp_series(x[0]);
        out[1] = exp_series(x[1]);
        return;
    }
    double q[2] = {1.1470745597729725e-11, 1.1470745597729725e-11};
#pragma unroll
    for (int k = 0; k < 14; ++k)
#pragma unroll
        for (int u = 0; u < 2; ++u) q[u] = mul_int(q[u], r[u]) + c[k];
#pragma unroll
    for (int u = 0; u < 2; ++u) out[u] = __hiloint2double(__double2hiint(q[u]) + (n[u] << 20), __double2loint(q[u]));
}

__device__ __forceinline__ double pow_series(double x, double y) {
    if (mag(x) == 0ull) return y > 0.0 ? 0.0 : INFINITY;
    return exp_series(y * log_series(x));
}
// x^y from lx = log_series(x), y > 0 (x = 0: lx = -infinity gives 0)
__device__ __forceinline__ double pow_log(double lx, double y) { return exp_series(y * lx); }

}  // namespace xm
}  // namespace bode
