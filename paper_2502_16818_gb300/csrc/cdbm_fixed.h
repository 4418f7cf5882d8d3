// 64-bit block fixed-point arithmetic for sums that need not round as FP64 does: the raw
// moments of Delta* and the group sums of single-precision values.
//
// On GB300 one FP64 instruction occupies its pipe for 64 cycles per SM sub-partition
// (2 lanes/clk/SM, measured), a 32-bit integer instruction for 1 to 2.  So the doubles of a
// sum are brought to the largest exponent among them as 64-bit integers, added and
// multiplied exactly or to a few units of 2^-58 of that largest value, and the result
// is rounded to double once.  The FP64 form rounds after every operation, at 2^-53 of
// the intermediate value.
//
// A fixed-point value v of top exponent E (the biased exponent field of the largest
// double of the sum) stands for v 2^(E - 1023 - kLead): a double with exponent E has
// its leading one at bit kLead.  Three bits above are headroom for operands that may
// exceed E (fx_clamped) and for sums.  A double whose exponent lies at most 6 below E
// converts exactly, a smaller one is rounded at 2^-kLead of the largest.  Every
// shortening rounds to nearest: a truncation would bias each of the tens of thousands
// of updates of a run the same way.
//
// The same source compiles for the host, where a test compares it with exact
// rational arithmetic.
#pragma once

#include <cmath>
#include <cstdint>

#include "cdbm_convert.h"

#if defined(__CUDACC__)
#define CDBM_FX_HD __host__ __device__ __forceinline__
#else
#define CDBM_FX_HD inline
#endif

namespace cdbm {

constexpr int kLead = 58;                     // bit of the leading one at the top exponent
constexpr int kExpLo = 128, kExpSpan = 1800;  // top exponents the integer path handles

CDBM_FX_HD int fx_clz32(uint32_t v)
{
#if defined(__CUDA_ARCH__)
    return __clz((int)v);
#else
    return v ? __builtin_clz(v) : 32;
#endif
}

CDBM_FX_HD double fx_bits(uint32_t hi, uint32_t lo)
{
#if defined(__CUDA_ARCH__)
    return __hiloint2double((int)hi, (int)lo);
#else
    const uint64_t b = (uint64_t)hi << 32 | lo;
    double v;
    std::memcpy(&v, &b, sizeof v);
    return v;
#endif
}

// Magnitude key: orders like |v| up to the low word; key >> 21 is the exponent field.
CDBM_FX_HD uint32_t fx_key(double v) { return f64_hi(v) << 1; }
CDBM_FX_HD uint32_t fx_max(uint32_t a, uint32_t b) { return a > b ? a : b; }
CDBM_FX_HD int fx_imin(int a, int b) { return a < b ? a : b; }
CDBM_FX_HD int fx_imax(int a, int b) { return a > b ? a : b; }

// v at top exponent E, rounded to the nearest unit, with the leading one of a value of
// exponent E at bit kAt; v's exponent is at most E (kClamp: may be larger, values of
// exponent E + 3 and more keep their sign and mantissa at exponent E + 3).
template <bool kClamp, int kAt>
CDBM_FX_HD int64_t fx_from_t(double v, int E)
{
    const uint32_t hi = f64_hi(v), lo = f64_lo(v);
    int sh = E + (61 - kAt) - (int)((hi << 1) >> 21);
    if (kClamp) sh = fx_imax(sh, 0);
    sh = fx_imin(sh, 63);
    const uint32_t mh = (hi & 0xfffffu) | 0x100000u;
    const uint64_t m = (((uint64_t)mh << 32) | lo) << 10;     // leading one at bit 62
    const int64_t w = (int64_t)(m >> sh);                     // in half units
    const int64_t s = (int64_t)((int32_t)hi >> 31);
    return ((w ^ s) + (1 - s)) >> 1;
}
CDBM_FX_HD int64_t fx_from(double v, int E) { return fx_from_t<false, kLead>(v, E); }
CDBM_FX_HD int64_t fx_clamped(double v, int E) { return fx_from_t<true, kLead>(v, E); }

// Single-precision values: key >> 24 is their exponent field; v, whose exponent is at
// most E, with the leading one of a value of exponent E at bit kLead, rounded to the
// nearest unit (exact up to 34 binades below; subnormals count as zero).  It stands for
// v 2^(E - 127 - kLead).
CDBM_FX_HD uint32_t fx_key(float v) { return f32_bits(v) << 1; }
CDBM_FX_HD int64_t fx_from(float v, int E)
{
    const uint32_t b = f32_bits(v);
    const int e = (int)((b << 1) >> 24);
    const uint32_t m = e ? (b & 0x7fffffu) | 0x800000u : 0u;
    const int64_t w = (int64_t)(((uint64_t)m << 39) >> fx_imin(E + 3 - e, 63));   // in half units
    const int64_t s = (int64_t)((int32_t)b >> 31);
    return ((w ^ s) + (1 - s)) >> 1;
}

// v 2^(E - 1023 - kLead) rounded to double, to nearest, ties to even.  |v| < 2^63.
CDBM_FX_HD double fx_to(int64_t v, int E)
{
    const int64_t s = v >> 63;
    const uint64_t m = (uint64_t)((v ^ s) - s);
    const uint32_t mh = (uint32_t)(m >> 32);
    int n = fx_clz32(mh);                                     // >= 1
    if (mh == 0) {
        if ((uint32_t)m == 0) return 0.0;
        n = 32 + fx_clz32((uint32_t)m);
    }
    const uint64_t ms = m << (n - 1);                         // leading one at bit 62
    const uint64_t q = (ms + 0x1ff + ((ms >> 10) & 1)) >> 10;
    const uint32_t hi = (uint32_t)(q >> 32) + ((uint32_t)(E - kLead + 62 - n) << 20);
    return fx_bits(hi | ((uint32_t)(s >> 32) & 0x80000000u), (uint32_t)q);
}

// A constant of the run as hi 2^32 + lo (lo signed).
struct FxC {
    int32_t hi, lo;
};

// A constant of the run as b1 2^30 + b0 in units of 2^-59; b0x4 = 4 b0.
struct FxK {
    int32_t b1, b0, b0x4;
};

// Sum of products x b, all four partial products kept.  No partial sum overflows for the
// moments: the four |x| add up to less than 2^63, |b| <= 1 in 2^-59.
struct FxSum {
    int64_t r, mid, low;
};
CDBM_FX_HD void fx_mul(FxSum &a, int64_t x, FxK b)
{
    const int32_t x0 = (int32_t)x;
    const int32_t x1 = (int32_t)(x >> 32) + (int32_t)((uint32_t)x0 >> 31);
    a.r += (int64_t)x1 * b.b1;
    a.mid += (int64_t)x1 * b.b0x4;
    a.mid += (int64_t)x0 * b.b1;
    a.low += (int64_t)x0 * b.b0;
}
// The sum in the units of x, rounded to nearest, for constants in units of 2^-59, of an
// FxSum that starts from kFxHalfUnit.
constexpr FxSum kFxHalfUnit = {0, 1 << 28, 0};
CDBM_FX_HD int64_t fx_sum59(const FxSum &a)
{
    return (int64_t)((uint64_t)a.r << 3) + ((a.mid + (a.low >> 30)) >> 29);
}
inline FxC fx_split(int64_t b)
{
    FxC c;
    c.lo = (int32_t)(uint32_t)b;
    c.hi = (int32_t)((b >> 32) + (c.lo < 0));
    return c;
}
inline int64_t fx_int(FxC c) { return ((int64_t)c.hi << 32) + c.lo; }
// v 2^bits (|v| <= 2) as a constant.
inline FxC fx_const(double v, int bits) { return fx_split(std::llrint(std::ldexp(v, bits))); }

inline FxK fx_k(FxC a)
{
    const int64_t b = fx_int(a) / 2;                           // in twice the unit of a
    FxK k;
    k.b1 = (int32_t)((b + (1 << 29)) >> 30);
    k.b0 = (int32_t)(b - ((int64_t)k.b1 << 30));
    k.b0x4 = 4 * k.b0;
    return k;
}

// Exponent of the smallest power of two that is at least the largest of v[0..n-1].
inline int fx_exponent(const double *v, int n)
{
    double m = 0.0;
    for (int k = 0; k < n; ++k) m = v[k] > m ? v[k] : m;
    int e = 0;
    const double f = std::frexp(m, &e);
    return f == 0.5 ? e - 1 : e;
}

// ---- The update of a Runge-Kutta stage ----
// No kernel takes it: it is about as exact as FP64 arithmetic but rounds otherwise, and the
// time step amplifies that (cdbm_exact.h).  Kept under its host check.

// Sum of products x b: r holds the high parts, mid the cross terms and the rounded high
// word of the products of the two low halves.
struct FxAcc {
    int64_t r, mid;
};
CDBM_FX_HD void fx_mac(FxAcc &a, int64_t x, FxC b)
{
    const int32_t x0 = (int32_t)x;
    const int32_t x1 = (int32_t)(x >> 32) + (int32_t)((uint32_t)x0 >> 31);   // x = x1 2^32 + x0
    a.r += (int64_t)x1 * b.hi;
    a.mid += (int64_t)x1 * b.lo;
    a.mid += (int64_t)x0 * b.hi;
    a.mid += ((int64_t)x0 * b.lo + 0x80000000ll) >> 32;
}
// The sum in the units of x, rounded to nearest, for constants scaled by 2^kBits.
template <int kBits>
CDBM_FX_HD int64_t fx_sum(const FxAcc &a)
{
    return (int64_t)((uint64_t)a.r << (64 - kBits)) + ((a.mid + ((int64_t)1 << (kBits - 33))) >> (kBits - 32));
}

CDBM_FX_HD int64_t fx_min64(int64_t a, int64_t b) { return a < b ? a : b; }
CDBM_FX_HD int64_t fx_max64(int64_t a, int64_t b) { return a > b ? a : b; }

// Twice the NND transport difference of Eqs. (12)-(20) in upwind order (nnd()), on
// fixed-point operands: 2 a + minmod(b, a) - minmod(a, e) with a = c - u1, b = d1 - c,
// e = u1 - u2.  minmod(b, a) is b clamped to the interval between 0 and a.
CDBM_FX_HD int64_t fx_nnd2(int64_t u2, int64_t u1, int64_t c, int64_t d1)
{
    const int64_t a = (int64_t)((uint64_t)c - (uint64_t)u1), b = (int64_t)((uint64_t)d1 - (uint64_t)c),
                  e = (int64_t)((uint64_t)u1 - (uint64_t)u2);
    const int64_t s = a >> 63;
    const int64_t lo = a & s, hi = a & ~s;
    return a + a + fx_max64(fx_min64(b, hi), lo) - fx_max64(fx_min64(e, hi), lo);
}

// The bits of v as an integer: for doubles of one sign and exponent, differences of
// these are the differences of the magnitudes in units in the last place.
CDBM_FX_HD int64_t fx_raw(double v) { return (int64_t)((uint64_t)f64_hi(v) << 32 | f64_lo(v)); }

// fx_mul() with a constant as hi 2^32 + lo: the sum is r 2^64 + mid 2^32 + low, so that the
// shift by 64 that the scale of the operands is chosen for below costs nothing.  Two products at most, lo of
// one of the constants above -2^31.
CDBM_FX_HD void fx_mul(FxSum &a, int64_t x, FxC b)
{
    const int32_t x0 = (int32_t)x;
    const int32_t x1 = (int32_t)(x >> 32) + (int32_t)((uint32_t)x0 >> 31);
    a.r += (int64_t)x1 * b.hi;
    a.mid += (int64_t)x1 * b.lo;
    a.mid += (int64_t)x0 * b.hi;
    a.low += (int64_t)x0 * b.lo;
}
// The sum in 1/64 of the units of y, rounded to nearest, of an FxSum that starts from
// kFxHalf and takes x = y 2^9 with constants in units of 2^-61 (|y| < 2^53; relaxation
// |b| <= 2, base |b| <= 1/2).
constexpr int kFxUp = 9;
constexpr FxSum kFxHalf = {0, (int64_t)1 << 31, 0};
CDBM_FX_HD int64_t fx_sum64ths(const FxSum &a) { return a.r + ((a.mid + (a.low >> 32)) >> 32); }
// 64ths rounded to the nearest unit so that C plus the result is even on a tie.
CDBM_FX_HD int64_t fx_round64ths(int64_t t, int64_t C) { return (t + 31 + (((t >> 6) ^ C) & 1)) >> 6; }
// The sum rounded to the nearest unit of x, a tie toward zero, for constants in units of
// 2^-64 (-1/2 <= b <= 0; two that add up to less than -1/2 by rounding only).
CDBM_FX_HD int64_t fx_sum_units(const FxSum &a)
{
    const int64_t m = a.mid + (a.low >> 32);
    const int64_t v = a.r + (m >> 32);
    const uint32_t tie = 0x7fffffffu + (uint32_t)((uint64_t)v >> 63);
    return v + (int64_t)(((uint64_t)(uint32_t)m + tie) >> 32);
}

// Stage coefficients, out = base base + self g + heq - sum l D, times 2^61; for operands of
// one exponent self + base - 1 = -gamma h.
struct FxCoef {
    FxC self, base, relax;
};
// Transport coefficients -l / 2 (fx_nnd2 gives 2 D) times 2^61, and times 2^64 for operands
// of one exponent.
struct FxFlux {
    FxC lx[4], ly[4];
    FxC klx[4], kly[4];
};

inline FxCoef fx_coef(double self, double base)
{
    FxCoef k;
    k.self = fx_const(self, 61);
    k.base = fx_const(base, 61);
    // the same real numbers in both forms: self + base - 1 from the rounded constants
    k.relax = fx_split(fx_int(k.self) + fx_int(k.base) - ((int64_t)1 << 61));
    if (k.relax.lo == INT32_MIN) {       // see fx_mul
        k.self = fx_split(fx_int(k.self) + 1);
        k.relax.lo += 1;
    }
    return k;
}
// lx, ly: gamma dt c_g / dr; along an axis of one cell every difference is zero and l
// is not bounded by the stability limit.
inline FxFlux fx_flux(const double lx[4], const double ly[4], bool along_x, bool along_y)
{
    FxFlux f;
    auto set = [](double l, FxC &c, FxC &k) {
        int64_t b = std::llrint(std::ldexp(-0.5 * l, 61));
        if (b < -((int64_t)1 << 60)) b = -((int64_t)1 << 60);    // l = 1 but for rounding
        if ((uint32_t)((uint64_t)b << 3) == 0x80000000u) ++b;    // see fx_mul
        c = fx_split(b);
        k = fx_split((int64_t)((uint64_t)b << 3));
    };
    for (int g = 0; g < 4; ++g) {
        set(along_x ? lx[g] : 0.0, f.lx[g], f.klx[g]);
        set(along_y ? ly[g] : 0.0, f.ly[g], f.kly[g]);
    }
    return f;
}

}  // namespace cdbm
