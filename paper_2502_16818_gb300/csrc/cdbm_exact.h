// Double-precision sums and differences on the integer pipes, with the bits of the FP64
// operations they stand for.
//
// On GB300 one FP64 instruction occupies its pipe for 64 cycles per SM sub-partition, a
// 32-bit integer instruction for 1 to 2.  Where the operands of a sum share sign and
// exponent (the usual case in smooth flow: the members of a velocity group, a value and
// its neighbours), their mantissas are integers of one scale: differences are exact in
// 53 bits, a sum of two rounds by one bit.  Every other case takes the FP64 operations.
// The time step must round as FP64 arithmetic does: on fine grids the scheme amplifies a
// difference of one unit in the last place by many orders of magnitude (a Sod tube of 8192
// cells: 1e10 in 500 steps), so results are reproducible only with the same rounding.
//
// The same source compiles for the host, where a test compares it with the C operations
// bit for bit.
#pragma once

#include <cstdint>

#include "cdbm_convert.h"
#include "cdbm_fixed.h"

#if defined(__CUDACC__)
#define CDBM_EX_HD __host__ __device__ __forceinline__
#else
#define CDBM_EX_HD inline
#endif

namespace cdbm {

CDBM_EX_HD int ex_clz64(uint64_t v)   // v != 0
{
#if defined(__CUDA_ARCH__)
    return __clzll((long long)v);
#else
    return __builtin_clzll(v);
#endif
}

CDBM_EX_HD int64_t ex_bits(double v) { return (int64_t)((uint64_t)f64_hi(v) << 32 | f64_lo(v)); }
CDBM_EX_HD double ex_double(uint64_t b) { return f64_from_words((uint32_t)(b >> 32), (uint32_t)b); }
CDBM_EX_HD int64_t ex_min(int64_t a, int64_t b) { return a < b ? a : b; }
CDBM_EX_HD int64_t ex_max(int64_t a, int64_t b) { return a > b ? a : b; }

// Exponent fields for which every result below is a normal number: differences of one unit
// in the last place lie 53 binades below their operands, sums of four two above.
CDBM_EX_HD bool ex_range(uint32_t hi) { return ((hi >> 20) & 0x7ffu) - 64u < 1980u; }

// m 2^(X - 1075), |m| < 2^53, with the sign bit `flip` applied; +0 for m = 0.
CDBM_EX_HD double ex_to_double(int64_t m, int X, uint32_t flip)
{
    const int64_t s = m >> 63;
    const uint64_t a = (uint64_t)((m ^ s) - s);
    if (a == 0) return 0.0;
    const int n = ex_clz64(a);
    const uint64_t b = (a << (n - 11)) + ((uint64_t)(uint32_t)(X + 10 - n) << 52);
    return f64_from_words((uint32_t)(b >> 32) | (((uint32_t)(s >> 32) ^ flip) & 0x80000000u), (uint32_t)b);
}

// a + b in units of twice that of the mantissas a, b (2^52 <= a, b <= 2^53): a sum of two
// doubles of one exponent, to nearest, ties to even.
CDBM_EX_HD int64_t ex_half_sum(int64_t a, int64_t b)
{
    const uint64_t m = (uint64_t)(a + b);
    return (int64_t)((m + ((m >> 1) & 1)) >> 1);
}

// Components of a group of members E N W S (axis group) or NE NW SW SE (diagonal group): s0
// their sum, sx and sy their x- and y-odd sums; of an axis group the x pair a and the y pair
// b, of a diagonal one a, odd in x and y.
struct GroupSums {
    double s0, sx, sy, a, b;
};

// ... by FP64 operations, the ones of conserved().
CDBM_EX_HD GroupSums group_sums(bool diag, const double q[4])
{
    if (!diag) {
        const double x = q[0] + q[2], y = q[1] + q[3];
        return {x + y, q[0] - q[2], q[1] - q[3], x, y};
    }
    const double e = q[0] + q[3], w = q[1] + q[2];
    return {e + w, e - w, (q[0] + q[1]) - (q[2] + q[3]), (q[0] + q[2]) - (q[1] + q[3]), 0.0};
}

// ... on the integer pipes, with the same bits.
CDBM_EX_HD GroupSums ex_group_sums(bool diag, const double q[4])
{
    const uint32_t h = f64_hi(q[0]);
    const uint32_t diff = (f64_hi(q[1]) ^ h) | (f64_hi(q[2]) ^ h) | (f64_hi(q[3]) ^ h);
    if ((diff >> 20) != 0 || !ex_range(h)) return group_sums(diag, q);
    const int E = (int)((h >> 20) & 0x7ffu);
    const uint32_t sign = h & 0x80000000u;
    const uint64_t one = (uint64_t)1 << 52;
    auto mantissa = [&](double v) { return (int64_t)(((uint64_t)ex_bits(v) & (one - 1)) | one); };
    auto sum = [&](int64_t m, int X) {                    // m of exponent X, 2^52 <= m <= 2^53
        const uint64_t b = (uint64_t)m + ((uint64_t)(uint32_t)(X - 1) << 52);
        return f64_from_words((uint32_t)(b >> 32) | sign, (uint32_t)b);
    };
    const int64_t m0 = mantissa(q[0]), m1 = mantissa(q[1]), m2 = mantissa(q[2]), m3 = mantissa(q[3]);
    if (!diag) {
        const int64_t x = ex_half_sum(m0, m2), y = ex_half_sum(m1, m3);
        return {sum(ex_half_sum(x, y), E + 2), ex_to_double(m0 - m2, E, sign), ex_to_double(m1 - m3, E, sign),
                sum(x, E + 1), sum(y, E + 1)};
    }
    const int64_t e = ex_half_sum(m0, m3), w = ex_half_sum(m1, m2);
    return {sum(ex_half_sum(e, w), E + 2), ex_to_double(e - w, E + 1, sign),
            ex_to_double(ex_half_sum(m0, m1) - ex_half_sum(m2, m3), E + 1, sign),
            ex_to_double(ex_half_sum(m0, m2) - ex_half_sum(m1, m3), E + 1, sign), 0.0};
}

// ... of single-precision members, summed as integers and rounded once: the FP64 sums are
// exact while the members lie within 27 binades, and these have their bits then; beyond,
// they round less often.
CDBM_EX_HD GroupSums ex_group_sums(bool diag, const float q[4])
{
    const int E = (int)(fx_max(fx_max(fx_key(q[0]), fx_key(q[1])), fx_max(fx_key(q[2]), fx_key(q[3]))) >> 24);
    if (E < 35 || E == 255) {             // a subnormal member could count; infinities, NaN
        const double w[4] = {(double)q[0], (double)q[1], (double)q[2], (double)q[3]};
        return group_sums(diag, w);
    }
    const int64_t m0 = fx_from(q[0], E), m1 = fx_from(q[1], E), m2 = fx_from(q[2], E), m3 = fx_from(q[3], E);
    auto to = [&](int64_t m) { return fx_to(m, E + (1023 - 127)); };
    const int64_t d = m0 - m2, b = m1 - m3, x = m0 + m2, y = m1 + m3;
    if (!diag) return {to(x + y), to(d), to(b), to(x), to(y)};
    return {to(x + y), to(d - b), to(d + b), to(x - y), 0.0};
}

// The transport difference nnd() of values of one sign and exponent: a = c - u1, b = d1 - c
// and e = u1 - u2 are exact, minmod(b, a) is b clamped to the interval between 0 and a, the
// difference of the limited slopes is exact because both lie in that interval, and the
// result (2 a + minmod(b, a) - minmod(a, e)) / 2 is exact while it is below 2^52 units.
// false: not that case.
CDBM_EX_HD bool ex_nnd(double u2, double u1, double c, double d1, double &out)
{
    const uint32_t h = f64_hi(c);
    const uint32_t diff = (f64_hi(u2) ^ h) | (f64_hi(u1) ^ h) | (f64_hi(d1) ^ h);
    const uint64_t C = (uint64_t)ex_bits(c), U = (uint64_t)ex_bits(u1);
    const int64_t a = (int64_t)(C - U), b = (int64_t)((uint64_t)ex_bits(d1) - C),
                  e = (int64_t)(U - (uint64_t)ex_bits(u2));
    const int64_t s = a >> 63;
    const int64_t lo = a & s, hi = a & ~s;
    const int64_t d = (int64_t)(2 * (uint64_t)a + (uint64_t)ex_max(ex_min(b, hi), lo) - (uint64_t)ex_max(ex_min(e, hi), lo));
    const bool ok = (diff >> 20) == 0 && ex_range(h) && ((uint64_t)d + ((uint64_t)1 << 53) - 1) < ((uint64_t)1 << 54) - 1;
    if (ok) out = ex_to_double(d, (int)((h >> 20) & 0x7ffu) - 1, h);
    return ok;
}

}  // namespace cdbm

#undef CDBM_EX_HD
