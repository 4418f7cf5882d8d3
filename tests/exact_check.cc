// Host check of csrc/cdbm_exact.h: the sums and transport differences formed from integers
// against the C double operations, bit for bit.  Prints one "name mismatches" pair per check.
#include <cmath>
#include <cstdio>
#include <cstring>
#include <random>

#include "cdbm_exact.h"

using namespace cdbm;

static std::mt19937_64 R(11);
static bool same(double a, double b) { return std::memcmp(&a, &b, sizeof a) == 0; }
// + 0.0: the sign of an exact zero is left open
static bool same(const GroupSums &a, const GroupSums &b)
{
    return same(a.s0 + 0.0, b.s0 + 0.0) && same(a.sx + 0.0, b.sx + 0.0) && same(a.sy + 0.0, b.sy + 0.0) &&
           same(a.a + 0.0, b.a + 0.0) && same(a.b + 0.0, b.b + 0.0);
}
static double minmod(double X, double Y)
{
    if (X == 0 || Y == 0 || std::signbit(X) != std::signbit(Y)) return 0;
    return std::fabs(X) <= std::fabs(Y) ? X : Y;
}
static double nnd(double u2, double u1, double c, double d1)
{
    const double a = c - u1, b = d1 - c, e = u1 - u2;
    return std::fma(0.5, minmod(b, a) - minmod(a, e), a);
}
// A value of exponent field E whose mantissa spreads over `bits` bits around 1.5.
static double value(int E, int bits, bool neg)
{
    uint64_t m = R() >> 12;
    if (bits < 52) m = (1ull << 51) + (m >> (52 - bits));
    const uint64_t b = ((uint64_t)E << 52) | m | (neg ? 1ull << 63 : 0);
    double v;
    std::memcpy(&v, &b, sizeof v);
    return v;
}

int main()
{
    long bad_nnd = 0, bad_sums = 0, bad_float = 0, taken = 0, ranged = 0;
    for (int k = 0; k < 3000000; ++k) {
        // exponents over the whole range, its ends (subnormal results, overflow) oftener
        const int E = k % 5 == 0 ? 1 + (int)(R() % 130) : (k % 7 == 0 ? 2030 + (int)(R() % 16) : 1 + (int)(R() % 2046));
        const int bits = 1 + (int)(R() % 52);
        const bool neg = R() & 1;
        double q[4];
        for (double &v : q) v = value(k % 11 == 0 && E < 2046 ? E + (int)(R() & 1) : E, bits, k % 13 == 0 ? R() & 1 : neg);
        if (k % 17 == 0) q[R() % 4] = 0.0;
        if (k % 19 == 0) q[R() % 4] = q[R() % 4];
        double d;
        if (ex_nnd(q[0], q[1], q[2], q[3], d)) {
            ++taken;
            if (!same(d, nnd(q[0], q[1], q[2], q[3]))) ++bad_nnd;
        }
        ranged += E >= 64 && E < 2044;
        for (int diag = 0; diag < 2; ++diag)
            if (!same(ex_group_sums(diag, q), group_sums(diag, q))) ++bad_sums;
        // single-precision members within 27 binades, where the double sums are exact
        float f[4];
        double w[4];
        const int e0 = (int)(R() % 200) - 90;
        for (int j = 0; j < 4; ++j) {
            f[j] = (float)std::ldexp(value(1023, 52, R() & 1), e0 + (int)(R() % 27));
            w[j] = f[j];
        }
        if (k % 23 == 0) f[1] = 0.0f, w[1] = 0.0;
        if (k % 29 == 0)
            for (int j = 0; j < 4; ++j) w[j] = f[j] = std::ldexp(1.5f, -149 + (int)(R() % 40));   // subnormal and small
        for (int diag = 0; diag < 2; ++diag)
            if (!same(ex_group_sums(diag, f), group_sums(diag, w))) ++bad_float;
    }
    // the integer forms are what runs where they can: one sign and exponent, in range
    std::printf("nnd %ld\nsums %ld\nfloat %ld\ntaken %d\n", bad_nnd, bad_sums, bad_float, taken > ranged / 2 ? 0 : 1);
}
