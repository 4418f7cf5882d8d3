// Host check of the fixed-point arithmetic of the FP64 stage (csrc/cdbm_fixed.h) against
// 113-bit arithmetic: prints one "name worst" pair per check, errors in units of half a
// unit in the last place of the result's scale.
#include <algorithm>
#include <cstdio>
#include <random>

#include "cdbm_fixed.h"

#if defined(__aarch64__)
typedef long double Quad;            // IEEE quadruple precision
#else
typedef __float128 Quad;
#endif
using namespace cdbm;

static std::mt19937_64 R(7);
static double uni() { return (double)(R() >> 11) * 0x1p-53; }
static Quad qabs(Quad v) { return v < 0 ? -v : v; }
static Quad qmm(Quad x, Quad y)
{
    if (x == 0 || y == 0 || (x < 0) != (y < 0)) return 0;
    return qabs(x) <= qabs(y) ? x : y;
}
static Quad qnnd(Quad u2, Quad u1, Quad c, Quad d1)
{
    return (c - u1) + (qmm(d1 - c, c - u1) - qmm(c - u1, u1 - u2)) / 2;
}

int main()
{
    // conversion of integers to double: to nearest, ties to even, as the C conversion
    long bad = 0;
    for (int k = 0; k < 3000000; ++k) {
        int64_t v = (int64_t)(R() >> (1 + R() % 62));
        if (k % 3 == 0) v = (int64_t)((R() >> 11) | (1ull << 52)) * 512 + 256 * (int64_t)(R() % 3);   // near ties
        if (R() & 1) v = -v;
        const int E = 1000 + (int)(R() % 50);
        if (fx_to(v, E) != std::ldexp((double)v, E - 1023 - kLead)) ++bad;
    }
    std::printf("to_double %ld\n", bad);
    // double to fixed point and back: exact up to 6 binades below the top exponent
    bad = 0;
    for (int k = 0; k < 1000000; ++k) {
        const int d = (int)(R() % 7);
        const double v = std::ldexp(1.0 + uni(), 5 - d) * ((R() & 1) ? 1 : -1);
        if (fx_to(fx_from(v, 1023 + 5), 1023 + 5) != v) ++bad;
    }
    std::printf("round_trip %ld\n", bad);
    // transport, relaxation and base: the two forms of the update against quadruple precision
    double fast = 0, any = 0;
    long used = 0;
    for (int k = 0; k < 400000; ++k) {
        const double b0 = std::ldexp(1 + uni(), (int)(R() % 40) - 20) * ((R() & 1) ? 1 : -1);
        const double amp = std::ldexp(1.0, -(int)(R() % 30));
        double s[8];
        for (double &v : s) v = b0 * (1 + amp * (2 * uni() - 1));
        const bool wide = k % 4 == 3;                  // neighbours over many binades and of both signs
        if (wide)
            for (int j = 1; j < 7; ++j) s[j] = std::ldexp(s[j], (int)(R() % 31) - 15) * ((R() & 1) ? 1 : -1);
        const double h = uni(), self = 0.5 - 0.5 * h, base = 0.5, l = 0.5 * uni();
        const double lx[4] = {l, l, l, l}, ly[4] = {0.5 - l, 0.5 - l, 0.5 - l, 0.5 - l};
        const FxCoef c = fx_coef(self, base);
        const FxFlux f = fx_flux(lx, ly, true, true);
        const Quad T = (Quad)lx[0] * qnnd(s[1], s[2], s[0], s[3]) + (Quad)ly[0] * qnnd(s[4], s[5], s[0], s[6]);
        const Quad ref = (Quad)self * s[0] + (Quad)base * s[7] - T;
        const double big = std::max({std::fabs(s[0]), std::fabs(s[2]), std::fabs(s[5]), std::fabs(s[7])});
        const int E = (int)(fx_key(big) >> 21);
        FxAcc a = {0, 0};
        const int64_t x = fx_from(s[0], E);
        fx_mac(a, x, c.self);
        fx_mac(a, fx_from(s[7], E), c.base);
        fx_mac(a, fx_nnd2(fx_clamped(s[1], E), fx_from(s[2], E), x, fx_clamped(s[3], E)), f.lx[0]);
        fx_mac(a, fx_nnd2(fx_clamped(s[4], E), fx_from(s[5], E), x, fx_clamped(s[6], E)), f.ly[0]);
        any = std::max(any, (double)(qabs((Quad)fx_to(fx_sum<61>(a), E) - ref) / big) * 0x1p53);
        uint32_t diff = 0;
        for (int j = 1; j < 8; ++j) diff |= f64_hi(s[j]) ^ f64_hi(s[0]);
        if (diff & 0xfff00000u) continue;
        ++used;
        const int64_t C = fx_raw(s[0]), M = (C & 0xfffffffffffffll) | 0x10000000000000ll;
        FxSum r = kFxHalf, t = {0, 0, 0};
        fx_mul(r, M << kFxUp, c.relax);
        fx_mul(r, (fx_raw(s[7]) - C) * (1 << kFxUp), c.base);
        fx_mul(t, fx_nnd2(fx_raw(s[1]), fx_raw(s[2]), C, fx_raw(s[3])), f.klx[0]);
        fx_mul(t, fx_nnd2(fx_raw(s[4]), fx_raw(s[5]), C, fx_raw(s[6])), f.kly[0]);
        // the increment alone, in units in the last place of the cell's value
        const double ulp = std::ldexp(1.0, (int)((f64_hi(s[0]) >> 20) & 0x7ff) - 1023 - 52) * (s[0] < 0 ? -1 : 1);
        const Quad inc = (ref - s[0]) / ulp;
        const int64_t got = fx_round64ths(fx_sum64ths(r), C) + fx_sum_units(t);
        fast = std::max(fast, (double)qabs((Quad)got - inc));
    }
    std::printf("any %.3f\nfast %.3f\nused %ld\n", any, fast, used > 50000 ? 0l : used);
    // ties of the transport sum go toward zero
    bad = 0;
    const double half[4] = {1, 1, 1, 1};
    for (int64_t v = -9; v <= 9; ++v) {
        FxSum s = {0, 0, 0};
        fx_mul(s, v, fx_flux(half, half, true, true).klx[0]);   // -v / 2 of fx_nnd2's 2 D
        if (fx_sum_units(s) != -v / 2) ++bad;
    }
    std::printf("ties %ld\n", bad);
}
