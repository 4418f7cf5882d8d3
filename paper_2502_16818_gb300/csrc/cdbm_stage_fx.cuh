// One cell of a Runge-Kutta stage in double precision with the sums, the transport
// and the update on the integer pipes (cdbm_fixed.h) and the equilibrium's
// polynomials on the FP64 pipe.
//
// The operations are those of primitives(), equilibrium() and nnd():
//   - the 16 values of the cell are brought to the cell's largest exponent and summed
//     exactly to the group components; rho, j and E are rounded to double once;
//   - u, T and the factors of the equilibrium are formed in double (68 FP64
//     instructions with the four groups', against 246 / 262 of the all-FP64 stage);
//   - the four components of a group are brought to their largest exponent, and the
//     members are their exact sums;
//   - each velocity is updated in one of two ways that evaluate the same sum of
//     products: where its stencil, base value and result share one sign and exponent
//     (fx_update; the usual case in smooth flow), differences are differences of the
//     doubles' bits, and the increment is added to them; elsewhere (fx_transport_any,
//     fx_relax_any) the operands are brought to the largest exponent among them.
//     Relaxation and transport are rounded one after the other: differences too small
//     to move a value by half a unit leave it unchanged, as in double arithmetic.  (With
//     one rounding of the whole sum, differences of one unit ahead of the Ma = 15 shock
//     survive and the scheme's own instability of that velocity set amplifies them
//     until the run fails after 7000 steps.)
// A velocity whose top exponent is outside [2^-895, 2^905) (zeros only, infinities,
// NaN) is left to the all-FP64 form.
#pragma once

#include "cdbm_device.cuh"
#include "cdbm_fixed.h"

namespace cdbm {

__device__ __forceinline__ bool fx_out_of_range(int E) { return (unsigned)(E - kExpLo) >= (unsigned)kExpSpan; }

// The factors of the equilibrium of one cell.
struct EqFactors {
    double rho, E, jx, jy, T, ru2, m1416, W4, d57, m6, u2, dlt;
};

__device__ __forceinline__ EqFactors eq_factors(const ModelConsts &m, double rho, double jx, double jy, double E,
                                                unsigned *flag)
{
    EqFactors q;
    const double r = rcp64(rho);
    const double ux = jx * r, uy = jy * r;
    const double jyuy = __dmul_rn(jy, uy), uy2 = __dmul_rn(uy, uy);
    q.ru2 = fma(jx, ux, jyuy);
    const double P = (E - q.ru2) * m.invK;
    q.T = P * r;
    if (!(positive_finite(rho) && positive_finite(P))) atomicOr(flag, kFlagNonPhys);
    q.rho = rho;
    q.E = E;
    q.jx = jx;
    q.jy = jy;
    q.u2 = fma(ux, ux, uy2);
    q.dlt = fma(ux, ux, -uy2);
    q.m1416 = fma(q.T, fma(m.Kp6, q.ru2, __dmul_rn(m.twoKp2, P)), __dmul_rn(q.ru2, q.u2));
    q.W4 = fma(m.Kp4, q.T, q.u2);
    q.d57 = fma(jx, ux, -jyuy);
    q.m6 = jx * uy;
    // kept in registers: the compiler otherwise repeats FP64 instructions in the loop
    // over the groups to save some
    asm volatile("" : "+d"(q.T), "+d"(q.ru2), "+d"(q.m1416), "+d"(q.W4), "+d"(q.d57), "+d"(q.m6), "+d"(q.u2), "+d"(q.dlt));
    return q;
}

// eq_factors() of a y-symmetric state (j_y = u_y = 0).
__device__ __forceinline__ EqFactors eq_factors_sym(const ModelConsts &m, double rho, double jx, double E, unsigned *flag)
{
    EqFactors q;
    const double r = rcp64(rho);
    const double ux = jx * r;
    q.ru2 = __dmul_rn(jx, ux);
    const double P = (E - q.ru2) * m.invK;
    q.T = P * r;
    if (!(positive_finite(rho) && positive_finite(P))) atomicOr(flag, kFlagNonPhys);
    q.rho = rho;
    q.E = E;
    q.jx = jx;
    q.jy = 0.0;
    q.u2 = __dmul_rn(ux, ux);
    q.dlt = q.u2;
    q.m1416 = fma(q.T, fma(m.Kp6, q.ru2, __dmul_rn(m.twoKp2, P)), __dmul_rn(q.ru2, q.u2));
    q.W4 = fma(m.Kp4, q.T, q.u2);
    q.d57 = q.ru2;
    q.m6 = 0.0;
    asm volatile("" : "+d"(q.T), "+d"(q.ru2), "+d"(q.m1416), "+d"(q.W4), "+d"(q.u2));
    q.dlt = q.u2;
    q.d57 = q.ru2;
    return q;
}

// ---- conserved moments ----

// Conserved moments rho, j_x, j_y, E of a cell; ok: in range.
struct FxCons {
    double rho, jx, jy, E;
    bool ok;
};

struct FxMoments {
    int64_t r;
    FxSum jx, jy, E;
};
constexpr FxMoments kFxNoMoments = {0, kFxHalfUnit, kFxHalfUnit, kFxHalfUnit};

// Group sums of the fixed-point members E N W S or NE NW SW SE of group g.
__device__ __forceinline__ void fx_group_sums(int g, const int64_t q[4], int64_t &s0, int64_t &sx, int64_t &sy)
{
    s0 = (q[0] + q[2]) + (q[1] + q[3]);
    const int64_t d = q[0] - q[2], b = q[1] - q[3];
    sx = (g & 1) == 0 ? d : d - b;
    sy = (g & 1) == 0 ? b : d + b;
}

__device__ __forceinline__ void fx_add_sums(const FxModel &fm, int g, int64_t s0, int64_t sx, int64_t sy, FxMoments &m)
{
    m.r += s0;
    fx_mul(m.jx, sx, fm.c[g]);
    fx_mul(m.jy, sy, fm.c[g]);
    fx_mul(m.E, s0, fm.w[g]);
}

__device__ __forceinline__ FxCons fx_round_moments(const FxModel &fm, const FxMoments &m, int top)
{
    return {fx_to(m.r, top), fx_to(fx_sum59(m.jx), top + fm.cexp), fx_to(fx_sum59(m.jy), top + fm.cexp),
            fx_to(fx_sum59(m.E), top + fm.wexp), !fx_out_of_range(top)};
}

// Of the 16 values value(i), doubles or floats (E and the range are those of doubles).
template <class Value>
__device__ __forceinline__ FxCons fx_conserved(const FxModel &fm, Value value)
{
    using T = decltype(value(0));
    T f[kNV];
    uint32_t key = 0;
#pragma unroll
    for (int i = 0; i < kNV; ++i) f[i] = value(i);
#pragma unroll
    for (int i = 0; i < kNV; ++i) key = fx_max(key, fx_key(f[i]));
    const int top = (int)(key >> (kSingle<T> ? 24 : 21));
    FxMoments m = kFxNoMoments;
#pragma unroll
    for (int g = 0; g < 4; ++g) {
        int64_t q[4], s0, sx, sy;
#pragma unroll
        for (int j = 0; j < 4; ++j) q[j] = fx_from(f[4 * g + j], top);
        fx_group_sums(g, q, s0, sx, sy);
        fx_add_sums(fm, g, s0, sx, sy, m);
    }
    FxCons c = fx_round_moments(fm, m, kSingle<T> ? top + (1023 - 127) : top);
    if (kSingle<T>) c.ok = top < 255;
    return c;
}

// ---- equilibrium of a group ----

constexpr int kGroupLead = 60;   // bit of the leading one of a component at the group's top exponent

// The four members of a group of the scaled equilibrium in fixed point.
struct FxGroup {
    int64_t h0, h1, h2, h3;
    int G;                       // their top exponent
    __device__ __forceinline__ int64_t member(int j) const { return (j & 2) ? ((j & 1) ? h3 : h2) : ((j & 1) ? h1 : h0); }
};

// Group g.  The products with the blocks stay in FP64: as integer dot products at one
// exponent per cell they leave 30 of the 68 FP64 instructions, but the stage is not bound
// by that pipe any more (1.28 against 1.02 ms per step of 1500 x 1300 cells).
// kSym: of a y-symmetric state, whose y-odd components and diagonal quadrupole
// are zero.
template <bool kSym = false>
__device__ __forceinline__ FxGroup fx_group(const EqBlocks &B, const EqFactors &q, int g)
{
    const double *S = B.S + 4 * g, *W = B.Vc + 4 * g;
    const double s0 = fma(S[3], q.m1416, fma(S[2], q.ru2, fma(S[1], q.E, S[0] * q.rho)));
    const double qv = (g & 1) == 0 ? q.d57 * fma(B.B1[g + 1], q.W4, B.B1[g])
                      : kSym       ? 0.0
                                   : q.m6 * fma(B.B2[g], q.W4, B.B2[g - 1]);
    const double cm = fma(W[2], q.u2, fma(W[1], q.T, W[0]));
    const double sx = q.jx * fma(W[3], q.dlt, cm), sy = kSym ? 0.0 : q.jy * fma(-W[3], q.dlt, cm);
    const int G = (int)(fx_max(fx_max(fx_key(s0), fx_key(qv)), fx_max(fx_key(sx), fx_key(sy))) >> 21);
    auto from = [G](double v) { return fx_from_t<false, kGroupLead>(v, G); };
    const int64_t a = from(s0), d = from(qv), x = from(sx), y = from(sy);
    const int64_t A = a + d, D = a - d;
    if ((g & 1) == 0) return {A + x, D + y, A - x, D - y, G};
    const int64_t U = x + y, V = x - y;
    return {A + U, D - V, A - U, D + V, G};
}

// ---- update of a velocity ----

// Cell, its upwind-ordered neighbours (two up, one up, one down) along x and y, and its
// base value.
struct FxStencil {
    double c, x2, x1, xd, y2, y1, yd, base;
};

// h 2^-n rounded to nearest, n >= 0.
__device__ __forceinline__ int64_t fx_shift(int64_t h, int n)
{
    n = fx_imin(n, 63);
    return (h >> n) + (int64_t)((((uint32_t)h << 1) >> fx_imin(n, 31)) & 1u);
}

// Any operands: the transport -sum l D in fixed point at the top exponent E of the cell
// and its upwind neighbours.  The two outer stencil values enter it only through minmod,
// which a value three binades above that exponent cannot win, so those are clamped.
// Where the velocity has no component along an axis the neighbours are the cell itself.
// One body for both axes keeps the code small: unrolled over axes and members it takes
// longer to fetch than to run (2.9 against 1.8 ms per step of piecewise-constant
// 1500 x 1300 fields).
struct FxTransport {
    int64_t t;
    int E;
};
template <bool kFlatY>
__device__ __forceinline__ FxTransport fx_transport_any(FxC lx, FxC ly, const FxStencil &v)
{
    uint32_t key = fx_max(fx_key(v.c), fx_key(v.x1));
    if (!kFlatY) key = fx_max(key, fx_key(v.y1));
    const int E = (int)(key >> 21);
    const int64_t c = fx_from(v.c, E);
    FxAcc l = {0, 0};
#pragma unroll 1
    for (int axis = 0; axis < (kFlatY ? 1 : 2); ++axis) {
        const double u2 = axis ? v.y2 : v.x2, u1 = axis ? v.y1 : v.x1, d1 = axis ? v.yd : v.xd;
        fx_mac(l, fx_nnd2(fx_clamped(u2, E), fx_from(u1, E), c, fx_clamped(d1, E)), axis ? ly : lx);
    }
    return {fx_sum<61>(l), E};
}
// ... and the update with it: relaxation and base at the top exponent of their terms,
// rounded to double, then the transport.  ok: in range.
template <bool kBase>
__device__ __forceinline__ double fx_relax_any(const FxCoef &k, const FxStencil &v, int64_t h, int G,
                                               const FxTransport &t, bool &ok)
{
    uint32_t key = fx_key(v.c);
    if (kBase) key = fx_max(key, fx_key(v.base));
    const int E = fx_imax((int)(key >> 21), G);
    FxAcc a = {0, 0};
    fx_mac(a, fx_from(v.c, E), k.self);
    if (kBase) fx_mac(a, fx_from(v.base, E), k.base);
    const double o = fx_to(fx_sum<61>(a) + fx_shift(h, E - G + (kGroupLead - kLead)), E);
    const int F = fx_imax(t.E, (int)(fx_key(o) >> 21));
    ok = !fx_out_of_range(E) && !fx_out_of_range(F);
    return fx_to(fx_from(o, F) + fx_shift(t.t, F - t.E), F);
}

// Operands of one sign and exponent: no conversion; the sum is in 64ths of c's unit in
// the last place and is added to c's bits.  false: not that case, or the result leaves
// the binade.
template <bool kX, bool kY, bool kBase>
__device__ __forceinline__ bool fx_update(const FxCoef &k, FxC lx, FxC ly, const FxStencil &v, int64_t h, int G,
                                          double &out)
{
    const uint32_t hc = f64_hi(v.c);
    uint32_t diff = 0;
    if (kX) diff |= (f64_hi(v.x2) ^ hc) | (f64_hi(v.x1) ^ hc) | (f64_hi(v.xd) ^ hc);
    if (kY) diff |= (f64_hi(v.y2) ^ hc) | (f64_hi(v.y1) ^ hc) | (f64_hi(v.yd) ^ hc);
    if (kBase) diff |= f64_hi(v.base) ^ hc;
    const int E = (int)((hc << 1) >> 21), n = E - G;
    const int64_t C = fx_raw(v.c), s = (int64_t)((int32_t)hc >> 31);
    const int64_t M = (C & 0xfffffffffffffll) | 0x10000000000000ll;
    FxSum a = kFxHalf, l = {0, 0, 0};
    fx_mul(a, M << kFxUp, k.relax);
    if (kBase) fx_mul(a, (int64_t)((uint64_t)(fx_raw(v.base) - C) << kFxUp), k.base);
    if (kX) fx_mul(l, fx_nnd2(fx_raw(v.x2), fx_raw(v.x1), C, fx_raw(v.xd)), lx);
    if (kY) fx_mul(l, fx_nnd2(fx_raw(v.y2), fx_raw(v.y1), C, fx_raw(v.yd)), ly);
    const int64_t m = (h ^ s) - s;                   // the sums are those of the magnitudes
    int64_t O = C + fx_round64ths(fx_sum64ths(a) + fx_shift(m, n + (kGroupLead - kLead)), C);
    if (kX || kY) O += fx_sum_units(l);
    diff |= (uint32_t)(O >> 32) ^ hc;
    out = fx_bits((uint32_t)(O >> 32), (uint32_t)O);
    return (diff & 0xfff00000u) == 0 && n >= -2 && !fx_out_of_range(E);
}

// The all-FP64 stage of one velocity: the constants it takes.
struct FxDouble {
    double a_self, a_base;
    const double *lx, *ly;
};

// The members in `mask` of group g of one cell in FP64.  A cell gives
// stencil<kFlatY>(i, dx, dy, base) and base(i), and takes put(i, v).
template <class Cell, bool kBase, bool kFlatY>
__device__ __noinline__ void fx_double_group(const Cell cell, const EqBlocks &B, const ModelConsts &m, const FxDouble d,
                                             int g, unsigned mask, unsigned *flag)
{
    double f[kNV], heq[kNV];
    for (int i = 0; i < kNV; ++i) f[i] = cell.template stencil<true>(i, 0, 0, 0.0).c;
    const Prim s = primitives<false>(f, m, 0.0, 0.0, flag);
    equilibrium<false>(B, m, s.q.rho, s.q.E, s.q.jx, s.q.jy, s.ux, s.uy, s.ru2, s.jyuy, s.p, s.T, heq);
#pragma unroll 1
    for (int j = 0; j < 4; ++j) {
        const int i = 4 * g + j, sx = dirx(i), sy = kFlatY ? 0 : diry(i);
        if (!(mask >> j & 1u)) continue;
        const FxStencil v = cell.template stencil<kFlatY>(i, sx, sy, kBase ? cell.base(i) : 0.0);
        double o = fma(d.a_self, v.c, heq[i]);
        if (kBase) o = fma(d.a_base, v.base, o);
        if (sx != 0) o = fma(-d.lx[g], nnd(v.x2, v.x1, v.c, v.xd), o);
        if (sy != 0) o = fma(-d.ly[g], nnd(v.y2, v.y1, v.c, v.yd), o);
        cell.put(i, o);
    }
}

// The members in `mask` of group g of one cell that fx_update() declined.
template <class Cell, bool kBase, bool kFlatY>
__device__ __noinline__ void fx_rest_of_group(const Cell cell, const EqBlocks &B, const ModelConsts &m, const FxCoef &k,
                                              const FxFlux &l, const FxDouble d, int g, unsigned mask, bool cell_ok,
                                              const FxGroup h, unsigned *flag)
{
    unsigned slow = cell_ok ? 0u : mask;
#pragma unroll 1
    for (int j = 0; j < 4; ++j) {
        if (!cell_ok || !(mask >> j & 1u)) continue;
        const int i = 4 * g + j;
        const FxStencil v = cell.template stencil<kFlatY>(i, dirx(i), diry(i), kBase ? cell.base(i) : 0.0);
        bool ok;
        const double o = fx_relax_any<kBase>(k, v, h.member(j), h.G, fx_transport_any<kFlatY>(l.lx[g], l.ly[g], v), ok);
        if (ok) cell.put(i, o);
        else slow |= 1u << j;
    }
    if (slow) fx_double_group<Cell, kBase, kFlatY>(cell, B, m, d, g, slow, flag);
}

// ---- a cell on 16 threads ----

// Shared memory of 32 cells whose velocities are on 16 warps.
struct FxCells16 {
    uint32_t key[kNV][32];
    int64_t q[kNV][32];
    double moment[4][32];
    EqFactors factors[32];
    int64_t h[kNV][32];
    int G[4][32];
};

// The velocity of warp w of 16: first the four that a 1-D grid does not move, whose warps
// (one on each SM sub-partition) also form the cell's equilibrium.
__device__ __forceinline__ int cell16_velocity(int w)
{
    return w < 4 ? (w < 2 ? 1 + 2 * w : 5 + 2 * w) : (w < 8 ? (w < 6 ? 2 * (w - 4) : 2 * w - 4) : (w < 12 ? w - 4 : w));
}

// One stage of the lane's cell for the velocity i of warp w: on a grid of a few hundred or
// thousand cells the time of a stage is the chain of one thread (about 4 cycles per
// integer instruction and 64 per FP64 one, the rate of each SM sub-partition), which is
// shortest with one velocity per thread.  Four warps form one moment each, one of them
// the factors while the others take the transport (of a 1-D grid; on 2-D grids the warp of
// the factors takes its own later), and four one group each; five block
// barriers, which every thread of the block reaches, separate the exchanges through
// shared memory.  (Repeating the moments and factors on the four group warps saves two
// barriers but lengthens the chain: 4.6 against 4.2 us on 500 cells.)  The values are
// those of the one-thread form.  v: the cell's value, its neighbours (the cell itself
// along an axis without component) and base.  `lead`: the warp that forms the
// factors, below 4.  Returns whether `out` is the result; otherwise the cell is outside
// the integer path (fx_double_group).
template <bool kFlatY, bool kBase>
__device__ __forceinline__ bool fx_cell16(const StageArgs &a, FxCells16 &s, int w, int lead, int i, const FxStencil &v,
                                          unsigned *flag, double &out)
{
    const int lane = threadIdx.x & 31, g = i >> 2;
    s.key[i][lane] = fx_key(v.c);
    __syncthreads();
    uint32_t key = 0;
#pragma unroll
    for (int k = 0; k < kNV; ++k) key = fx_max(key, s.key[k][lane]);
    const int top = (int)(key >> 21);
    const bool cell_ok = !fx_out_of_range(top);
    s.q[i][lane] = fx_from(v.c, top);
    __syncthreads();
    if (w < 4) {                          // moment w: rho, j_x, j_y, E
        FxSum m = kFxHalfUnit;
        int64_t r = 0;
#pragma unroll
        for (int k = 0; k < 4; ++k) {
            int64_t q[4], s0, sx, sy;
#pragma unroll
            for (int j = 0; j < 4; ++j) q[j] = s.q[4 * k + j][lane];
            fx_group_sums(k, q, s0, sx, sy);
            r += s0;
            fx_mul(m, w == 1 ? sx : (w == 2 ? sy : s0), w == 3 ? a.fx.m.w[k] : a.fx.m.c[k]);
        }
        s.moment[w][lane] = w == 0 ? fx_to(r, top) : fx_to(fx_sum59(m), top + (w == 3 ? a.fx.m.wexp : a.fx.m.cexp));
    }
    __syncthreads();
    const uint32_t hc = f64_hi(v.c);
    uint32_t diff = (f64_hi(v.x2) ^ hc) | (f64_hi(v.x1) ^ hc) | (f64_hi(v.xd) ^ hc);
    if (!kFlatY) diff |= (f64_hi(v.y2) ^ hc) | (f64_hi(v.y1) ^ hc) | (f64_hi(v.yd) ^ hc);
    if (kBase) diff |= f64_hi(v.base) ^ hc;
    const bool same = (diff & 0xfff00000u) == 0;
    FxTransport t = {0, 0};
    auto transport = [&]() {
        if (same) {
            FxSum l = {0, 0, 0};
            fx_mul(l, fx_nnd2(fx_raw(v.x2), fx_raw(v.x1), fx_raw(v.c), fx_raw(v.xd)), a.fx.l.klx[g]);
            if (!kFlatY) fx_mul(l, fx_nnd2(fx_raw(v.y2), fx_raw(v.y1), fx_raw(v.c), fx_raw(v.yd)), a.fx.l.kly[g]);
            t.t = fx_sum_units(l);
        } else {
            t = fx_transport_any<kFlatY>(a.fx.l.lx[g], a.fx.l.ly[g], v);
        }
    };
    if (w == lead)
        s.factors[lane] = eq_factors(a.m, s.moment[0][lane], s.moment[1][lane], s.moment[2][lane], s.moment[3][lane],
                                     flag);
    else if (!kFlatY || w >= 4)           // the first four of a 1-D grid have none
        transport();
    __syncthreads();
    if (w < 4) {                          // group w
        const FxGroup e = fx_group(a.eq, s.factors[lane], w);
        s.h[4 * w][lane] = e.h0;
        s.h[4 * w + 1][lane] = e.h1;
        s.h[4 * w + 2][lane] = e.h2;
        s.h[4 * w + 3][lane] = e.h3;
        s.G[w][lane] = e.G;
    }
    if (!kFlatY && w == lead) transport();
    __syncthreads();
    const int64_t h = s.h[i][lane];
    const int G = s.G[g][lane];
    bool ok = same;
    if (same) {                           // fx_update() with the transport at hand
        const int E = (int)((hc << 1) >> 21), n = E - G;
        const int64_t C = fx_raw(v.c), sg = (int64_t)((int32_t)hc >> 31);
        const int64_t M = (C & 0xfffffffffffffll) | 0x10000000000000ll;
        FxSum r = kFxHalf;
        fx_mul(r, M << kFxUp, a.fx.k.relax);
        if (kBase) fx_mul(r, (int64_t)((uint64_t)(fx_raw(v.base) - C) << kFxUp), a.fx.k.base);
        const int64_t m = (h ^ sg) - sg;
        const int64_t O = C + fx_round64ths(fx_sum64ths(r) + fx_shift(m, n + (kGroupLead - kLead)), C) + t.t;
        out = fx_bits((uint32_t)(O >> 32), (uint32_t)O);
        ok = (((uint32_t)(O >> 32) ^ hc) & 0xfff00000u) == 0 && n >= -2 && !fx_out_of_range(E);
    }
    if (!ok) {
        if (same || (kFlatY && w < 4)) t = fx_transport_any<kFlatY>(a.fx.l.lx[g], a.fx.l.ly[g], v);
        out = fx_relax_any<kBase>(a.fx.k, v, h, G, t, ok);
    }
    return ok && cell_ok;
}

}  // namespace cdbm
