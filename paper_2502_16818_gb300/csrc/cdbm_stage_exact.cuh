// One cell of a Runge-Kutta stage in double precision: the operations and the rounding of
// primitives(), equilibrium() and nnd(), with the sums of the velocity groups and the
// transport differences on the integer pipes where they have the bits of the FP64
// operations (cdbm_exact.h).  That leaves 141 / 157 of the 246 / 262 FP64 instructions per
// cell in the two stages.
//
// rounded: the quadrupole of a group is rounded before it is added to the group sum.  The
// stages of tubes of up to kRoundedTube cells round so, all other grids fuse the product
// into the sum.  (Each keeps the rounding it has always had: the scheme amplifies one unit
// in the last place by many orders of magnitude.)
#pragma once

#include "cdbm_device.cuh"
#include "cdbm_exact.h"

namespace cdbm {

constexpr int kRoundedTube = 8192;

// nnd() with the bits of its FP64 form.
__device__ __forceinline__ double nnd_exact(double u2, double u1, double c, double d1)
{
    double d;
    if (!ex_nnd(u2, u1, c, d1, d)) d = nnd(u2, u1, c, d1);
    return d;
}

// The conserved moments from the group sums, in the order of conserved().
__device__ __forceinline__ double group_dot(const double c[4], const double s[4])
{
    return fma(c[3], s[3], fma(c[2], s[2], fma(c[1], s[1], __dmul_rn(c[0], s[0]))));
}
__device__ __forceinline__ Cons group_moments(const ModelConsts &m, const double s0[4], const double sx[4], const double sy[4])
{
    return {(s0[0] + s0[1]) + (s0[2] + s0[3]), group_dot(m.c, sx), group_dot(m.c, sy), group_dot(m.w, s0)};
}
template <typename TS>
__device__ __forceinline__ Cons moments_exact(const ModelConsts &m, const TS f[kNV])
{
    double s0[4], sx[4], sy[4];
#pragma unroll
    for (int g = 0; g < 4; ++g) {
        const GroupSums s = ex_group_sums(g & 1, f + 4 * g);
        s0[g] = s.s0;
        sx[g] = s.sx;
        sy[g] = s.sy;
    }
    return group_moments(m, s0, sx, sy);
}

// The four members of a group of the scaled equilibrium.
struct EqGroup {
    double h0, h1, h2, h3;
    __device__ __forceinline__ double member(int j) const { return (j & 2) ? ((j & 1) ? h3 : h2) : ((j & 1) ? h1 : h0); }
};

// Group g, an axis or a diagonal one (kDiag).  kSym: of a y-symmetric state, whose y-odd
// components and diagonal quadrupole are zero.
template <bool kDiag, bool kSym = false>
__device__ __forceinline__ EqGroup eq_group(const EqBlocks &B, const EqFactors &q, int g, bool rounded)
{
    const double *S = B.S + 4 * g, *W = B.Vc + 4 * g;
    const double s0 = fma(S[3], q.m1416, fma(S[2], q.ru2, fma(S[1], q.E, __dmul_rn(S[0], q.rho))));
    const double f = kDiag ? q.m6 : q.d57;
    const double X = kDiag ? fma(B.B2[g], q.W4, B.B2[g - 1]) : fma(B.B1[g + 1], q.W4, B.B1[g]);
    double A, D;                          // s0 plus and minus the quadrupole f X
    if constexpr (kSym && kDiag) {
        A = D = s0;
    } else if (rounded) {
        const double d = __dmul_rn(f, X);
        A = __dadd_rn(s0, d);
        D = __dsub_rn(s0, d);
    } else {
        A = fma(f, X, s0);
        D = fma(-f, X, s0);
    }
    const double cm = fma(W[2], q.u2, fma(W[1], q.T, W[0]));
    const double px = fma(W[3], q.dlt, cm), py = fma(-W[3], q.dlt, cm);
    if constexpr (!kDiag) {
        const double n = kSym ? D : fma(q.jy, py, D), s = kSym ? D : fma(-q.jy, py, D);
        return {fma(q.jx, px, A), n, fma(-q.jx, px, A), s};
    } else {
        const double sy = kSym ? 0.0 : __dmul_rn(q.jy, py);
        const double U = kSym ? __dmul_rn(q.jx, px) : fma(q.jx, px, sy), V = kSym ? U : fma(q.jx, px, -sy);
        return {A + U, D - V, A - U, D + V};
    }
}

// Cell, its upwind-ordered neighbours (two up, one up, one down) along x and y, and its
// base value.
struct Stencil {
    double c, x2, x1, xd, y2, y1, yd, base;
};

// ---- a cell on 16 threads ----

// Shared memory of 32 cells whose velocities are on 16 warps.
struct Cells16 {
    double f[kNV][32];
    double s0[4][32], sx[4][32], sy[4][32];
    double moment[4][32];
    EqFactors factors[32];
    double h[kNV][32];
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
// shortest with one velocity per thread.  Four warps form one group's sums and one moment
// each, one of them the factors of the equilibrium while the others take the transport (of
// a 1-D grid; on 2-D grids the warp of the factors takes its own later), and four one group
// each; five block barriers, which every thread of the block reaches, separate the
// exchanges through shared memory.  v: the cell's value, its neighbours (the cell itself
// along an axis without component) and base.  `lead`: the warp that forms the factors,
// below 4.
template <bool kFlatY, bool kBase, bool kRounded>
__device__ __forceinline__ double cell16(const StageArgs &a, Cells16 &s, int w, int lead, int i, const Stencil &v,
                                         unsigned *flag)
{
    const int lane = threadIdx.x & 31, g = i >> 2;
    s.f[i][lane] = v.c;
    __syncthreads();
    if (w < 4) {                          // group w
        double q[4];
#pragma unroll
        for (int j = 0; j < 4; ++j) q[j] = s.f[4 * w + j][lane];
        const GroupSums r = (w & 1) ? ex_group_sums(true, q) : ex_group_sums(false, q);
        s.s0[w][lane] = r.s0;
        s.sx[w][lane] = r.sx;
        s.sy[w][lane] = r.sy;
    }
    __syncthreads();
    if (w < 4) {                          // moment w: rho, j_x, j_y, E
        double x[4];
#pragma unroll
        for (int k = 0; k < 4; ++k) x[k] = w == 1 ? s.sx[k][lane] : (w == 2 ? s.sy[k][lane] : s.s0[k][lane]);
        s.moment[w][lane] = w == 0 ? (x[0] + x[1]) + (x[2] + x[3]) : (w == 3 ? group_dot(a.m.w, x) : group_dot(a.m.c, x));
    }
    __syncthreads();
    const int dx = dirx(i), dy = kFlatY ? 0 : diry(i);
    double tx = 0.0, ty = 0.0;
    auto transport = [&]() {
        if (dx != 0) tx = nnd_exact(v.x2, v.x1, v.c, v.xd);
        if (dy != 0) ty = nnd_exact(v.y2, v.y1, v.c, v.yd);
    };
    if (w == lead)
        s.factors[lane] = eq_factors(a.m, s.moment[0][lane], s.moment[1][lane], s.moment[2][lane], s.moment[3][lane],
                                     flag);
    else
        transport();
    __syncthreads();
    if (w < 4) {                          // group w
        const EqFactors &q = s.factors[lane];
        const EqGroup e = (w & 1) ? eq_group<true>(a.eq, q, w, kRounded) : eq_group<false>(a.eq, q, w, kRounded);
        s.h[4 * w][lane] = e.h0;
        s.h[4 * w + 1][lane] = e.h1;
        s.h[4 * w + 2][lane] = e.h2;
        s.h[4 * w + 3][lane] = e.h3;
    }
    if (w == lead) transport();           // nothing on a 1-D grid
    __syncthreads();
    double o = fma(a.a_self, v.c, s.h[i][lane]);
    if (kBase) o = fma(a.a_base, v.base, o);
    if (dx != 0) o = fma(-a.lx[g], tx, o);
    if (dy != 0) o = fma(-a.ly[g], ty, o);
    return o;
}

}  // namespace cdbm
