// Runge-Kutta stage kernels of the double-precision state on a grid: a cell per thread, on
// two threads or on 16, all with the same values bit for bit (cdbm_stage_exact.cuh).
#include "cdbm_stage_exact.cuh"

namespace cdbm {

namespace {

constexpr int kThreads = 128;

// Row pointers and offsets of a cell's stencil.  The row pointers are uniform over a
// block, the offsets in a row 32 bits wide (kWide: 64 bits, for rows of 2^29 cells and
// more), which saves the 64-bit address arithmetic of about 100 loads per cell.
template <bool kWide>
struct GridStencil {
    using Off = std::conditional_t<kWide, size_t, unsigned>;
    Off c, m2, m1, p1, p2;
    size_t row, rm2, rm1, rp1, rp2;
    __device__ __forceinline__ GridStencil(int x, int nx, int bc)
        : c((Off)8 * x), m2((Off)8 * neighbour_near(x - 2, nx, bc)), m1((Off)8 * neighbour_near(x - 1, nx, bc)),
          p1((Off)8 * neighbour_near(x + 1, nx, bc)), p2((Off)8 * neighbour_near(x + 2, nx, bc))
    {
    }
    template <bool kFlatY>
    __device__ __forceinline__ void at_row(int y, int nx, int ny, int bc)
    {
        row = (size_t)y * nx;
        if (!kFlatY) {
            rm2 = (size_t)neighbour_near(y - 2, ny, bc) * nx;
            rm1 = (size_t)neighbour_near(y - 1, ny, bc) * nx;
            rp1 = (size_t)neighbour_near(y + 1, ny, bc) * nx;
            rp2 = (size_t)neighbour_near(y + 2, ny, bc) * nx;
        }
    }
    static __device__ __forceinline__ double get(const double *p, Off o) { return __ldg((const double *)((const char *)p + o)); }
};

// The four members of group grp of one cell: loads, update and stores, one member per
// pass.  The passes differ in the offsets of the neighbours only and share their code:
// unrolled, the members' independent chains overlap, but the code outgrows the instruction
// cache as soon as other paths run beside it.
template <int kUnroll, bool kDiag, bool kFlatY, bool kBase, bool kWide>
__device__ __forceinline__ void grid_group(const double *g, const double *base, double *out, const StageArgs &a,
                                           const GridStencil<kWide> &st, size_t P, int grp, const EqGroup h, bool live)
{
    using St = GridStencil<kWide>;
    auto pass = [&](int j, auto transport) {
        constexpr bool kX = decltype(transport)::value;
        const size_t plane = (4 * grp + j) * P;
        const double *gp = g + plane, *gr = gp + st.row;
        const double c = St::get(gr, st.c);
        double o = fma(a.a_self, c, h.member(j));
        if (kBase) o = fma(a.a_base, *(const double *)((const char *)(base + plane + st.row) + st.c), o);
        if constexpr (kX && (kDiag || kFlatY)) {
            const bool west = kDiag ? j == 1 || j == 2 : j == 2;
            o = fma(-a.lx[grp], nnd_exact(St::get(gr, west ? st.p2 : st.m2), St::get(gr, west ? st.p1 : st.m1), c,
                                          St::get(gr, west ? st.m1 : st.p1)), o);
            if constexpr (kDiag && !kFlatY)
                o = fma(-a.ly[grp], nnd_exact(St::get(gp + (j < 2 ? st.rm2 : st.rp2), st.c),
                                              St::get(gp + (j < 2 ? st.rm1 : st.rp1), st.c), c,
                                              St::get(gp + (j < 2 ? st.rp1 : st.rm1), st.c)), o);
        } else if constexpr (kX) {     // E, W along x; N, S along y
            const bool up = j & 1, neg = j >= 2;
            const double u2 = St::get(gp + (up ? (neg ? st.rp2 : st.rm2) : st.row), up ? st.c : (neg ? st.p2 : st.m2));
            const double u1 = St::get(gp + (up ? (neg ? st.rp1 : st.rm1) : st.row), up ? st.c : (neg ? st.p1 : st.m1));
            const double d1 = St::get(gp + (up ? (neg ? st.rm1 : st.rp1) : st.row), up ? st.c : (neg ? st.m1 : st.p1));
            o = fma(-(up ? a.ly[grp] : a.lx[grp]), nnd_exact(u2, u1, c, d1), o);
        }
        if (live) *(double *)((char *)(out + plane + st.row) + st.c) = o;
    };
    if constexpr (!kDiag && kFlatY) {
#pragma unroll kUnroll
        for (int j = 0; j < 4; j += 2) pass(j, std::true_type{});
#pragma unroll kUnroll
        for (int j = 1; j < 4; j += 2) pass(j, std::false_type{});    // N, S of a 1-D grid: no transport
    } else {
#pragma unroll kUnroll
        for (int j = 0; j < 4; ++j) pass(j, std::true_type{});
    }
}

// Stage in double precision, one cell per thread.  Bound by the FP64 pipe (141 / 157
// instructions of 64 cycles in the two stages, 86-87 % busy); with all sums and differences on that pipe
// it took 246 / 262 at best, rows marched and differences shared.  4.59 ms per 4096^2 stage
// of the vortex (7.91 before), 0.557 per 1500 x 1300 of smooth fields (1.02).  64 registers
// for 32 warps per SM, which hide the latency of the integer chains (20 warps: 4.59-4.72 and
// 0.563-0.576, 16: 4.75 and 0.564).
constexpr int kMinBlocks = 8;
template <bool kBase, bool kFlatY, bool kRounded, bool kWide>
__global__ void __launch_bounds__(kThreads, kMinBlocks)
    stage_double_kernel(const double *__restrict__ g, const double *base, double *out, const __grid_constant__ StageArgs a,
                        unsigned *flag)
{
    const int x = blockIdx.x * blockDim.x + threadIdx.x;
    if (x >= a.nx) return;
    const size_t P = (size_t)a.nx * a.ny;
    GridStencil<kWide> st(x, a.nx, a.bc_x);
    for (int y = blockIdx.y; y < a.ny; y += gridDim.y) {
        st.template at_row<kFlatY>(y, a.nx, a.ny, a.bc_y);
        const double *own = g + st.row + x;
        double f[kNV];
#pragma unroll
        for (int i = 0; i < kNV; ++i) f[i] = __ldg(own + i * P);
        const Cons m = moments_exact(a.m, f);
        const EqFactors q = eq_factors(a.m, m.rho, m.jx, m.jy, m.E, flag);
#pragma unroll 1
        for (int p = 0; p < 4; p += 2) {
            grid_group<1, false, kFlatY, kBase>(g, base, out, a, st, P, p, eq_group<false>(a.eq, q, p, kRounded), true);
            grid_group<1, true, kFlatY, kBase>(g, base, out, a, st, P, p + 1, eq_group<true>(a.eq, q, p + 1, kRounded), true);
        }
    }
}

// The same stage with a cell on two threads: on a grid of some ten thousand cells the time
// of a stage is the chain of one thread, which this shortens.  Two warps of a block have
// two velocity groups of 32 cells each; they exchange the groups' sums through shared
// memory, and each forms the moments and the factors of the equilibrium.  With few warps
// per SM the members' passes are unrolled so that their chains overlap.
template <bool kBase, bool kFlatY, bool kRounded>
__global__ void __launch_bounds__(128, 4)
    stage_double_split_kernel(const double *__restrict__ g, const double *base, double *out,
                              const __grid_constant__ StageArgs a, unsigned *flag)
{
    // by parity of the row: a warp that has passed the next row's barrier writes the other
    // half, and the half it reads is written again only after one more barrier
    __shared__ double sums[2][4][3][64];
    const int warp = threadIdx.x >> 5;
    const int way = warp & 1, at = (warp >> 1) * 32 + (threadIdx.x & 31);
    const int x0 = blockIdx.x * 64 + at;
    const bool live = x0 < a.nx;
    const int x = live ? x0 : a.nx - 1;              // idle lanes mirror the last cell
    const size_t P = (size_t)a.nx * a.ny;
    GridStencil<true> st(x, a.nx, a.bc_x);
    int b = 0;
    for (int y = blockIdx.y; y < a.ny; y += gridDim.y, b ^= 1) {
        st.template at_row<kFlatY>(y, a.nx, a.ny, a.bc_y);
        const double *own = g + (size_t)(8 * way) * P + st.row + x;
        const int grp = 2 * way;
        double f[8];
#pragma unroll
        for (int j = 0; j < 8; ++j) f[j] = __ldg(own + j * P);
#pragma unroll
        for (int k = 0; k < 2; ++k) {
            const GroupSums s = ex_group_sums(k, f + 4 * k);
            sums[b][grp + k][0][at] = s.s0;
            sums[b][grp + k][1][at] = s.sx;
            sums[b][grp + k][2][at] = s.sy;
        }
        __syncthreads();
        double s0[4], sx[4], sy[4];
#pragma unroll
        for (int h = 0; h < 4; ++h) {
            s0[h] = sums[b][h][0][at];
            sx[h] = sums[b][h][1][at];
            sy[h] = sums[b][h][2][at];
        }
        const Cons m = group_moments(a.m, s0, sx, sy);
        const EqFactors q = eq_factors(a.m, m.rho, m.jx, m.jy, m.E, flag);
        grid_group<4, false, kFlatY, kBase>(g, base, out, a, st, P, grp, eq_group<false>(a.eq, q, grp, kRounded), live);
        grid_group<4, true, kFlatY, kBase>(g, base, out, a, st, P, grp + 1, eq_group<true>(a.eq, q, grp + 1, kRounded), live);
    }
}

// The same stage with a cell on 16 threads (cell16): 512 threads per 32 cells of a row.
template <bool kBase, bool kFlatY, bool kRounded>
__global__ void __launch_bounds__(512, 2)
    stage_double_cell16_kernel(const double *__restrict__ g, const double *base, double *out,
                               const __grid_constant__ StageArgs a, unsigned *flag)
{
    __shared__ Cells16 s;
    const int w = threadIdx.x >> 5, i = cell16_velocity(w);
    const int x0 = blockIdx.x * 32 + (int)(threadIdx.x & 31);
    const bool live = x0 < a.nx;
    const int x = live ? x0 : a.nx - 1;              // idle lanes mirror the last cell
    const int dx = dirx(i), dy = kFlatY ? 0 : diry(i);
    const size_t P = (size_t)a.nx * a.ny;
    const int xm2 = neighbour_near(x - 2 * dx, a.nx, a.bc_x), xm1 = neighbour_near(x - dx, a.nx, a.bc_x),
              xp1 = neighbour_near(x + dx, a.nx, a.bc_x);
    for (int y = blockIdx.y; y < a.ny; y += gridDim.y) {
        const double *gp = g + i * P, *gr = gp + (size_t)y * a.nx;
        const size_t c = i * P + (size_t)y * a.nx + x;
        Stencil v = {gr[x], gr[xm2], gr[xm1], gr[xp1], 0, 0, 0, kBase ? base[c] : 0.0};
        if (!kFlatY) {
            v.y2 = gp[(size_t)neighbour_near(y - 2 * dy, a.ny, a.bc_y) * a.nx + x];
            v.y1 = gp[(size_t)neighbour_near(y - dy, a.ny, a.bc_y) * a.nx + x];
            v.yd = gp[(size_t)neighbour_near(y + dy, a.ny, a.bc_y) * a.nx + x];
        }
        const double o = cell16<kFlatY, kBase, kRounded>(a, s, w, 0, i, v, flag);
        if (live) out[c] = o;
        // the next row's writes to what this row still reads (s.h) follow four barriers
    }
}

template <bool kBase, bool kFlatY, bool kRounded>
void *stage_func(int ways, bool wide)
{
    if (ways == 16) return (void *)stage_double_cell16_kernel<kBase, kFlatY, kRounded>;
    if (ways == 2) return (void *)stage_double_split_kernel<kBase, kFlatY, kRounded>;
    if constexpr (!kRounded) {
        if (wide) return (void *)stage_double_kernel<kBase, kFlatY, false, true>;
    }
    return (void *)stage_double_kernel<kBase, kFlatY, kRounded, false>;
}

template <bool kBase>
void *stage_func(int ways, bool flat, bool rounded, bool wide)
{
    if (!flat) return stage_func<kBase, false, false>(ways, wide);
    return rounded ? stage_func<kBase, true, true>(ways, wide) : stage_func<kBase, true, false>(ways, wide);
}

}  // namespace

StageLaunch double_stage_launch_config(const StageArgs &a, bool with_base, int sm_count, bool allow_split)
{
    StageLaunch L;
    const bool flat = a.ny == 1, rounded = flat && a.nx <= kRoundedTube;
    auto pad = [&](unsigned t) { return ((size_t)a.nx + t - 1) / t * t; };
    // While the grid leaves most of the SMs' threads idle, the time is the chain of one
    // thread, and the cell is split over 16 threads or two; the lanes past a row's end count
    // as cells.  us per stage with 16 threads per cell, two and one: 5.4 / 10.6 / 17.5 at
    // 64^2, 16.5 / 19.8 / 23.0 at 160^2, 19.6 / 19.5 / 22.9 at 168^2, 21.7 / 20.0 / 23.4 at
    // 192^2, 26.0 / 33.1 / 24.6 at 200^2; tubes of 4000 cells 4.3 / 7.0 / 12.2, of 22000
    // 11.9 / 11.9 / 15.5, of 36000 17.3 / 15.0 / 16.1, of 40000 19.2 / 18.1 / 17.2; 3 x 4096
    // cells 70 / 111 / 54, 33 x 700 26.3 / 29.9 / 23.0, 63 x 420 17.5 / 17.0 / 20.5.
    int ways = 1;
    if (allow_split && pad(32) * a.ny <= (size_t)sm_count * 180) ways = 16;
    else if (allow_split && pad(64) * a.ny <= (size_t)sm_count * 255) ways = 2;
    unsigned w = ways == 16 ? 32 : 64;
    if (ways == 1) {
        // the widest block whose padding past the row's end is least
        w = kThreads;
        for (unsigned t = kThreads / 2; t >= 32; t /= 2)
            if (pad(t) < pad(w)) w = t;
    }
    const bool wide = a.nx >= (1 << 29);
    L.func = with_base ? stage_func<true>(ways, flat, rounded, wide) : stage_func<false>(ways, flat, rounded, wide);
    L.block = dim3(ways == 16 ? 512 : ways * w, 1, 1);
    L.grid = dim3((unsigned)(pad(w) / w), a.ny < 65535 ? a.ny : 65535, 1);
    return L;
}

}  // namespace cdbm
