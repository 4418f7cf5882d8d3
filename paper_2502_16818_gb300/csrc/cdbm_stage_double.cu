// Runge-Kutta stage kernels of the double-precision state entirely in FP64, for the run
// that the adjoint differentiates (cdbm_adjoint_forward and the recomputation of its
// segments).  cdbm_step takes the fixed-point kernels (cdbm_stage_fx.cuh), which agree to
// rounding and are twice as fast; but dL/dtau sums o . (f - f_eq) over the run, where
// f - f_eq is 1e-5 of f and the sum cancels over the cells, so it carries the rounding of
// every stage at 1e-9 to 1e-6 of its value.  Recorded gradients stay reproducible to the
// bit only with the rounding they were recorded with.
#include "cdbm_device.cuh"

namespace cdbm {

namespace {

constexpr int kThreads = 128;
constexpr int kMinBlocks = 3;     // resident blocks per SM the register budget must allow (168 registers)

__device__ __forceinline__ void stage_equilibrium(const StageArgs &a, const double f[kNV], double heq[kNV], unsigned *flag)
{
    const Prim s = primitives<false>(f, a.m, 0.0, 0.0, flag);
    equilibrium<false>(a.eq, a.m, s.q.rho, s.q.E, s.q.jx, s.q.jy, s.ux, s.uy, s.ru2, s.jyuy, s.p, s.T, heq);
}

// out = a_base base + a_self g + gamma h f_eq(g) - sum_r l_r D_r(g) for one cell:
// macros -> equilibrium -> BGK -> NND transport of all 16 velocities -> update.
template <bool kBase, bool kFlatY>
__global__ void __launch_bounds__(kThreads, kMinBlocks)
    stage_kernel(const double *__restrict__ g, const double *base, double *out, const StageArgs a, unsigned *flag)
{
    const int nx = a.nx, ny = a.ny;
    const int x = blockIdx.x * blockDim.x + threadIdx.x;
    if (x >= nx) return;
    const size_t P = (size_t)nx * ny;
    const int xm2 = neighbour_near(x - 2, nx, a.bc_x), xm1 = neighbour_near(x - 1, nx, a.bc_x);
    const int xp1 = neighbour_near(x + 1, nx, a.bc_x), xp2 = neighbour_near(x + 2, nx, a.bc_x);
    for (int y = blockIdx.y; y < ny; y += gridDim.y) {
        const size_t row = (size_t)y * nx;
        const size_t c = row + x;
        size_t rm2 = 0, rm1 = 0, rp1 = 0, rp2 = 0;
        if (!kFlatY) {
            rm2 = (size_t)neighbour_near(y - 2, ny, a.bc_y) * nx + x;
            rm1 = (size_t)neighbour_near(y - 1, ny, a.bc_y) * nx + x;
            rp1 = (size_t)neighbour_near(y + 1, ny, a.bc_y) * nx + x;
            rp2 = (size_t)neighbour_near(y + 2, ny, a.bc_y) * nx + x;
        }
        double fs[kNV];
#pragma unroll
        for (int i = 0; i < kNV; ++i) fs[i] = __ldg(g + i * P + c);
        double heq[kNV];
        stage_equilibrium(a, fs, heq, flag);

#pragma unroll
        for (int i = 0; i < kNV; ++i) {
            const int grp = i >> 2;
            const double *gp = g + i * P;
            double o = fma(a.a_self, fs[i], heq[i]);
            if (kBase) o = fma(a.a_base, base[i * P + c], o);
            if (dirx(i) != 0) {
                const double u2 = __ldg(gp + row + (dirx(i) > 0 ? xm2 : xp2));
                const double u1 = __ldg(gp + row + (dirx(i) > 0 ? xm1 : xp1));
                const double d1 = __ldg(gp + row + (dirx(i) > 0 ? xp1 : xm1));
                o = fma(-a.lx[grp], nnd(u2, u1, fs[i], d1), o);
            }
            if (!kFlatY && diry(i) != 0) {
                const double u2 = __ldg(gp + (diry(i) > 0 ? rm2 : rp2));
                const double u1 = __ldg(gp + (diry(i) > 0 ? rm1 : rp1));
                const double d1 = __ldg(gp + (diry(i) > 0 ? rp1 : rm1));
                o = fma(-a.ly[grp], nnd(u2, u1, fs[i], d1), o);
            }
            out[i * P + c] = o;
        }
    }
}

// Same stage for 2-D grids with the y-direction differences shared along a run of
// rows.  A block covers kThreads columns and a run of R = ceil(ny / gridDim.y)
// rows; each thread marches up its column.  For a velocity with y-sign s the
// upwind-ordered difference U_y = f_y - f_{y-s} and N_y = minmod(U_{y+s}, U_y) give
// the transport difference U_y + (N_y - N_{y-s}) / 2, which is the nnd() expression
// with a = U_y, b = U_{y-s}, e = U_{y+s}.  Each row computes one new U and one new N
// per velocity and carries them to the next row in shared memory, so a y-term costs
// 4 instead of 6 arithmetic instructions, with the same operations as stage_kernel.
constexpr int kNY = 12;                             // velocities with a y-component
constexpr size_t kMarchRowBytes = 2 * 12 * (kThreads + 2) * sizeof(double);   // FP64 x row buffers
__host__ __device__ constexpr int yvel(int k)       // k-th velocity with diry != 0
{
    return k < 2 ? 1 + 2 * k : (k < 6 ? k + 2 : (k < 8 ? 9 + 2 * (k - 6) : k + 4));
}

template <bool kBase>
__global__ void __launch_bounds__(kThreads, kMinBlocks)
    stage_march_kernel(const double *__restrict__ g, const double *base, double *out, const StageArgs a, unsigned *flag)
{
    // The x differences are shared as well: each thread computes
    // U_x = f_x - f_{x-s} of its cell once per velocity and reads U_{x+s}, U_{x-s} of
    // its neighbours from a row buffer (double-buffered in dynamic shared memory, so
    // one block barrier per row; the edge threads add the halo values), so an x-term
    // costs 4 FP64 instructions plus a share of the halo instead of 6.  The operands and operations are those of nnd(), so the
    // result is the same bit for bit.
    constexpr int kNXV = 12;                          // velocities with an x component
    __shared__ double carry_u[kNY][kThreads];
    __shared__ double carry_n[kNY][kThreads];
    extern __shared__ __align__(16) unsigned char march_dyn[];   // [2][kNXV][kThreads + 2] double
    double(*const row_buf)[kThreads + 2] = reinterpret_cast<double(*)[kThreads + 2]>(march_dyn);
    const int nx = a.nx, ny = a.ny;
    const int tid = threadIdx.x;
    const int x = blockIdx.x * blockDim.x + tid;
    const bool active = x < nx;
    const int R = (ny + gridDim.y - 1) / gridDim.y;
    const int y0 = blockIdx.y * R;
    const int y1 = y0 + R < ny ? y0 + R : ny;
    if (y0 >= y1) return;                             // the same for the whole block
    const int last = (nx - (int)(blockIdx.x * blockDim.x) < (int)blockDim.x
                          ? nx - (int)(blockIdx.x * blockDim.x) : (int)blockDim.x) - 1;   // last active thread
    const size_t P = (size_t)nx * ny;
    const int xc = active ? x : nx - 1;               // inactive threads only pass the barriers
    const int xm2 = neighbour_near(xc - 2, nx, a.bc_x), xm1 = neighbour_near(xc - 1, nx, a.bc_x);
    const int xp1 = neighbour_near(xc + 1, nx, a.bc_x), xp2 = neighbour_near(xc + 2, nx, a.bc_x);

    // prologue: U_{y0} and N_{y0 - 1} for s = +1, N_{y0} for s = -1
    if (active) {
        const size_t r0 = (size_t)y0 * nx + x;
        const size_t rm1 = (size_t)neighbour_near(y0 - 1, ny, a.bc_y) * nx + x;
        const size_t rm2 = (size_t)neighbour_near(y0 - 2, ny, a.bc_y) * nx + x;
        const size_t rp1 = (size_t)neighbour_near(y0 + 1, ny, a.bc_y) * nx + x;
#pragma unroll
        for (int k = 0; k < kNY; ++k) {
            const int i = yvel(k);
            const double *gp = g + i * P;
            const double f0 = __ldg(gp + r0), fm1 = __ldg(gp + rm1);
            if (diry(i) > 0) {
                const double u = f0 - fm1;                    // U_{y0}
                const double um = fm1 - __ldg(gp + rm2);      // U_{y0-1}
                carry_u[k][tid] = u;
                carry_n[k][tid] = minmod(u, um);          // N_{y0-1}
            } else {
                const double u = f0 - __ldg(gp + rp1);        // U_{y0}
                const double um = fm1 - f0;                   // U_{y0-1}
                carry_u[k][tid] = u;
                carry_n[k][tid] = minmod(um, u);          // N_{y0}
            }
        }
    }

    for (int y = y0; y < y1; ++y) {
        const size_t row = (size_t)y * nx;
        const size_t c = row + xc;
        // row y writes buffer y & 1; its readers have passed the next row's barrier
        // before row y + 2 writes the same buffer again
        double(*const row_u)[kThreads + 2] = row_buf + (y & 1) * kNXV;
        double fs[kNV], o[kNV];
        if (active) {
#pragma unroll
            for (int i = 0; i < kNV; ++i) fs[i] = __ldg(g + i * P + c);
            double heq[kNV];
            stage_equilibrium(a, fs, heq, flag);
            int k = 0;
#pragma unroll
            for (int i = 0; i < kNV; ++i) {
                o[i] = fma(a.a_self, fs[i], heq[i]);
                if (kBase) o[i] = fma(a.a_base, base[i * P + c], o[i]);
                if (dirx(i) != 0) {
                    const double *gp = g + i * P + row;
                    const double u1 = __ldg(gp + (dirx(i) > 0 ? xm1 : xp1));
                    row_u[k][tid + 1] = fs[i] - u1;            // U at x: the upwind-ordered a of nnd()
                    ++k;
                }
            }
        }
        {
            // Halo of the row buffer: U_{x-1} left of the block and U_{x+1} right of it (the
            // e or b of nnd() of the edge cells).  One branch taken by the edge threads only,
            // so the other warps do not issue these instructions.
            if (active && tid == 0) {
                int k = 0;
#pragma unroll
                for (int i = 0; i < kNV; ++i) {
                    if (dirx(i) == 0) continue;
                    const double *gp = g + i * P + row;
                    row_u[k][0] = dirx(i) > 0 ? __ldg(gp + xm1) - __ldg(gp + xm2) : __ldg(gp + xm1) - fs[i];
                    ++k;
                }
            }
            if (active && tid == last) {
                int k = 0;
#pragma unroll
                for (int i = 0; i < kNV; ++i) {
                    if (dirx(i) == 0) continue;
                    const double *gp = g + i * P + row;
                    row_u[k][last + 2] = dirx(i) > 0 ? __ldg(gp + xp1) - fs[i] : __ldg(gp + xp1) - __ldg(gp + xp2);
                    ++k;
                }
            }
            __syncthreads();
            if (active) {
                int k = 0;
#pragma unroll
                for (int i = 0; i < kNV; ++i) {
                    if (dirx(i) == 0) continue;
                    const int s = dirx(i);
                    const double av = row_u[k][tid + 1];              // c - u1
                    const double bv = row_u[k][tid + 1 + s];          // d1 - c
                    const double ev = row_u[k][tid + 1 - s];          // u1 - u2
                    const double t = minmod(bv, av) - minmod(av, ev);
                    o[i] = fma(-a.lx[i >> 2], fma(0.5, t, av), o[i]);
                    ++k;
                }
            }
        }
        if (active) {
            const size_t rp1 = (size_t)neighbour_near(y + 1, ny, a.bc_y) * nx + x;
            const size_t rp2 = (size_t)neighbour_near(y + 2, ny, a.bc_y) * nx + x;
#pragma unroll
            for (int k = 0; k < kNY; ++k) {
                const int i = yvel(k);
                const double *gp = g + i * P;
                const double u = carry_u[k][tid];
                const double n = carry_n[k][tid];
                double t;
                if (diry(i) > 0) {
                    const double un = __ldg(gp + rp1) - fs[i];                  // U_{y+1}
                    const double nn = minmod(un, u);                            // N_y
                    t = nn - n;                                             // N_y - N_{y-1}
                    carry_u[k][tid] = un;
                    carry_n[k][tid] = nn;
                } else {
                    const double un = __ldg(gp + rp1) - __ldg(gp + rp2);        // U_{y+1}
                    const double nn = minmod(u, un);                            // N_{y+1}
                    t = n - nn;                                             // N_y - N_{y+1}
                    carry_u[k][tid] = un;
                    carry_n[k][tid] = nn;
                }
                o[i] = fma(-a.ly[i >> 2], fma(0.5, t, u), o[i]);
            }
#pragma unroll
            for (int i = 0; i < kNV; ++i) out[i * P + c] = o[i];
        }
    }
}

template <bool kBase>
void *stage_func(bool march, bool flat)
{
    if (march) return (void *)stage_march_kernel<kBase>;
    return flat ? (void *)stage_kernel<kBase, true> : (void *)stage_kernel<kBase, false>;
}

}  // namespace

StageLaunch double_stage_launch_config(const StageArgs &a, bool with_base, int sm_count, bool allow_march,
                                       bool allow_split)
{
    StageLaunch L;
    const bool flat = a.ny == 1;
    const size_t cells = (size_t)a.nx * a.ny;
    if (allow_split && flat && a.nx <= 8192) {
        // short tubes: four threads per cell shorten the dependent chain of a stage (8.8
        // against 10.0 us at 8192 cells, 16.3 against 10.7 us at 16384)
        L.func = split_flat_func(with_base);
        L.block = dim3(kSplitFlatThreads, 1, 1);
        L.grid = dim3((unsigned)((4 * (size_t)a.nx + kSplitFlatThreads - 1) / kSplitFlatThreads), 1, 1);
        return L;
    }
    const unsigned xblocks = (unsigned)((a.nx + kThreads - 1) / kThreads);
    // Row-marching kernel when runs of at least 8 rows still give two full waves of
    // blocks; runs grow to 32 rows while at least 8 waves remain; on smaller grids runs of
    // 4 or 2 rows if they give two waves.
    const size_t wave = (size_t)sm_count * kMinBlocks;
    int R = 8;
    while (R < 32 && (size_t)xblocks * ((a.ny + 2 * R - 1) / (2 * R)) >= 8 * wave) R *= 2;
    bool march = allow_march && !flat && a.ny >= 16 && (size_t)xblocks * ((a.ny + 7) / 8) >= 2 * wave;
    for (int r = 4; allow_march && !march && !flat && a.ny >= 16 && r >= 2; r /= 2) {
        if ((size_t)xblocks * ((a.ny + r - 1) / r) >= 2 * wave) {
            march = true;
            R = r;
        }
    }
    L.func = with_base ? stage_func<true>(march, flat) : stage_func<false>(march, flat);
    if (march) {
        // the double-buffered x row buffer
        L.smem = kMarchRowBytes;
        if (cudaFuncSetAttribute(L.func, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)L.smem) != cudaSuccess)
            cudaGetLastError();   // the launch then reports the error
        L.block = dim3(kThreads, 1, 1);
        const unsigned yblocks = (unsigned)((a.ny + R - 1) / R);
        L.grid = dim3(xblocks, yblocks < 65535 ? yblocks : 65535, 1);
        return L;
    }
    // Small grids: narrower blocks so that more SMs share the cells.
    int threads = kThreads;
    while (threads > 32 && cells < (size_t)sm_count * threads * 2) threads >>= 1;
    L.block = dim3(threads, 1, 1);
    L.grid = dim3((a.nx + threads - 1) / threads, a.ny < 65535 ? a.ny : 65535, 1);
    return L;
}

}  // namespace cdbm
