// Persistent cluster kernel for small 1-D grids (Ny = 1): a whole run of Eq. (1) in
// one launch.
//
// On a grid of a few hundred or thousand cells a stage launch does a few
// microseconds of work, and a step of two launches is bound by launch latency.
// Here one thread-block cluster of C <= 16 CTAs keeps the whole state in shared
// memory for the whole run: CTA r owns the cells [r chunk, (r + 1) chunk) of both
// stage buffers, reads the stencil halo of its edge cells from the neighbouring
// CTAs' shared memory (distributed shared memory of the cluster), and the stages
// are separated by the cluster barrier, a hardware barrier over the co-scheduled
// CTAs (no software spin-wait).  In single precision the per-cell arithmetic is
// that of the flat stage kernel in the same order, so the result is the same bit for
// bit; the df64 variant splits a cell over two threads (split_stage_df), the FP64 variant
// over 16 (cell16 of cdbm_stage_exact.cuh, the arithmetic of its stage launches).
#include <cooperative_groups.h>

#include "cdbm_stage.cuh"
#include "cdbm_stage_exact.cuh"

namespace cg = cooperative_groups;

namespace cdbm {

namespace {

constexpr int kMaxCluster = 16;

// Value of velocity i at global cell gx (an index already mapped by neighbour())
// from the stage buffer `buf` ([16][chunk] in every CTA of the cluster).
template <typename TS>
__device__ __forceinline__ TS cluster_value(const cg::cluster_group &cl, const TS *buf, int chunk, int rank,
                                            int i, int gx)
{
    const int r = gx / chunk;
    const TS *p = r == rank ? buf : cl.map_shared_rank(buf, (unsigned)r);
    return p[i * chunk + (gx - r * chunk)];
}

// One stage over this CTA's cells: dst = a_base base + a_self src + gamma h f_eq(src)
// - sum l D(src), the operations of stage_kernel<TS, kBase, true, kEq> per cell.  All
// stencil values (and the base) are gathered into registers before the first store,
// so the loads of the edge cells from the neighbouring CTAs overlap instead of each
// waiting behind a store the compiler cannot prove independent.
template <bool kBase, int kEq>
__device__ __forceinline__ void cluster_stage(const cg::cluster_group &cl, const float *src, const float *base, float *dst,
                                              const StageArgs &a, int chunk, int rank, int x0, int len,
                                              unsigned *flag)
{
    constexpr int kNX = 12;                            // velocities with an x component
    const int nx = a.nx;
    for (int lx = threadIdx.x; lx < len; lx += blockDim.x) {
        const int gx = x0 + lx;
        float fs[kNV], bs[kNV], up2[kNX], up1[kNX], dn1[kNX];
#pragma unroll
        for (int i = 0; i < kNV; ++i) {
            fs[i] = src[i * chunk + lx];
            if (kBase) bs[i] = base[i * chunk + lx];
        }
        if (lx >= 2 && lx + 2 < len) {                 // stencil inside this CTA, no wrap
            int k = 0;
#pragma unroll
            for (int i = 0; i < kNV; ++i) {
                if (dirx(i) == 0) continue;
                const float *p = src + i * chunk + lx;
                up2[k] = p[dirx(i) > 0 ? -2 : 2];
                up1[k] = p[dirx(i) > 0 ? -1 : 1];
                dn1[k] = p[dirx(i) > 0 ? 1 : -1];
                ++k;
            }
        } else {
            const int xm2 = neighbour_near(gx - 2, nx, a.bc_x), xm1 = neighbour_near(gx - 1, nx, a.bc_x);
            const int xp1 = neighbour_near(gx + 1, nx, a.bc_x), xp2 = neighbour_near(gx + 2, nx, a.bc_x);
            int k = 0;
#pragma unroll
            for (int i = 0; i < kNV; ++i) {
                if (dirx(i) == 0) continue;
                up2[k] = cluster_value(cl, src, chunk, rank, i, dirx(i) > 0 ? xm2 : xp2);
                up1[k] = cluster_value(cl, src, chunk, rank, i, dirx(i) > 0 ? xm1 : xp1);
                dn1[k] = cluster_value(cl, src, chunk, rank, i, dirx(i) > 0 ? xp1 : xm1);
                ++k;
            }
        }
        float heq[kNV];
        stage_equilibrium<kEq>(a, fs, heq, flag);
        int k = 0;
#pragma unroll
        for (int i = 0; i < kNV; ++i) {
            float o = fmaf(a.a_self_f, fs[i], heq[i]);
            if (kBase) o = fmaf(a.a_base_f, bs[i], o);
            if (dirx(i) != 0) {
                o = fmaf(-a.lx_f[i >> 2], nnd(up2[k], up1[k], fs[i], dn1[k]), o);
                ++k;
            }
            dst[i * chunk + lx] = o;
        }
    }
}

template <int kEq>
__global__ void __launch_bounds__(256) small1d_kernel(float *f, int nsteps, const StageArgs a0, const StageArgs a1,
                                                      unsigned *flag, int chunk)
{
    extern __shared__ __align__(16) unsigned char smem_raw[];
    float *s0 = reinterpret_cast<float *>(smem_raw);     // state f^n, [16][chunk]
    float *s1 = s0 + kNV * chunk;                     // stage buffer
    const cg::cluster_group cl = cg::this_cluster();
    const int rank = (int)cl.block_rank();
    const int nx = a0.nx;
    const int x0 = rank * chunk;
    const int len = nx - x0 < chunk ? (nx - x0 > 0 ? nx - x0 : 0) : chunk;
    for (int k = threadIdx.x; k < kNV * len; k += blockDim.x) {
        const int i = k / len, lx = k - i * len;
        s0[i * chunk + lx] = f[(size_t)i * nx + x0 + lx];
    }
    cl.sync();
    for (int s = 0; s < nsteps; ++s) {
        cluster_stage<false, kEq>(cl, s0, nullptr, s1, a0, chunk, rank, x0, len, flag);
        cl.sync();
        cluster_stage<true, kEq>(cl, s1, s0, s0, a1, chunk, rank, x0, len, flag);
        cl.sync();
    }
    for (int k = threadIdx.x; k < kNV * len; k += blockDim.x) {
        const int i = k / len, lx = k - i * len;
        f[(size_t)i * nx + x0 + lx] = s0[i * chunk + lx];
    }
}

// FP64 stage in the cluster, a cell on 16 threads (cell16): warp w of the CTA has
// the velocity cell16_velocity(w mod 16) of the cells 32 (w / 16) .. + 31 of the CTA's chunk.
template <bool kBase>
__device__ __forceinline__ void cluster_stage16(const cg::cluster_group &cl, const double *src, const double *base,
                                                double *dst, const StageArgs &a, Cells16 *s, int chunk, int rank, int x0,
                                                int len, unsigned *flag)
{
    const int w = threadIdx.x >> 5, i = cell16_velocity(w & 15), set = w >> 4, nx = a.nx;
    const int l0 = 32 * set + (int)(threadIdx.x & 31);
    const bool live = l0 < len;
    const int lx = live ? l0 : len - 1;               // idle lanes mirror the last cell
    const int gx = x0 + lx;
    const double c = src[i * chunk + lx];
    Stencil v = {c, c, c, c, 0, 0, 0, kBase ? base[i * chunk + lx] : 0.0};
    const int d = dirx(i);
    if (d != 0) {
        if (lx >= 2 && lx + 2 < len) {
            const double *p = src + i * chunk + lx;
            v.x2 = p[-2 * d];
            v.x1 = p[-d];
            v.xd = p[d];
        } else {
            v.x2 = cluster_value(cl, src, chunk, rank, i, neighbour_near(gx - 2 * d, nx, a.bc_x));
            v.x1 = cluster_value(cl, src, chunk, rank, i, neighbour_near(gx - d, nx, a.bc_x));
            v.xd = cluster_value(cl, src, chunk, rank, i, neighbour_near(gx + d, nx, a.bc_x));
        }
    }
    const double o = cell16<true, kBase, true>(a, s[set], w & 15, set, i, v, flag);
    if (live) dst[i * chunk + lx] = o;
}

__global__ void __launch_bounds__(1024) small1d_double_kernel(double *f, int nsteps, const __grid_constant__ StageArgs a0,
                                                          const __grid_constant__ StageArgs a1, unsigned *flag, int chunk)
{
    extern __shared__ __align__(16) unsigned char smem_raw[];
    double *s0 = reinterpret_cast<double *>(smem_raw);
    double *s1 = s0 + kNV * chunk;
    Cells16 *cells = reinterpret_cast<Cells16 *>(s1 + kNV * chunk);
    const cg::cluster_group cl = cg::this_cluster();
    const int rank = (int)cl.block_rank();
    const int nx = a0.nx;
    const int x0 = rank * chunk;
    const int len = nx - x0 < chunk ? (nx - x0 > 0 ? nx - x0 : 0) : chunk;
    for (int k = threadIdx.x; k < kNV * len; k += blockDim.x) {
        const int i = k / len, lx = k - i * len;
        s0[i * chunk + lx] = f[(size_t)i * nx + x0 + lx];
    }
    cl.sync();
    for (int s = 0; s < nsteps; ++s) {
        cluster_stage16<false>(cl, s0, nullptr, s1, a0, cells, chunk, rank, x0, len, flag);
        cl.sync();
        cluster_stage16<true>(cl, s1, s0, s0, a1, cells, chunk, rank, x0, len, flag);
        cl.sync();
    }
    for (int k = threadIdx.x; k < kNV * len; k += blockDim.x) {
        const int i = k / len, lx = k - i * len;
        f[(size_t)i * nx + x0 + lx] = s0[i * chunk + lx];
    }
}

// df64 variant with a cell split over two threads: thread h of the pair takes the
// velocity groups 2h (axis) and 2h + 1 (diagonal), so both threads run the same
// instruction sequence.  The pair exchanges its group components by warp shuffles,
// both form the moments, primitives and raw-moment factors (df_scalars, the same
// operations), and each builds and updates only its own eight velocities.  Every
// value goes through the operations of the one-thread kernel in the same order, so
// the result is the same bit for bit; the dependent chain of a stage is about a third
// shorter, and that chain sets the time of a stage on these grids.
template <bool kBase>
__device__ __forceinline__ void split_stage_df(const cg::cluster_group &cl, const float *src, const float *base,
                                               float *dst, const StageArgs &a, int chunk, int rank, int x0, int len,
                                               unsigned *flag)
{
    const int t = threadIdx.x;
    const int h = t & 1;                              // groups 2h and 2h + 1 of the cell
    const int lx0 = t >> 1;
    const bool live = lx0 < len;
    const int lx = live ? lx0 : len - 1;              // idle threads mirror the last cell
    const int gx = x0 + lx;
    const int nx = a.nx;
    float q[8], bs[8], up2[8], up1[8], dn1[8];
#pragma unroll
    for (int j = 0; j < 8; ++j) {
        q[j] = src[(8 * h + j) * chunk + lx];
        bs[j] = kBase ? base[(8 * h + j) * chunk + lx] : 0.0f;
    }
    const bool inner = lx >= 2 && lx + 2 < len;
    const int xm2 = neighbour_near(gx - 2, nx, a.bc_x), xm1 = neighbour_near(gx - 1, nx, a.bc_x);
    const int xp1 = neighbour_near(gx + 1, nx, a.bc_x), xp2 = neighbour_near(gx + 2, nx, a.bc_x);
#pragma unroll
    for (int j = 0; j < 8; ++j) {
        const int i = 8 * h + j;
        const int sx = dirx(j);                       // dirx depends on i mod 8 only
        if (sx == 0) {
            up2[j] = up1[j] = dn1[j] = 0.0f;
        } else if (inner) {
            const float *p = src + i * chunk + lx;
            up2[j] = p[sx > 0 ? -2 : 2];
            up1[j] = p[sx > 0 ? -1 : 1];
            dn1[j] = p[sx > 0 ? 1 : -1];
        } else {
            up2[j] = cluster_value(cl, src, chunk, rank, i, sx > 0 ? xm2 : xp2);
            up1[j] = cluster_value(cl, src, chunk, rank, i, sx > 0 ? xm1 : xp1);
            dn1[j] = cluster_value(cl, src, chunk, rank, i, sx > 0 ? xp1 : xm1);
        }
    }
    const DFConsts &D = a.d;
    df a0, ax, ay, b0, bx, by;                        // own axis group 2h, diagonal group 2h + 1
    df_group_components(0, q, a0, ax, ay);
    df_group_components(1, q + 4, b0, bx, by);
    auto other = [](float v) { return __shfl_xor_sync(0xffffffffu, v, 1); };
    const df pa0 = {other(a0.hi), other(a0.lo)}, pax = {other(ax.hi), other(ax.lo)}, pay = {other(ay.hi), other(ay.lo)};
    const df pb0 = {other(b0.hi), other(b0.lo)}, pbx = {other(bx.hi), other(bx.lo)}, pby = {other(by.hi), other(by.lo)};
    df s0[4], sx4[4], sy4[4];
    s0[0] = h ? pa0 : a0;   sx4[0] = h ? pax : ax;   sy4[0] = h ? pay : ay;
    s0[1] = h ? pb0 : b0;   sx4[1] = h ? pbx : bx;   sy4[1] = h ? pby : by;
    s0[2] = h ? a0 : pa0;   sx4[2] = h ? ax : pax;   sy4[2] = h ? ay : pay;
    s0[3] = h ? b0 : pb0;   sx4[3] = h ? bx : pbx;   sy4[3] = h ? by : pby;
    const DFScalars<float> c = df_scalars(D.m, D.r, s0, sx4, sy4, (live && h == 0) ? flag : nullptr);
    float heq[8];
    df_group_equilibrium(2 * h, D.b, D.r, c, heq);
    df_group_equilibrium(2 * h + 1, D.b, D.r, c, heq + 4);
    float o[8];
#pragma unroll
    for (int j = 0; j < 8; ++j) {
        o[j] = fmaf(a.a_self_f, q[j], heq[j]);
        if (kBase) o[j] = fmaf(a.a_base_f, bs[j], o[j]);
        if (dirx(j) != 0) o[j] = fmaf(-a.lx_f[2 * h + (j >> 2)], nnd(up2[j], up1[j], q[j], dn1[j]), o[j]);
    }
    if (live) {
#pragma unroll
        for (int j = 0; j < 8; ++j) dst[(8 * h + j) * chunk + lx] = o[j];
    }
}

__global__ void __launch_bounds__(256) small1d_split_df_kernel(float *f, int nsteps, const StageArgs a0,
                                                               const StageArgs a1, unsigned *flag, int chunk)
{
    extern __shared__ __align__(16) unsigned char smem_raw[];
    float *s0 = reinterpret_cast<float *>(smem_raw);
    float *s1 = s0 + kNV * chunk;
    const cg::cluster_group cl = cg::this_cluster();
    const int rank = (int)cl.block_rank();
    const int nx = a0.nx;
    const int x0 = rank * chunk;
    const int len = nx - x0 < chunk ? (nx - x0 > 0 ? nx - x0 : 0) : chunk;
    for (int k = threadIdx.x; k < kNV * len; k += blockDim.x) {
        const int i = k / len, lx = k - i * len;
        s0[i * chunk + lx] = f[(size_t)i * nx + x0 + lx];
    }
    cl.sync();
    for (int s = 0; s < nsteps; ++s) {
        split_stage_df<false>(cl, s0, nullptr, s1, a0, chunk, rank, x0, len, flag);
        cl.sync();
        split_stage_df<true>(cl, s1, s0, s0, a1, chunk, rank, x0, len, flag);
        cl.sync();
    }
    for (int k = threadIdx.x; k < kNV * len; k += blockDim.x) {
        const int i = k / len, lx = k - i * len;
        f[(size_t)i * nx + x0 + lx] = s0[i * chunk + lx];
    }
}

template <int kEq>
void *small1d_func() { return (void *)small1d_kernel<kEq>; }

constexpr int kSplitDfMaxChunk = 128;     // two threads per cell within 256 threads

void *small1d_func_of(int prec, int chunk)
{
    if (prec == CDBM_FP32_DF64)
        return chunk <= kSplitDfMaxChunk ? (void *)small1d_split_df_kernel : small1d_func<kEqDF>();
    if (prec == CDBM_FP32_DEV) return small1d_func<kEqF32>();
    if (prec == CDBM_FP32_BULK) return small1d_func<kEqDouble>();
    return (void *)small1d_double_kernel;
}

}  // namespace

Small1D small1d_config(const StageArgs &a, int prec)
{
    Small1D L{};
    if (a.ny != 1 || a.nx < 1) return L;
    // Used while each CTA holds at most two warps' worth of cells (FP64) or eight
    // (single precision).  Measured per stage on 64-4096-cell tubes: single
    // precision with the df64 equilibrium 2.7-3.2 us against 4.3-5.8 us for one
    // launch per stage; FP64 4.0-5.2 us on 500-1000 cells, against 4.6 us per launch on
    // all SMs: 1024 threads hold 64 cells.
    const int per_cta_max = prec == CDBM_FP64 ? 64 : 256;
    const int C = (a.nx + per_cta_max - 1) / per_cta_max > kMaxCluster ? 0 : kMaxCluster;
    if (C == 0) return L;
    int cluster = a.nx < C ? a.nx : C;
    const int chunk = (a.nx + cluster - 1) / cluster;
    cluster = (a.nx + chunk - 1) / chunk;            // no empty CTAs
    const int sets = (chunk + 31) / 32;               // FP64: 32 cells on 16 warps each
    const size_t smem = 2 * kNV * (size_t)chunk * storage_bytes(prec) +
                        (prec == CDBM_FP64 ? sets * sizeof(Cells16) : 0);
    // df64: two threads per cell (split_stage_df, up to kSplitDfMaxChunk cells), all cells
    // of the CTA in one pass
    const int per_cell = prec == CDBM_FP32_DF64 && chunk <= kSplitDfMaxChunk ? 2 : 1;
    int threads = ((per_cell * chunk + 31) / 32) * 32;
    if (threads > 256) threads = 256;
    if (prec == CDBM_FP64) threads = 512 * sets;
    void *func = small1d_func_of(prec, chunk);
    if (cluster > 8 && cudaFuncSetAttribute(func, cudaFuncAttributeNonPortableClusterSizeAllowed, 1) != cudaSuccess) {
        cudaGetLastError();
        return L;
    }
    if (smem > 48 * 1024 &&
        cudaFuncSetAttribute(func, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)smem) != cudaSuccess) {
        cudaGetLastError();
        return L;
    }
    cudaLaunchConfig_t cfg = {};
    cudaLaunchAttribute attr[1];
    attr[0].id = cudaLaunchAttributeClusterDimension;
    attr[0].val.clusterDim.x = (unsigned)cluster;
    attr[0].val.clusterDim.y = 1;
    attr[0].val.clusterDim.z = 1;
    cfg.gridDim = dim3((unsigned)cluster, 1, 1);
    cfg.blockDim = dim3((unsigned)threads, 1, 1);
    cfg.dynamicSmemBytes = smem;
    cfg.attrs = attr;
    cfg.numAttrs = 1;
    int active = 0;
    if (cudaOccupancyMaxActiveClusters(&active, func, &cfg) != cudaSuccess || active < 1) {
        cudaGetLastError();
        return L;
    }
    L.ok = true;
    L.func = func;
    L.cluster = cluster;
    L.chunk = chunk;
    L.threads = threads;
    L.smem = smem;
    return L;
}

cudaError_t launch_small1d(const Small1D &L, void *f, int nsteps, const StageArgs &a0, const StageArgs &a1,
                           unsigned *flag, cudaStream_t s)
{
    cudaLaunchConfig_t cfg = {};
    cudaLaunchAttribute attr[1];
    attr[0].id = cudaLaunchAttributeClusterDimension;
    attr[0].val.clusterDim.x = (unsigned)L.cluster;
    attr[0].val.clusterDim.y = 1;
    attr[0].val.clusterDim.z = 1;
    cfg.gridDim = dim3((unsigned)L.cluster, 1, 1);
    cfg.blockDim = dim3((unsigned)L.threads, 1, 1);
    cfg.dynamicSmemBytes = L.smem;
    cfg.stream = s;
    cfg.attrs = attr;
    cfg.numAttrs = 1;
    int chunk = L.chunk;
    void *args[] = {&f, &nsteps, (void *)&a0, (void *)&a1, &flag, &chunk};
    return cudaLaunchKernelExC(&cfg, L.func, args);
}

}  // namespace cdbm
