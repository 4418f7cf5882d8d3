// Per-cell pieces of a Runge-Kutta stage shared by the stage kernels: the stage
// coefficients in the storage precision and the scaled equilibrium of one cell.
#pragma once

#include "cdbm_f32dev.cuh"

namespace cdbm {

// How a stage forms the equilibrium: in double (CDBM_FP64, CDBM_FP32_BULK), in df64
// (CDBM_FP32_DF64) or in single precision on the deviations (CDBM_FP32_DEV).
constexpr int kEqDouble = 0, kEqDF = 1, kEqF32 = 2;

// gamma h f_eq of one cell of a single-precision state (minus gamma h F for
// CDBM_FP32_DEV): moments, primitives and equilibrium in double, all of it in df64
// (kEq = kEqDF) or in single precision on the moment deviations (kEq = kEqF32).
template <int kEq>
__device__ __forceinline__ void stage_equilibrium(const StageArgs &a, const float fs[kNV], float heq[kNV],
                                                  unsigned *flag)
{
    if constexpr (kEq == kEqF32) {
        f32_equilibrium(a.d.b, a.d.m, a.d.r, a.dp, fs, heq, flag);
    } else if constexpr (kEq == kEqDF) {
        df_equilibrium(a.d.b, a.d.m, a.d.r, fs, heq, flag);
    } else {
        double f[kNV];
#pragma unroll
        for (int i = 0; i < kNV; ++i) f[i] = widen_f32(fs[i]);
        const Prim s = primitives<true>(f, a.m, a.rhoF, a.EF, flag);
        double h[kNV];
        equilibrium<true>(a.eq, a.m, s.q.rho, s.q.E, s.q.jx, s.q.jy, s.ux, s.uy, s.ru2, s.jyuy, s.p, s.T, h, a.sF);
#pragma unroll
        for (int i = 0; i < kNV; ++i) heq[i] = narrow_f64(h[i]);
    }
}

}  // namespace cdbm
