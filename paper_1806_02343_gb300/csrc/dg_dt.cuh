// Timestep reductions shared by dg_kernels.cu and dg_2d.cu.
#pragma once
#include <cfloat>

#include "dg_ctx.h"

namespace dgmhd {

// positive doubles order as their bit patterns
__device__ __forceinline__ unsigned long long dbits(double x) { return (unsigned long long)__double_as_longlong(x); }
__device__ __forceinline__ double warp_min(double x) {
  for (int o = 16; o > 0; o >>= 1) x = fmin(x, __shfl_xor_sync(0xffffffffu, x, o));
  return x;
}

__device__ __forceinline__ void dt_init(DevScalars* sc) {
  sc->dt_bits = dbits(DBL_MAX);
  sc->dt64_bits = dbits(DBL_MAX);
  sc->smax_bits = 0ull;
}

__device__ __forceinline__ void dt_finalize(const Geom& g, const dg_mhd_params& p, DevScalars* sc, const double* dt_in,
                                            double* dt_out) {
  // the FP32 form's refined FP64 minimum where that pass ran, else the FP64 pass's minimum
  const double dt64 = __longlong_as_double((long long)sc->dt64_bits);
  double dt = dt_in ? *dt_in : (dt64 < DBL_MAX ? dt64 : __longlong_as_double((long long)sc->dt_bits));
  if (!(dt > 0.0) || !isfinite(dt) || dt >= DBL_MAX) {
    atomicOr(&sc->status, 1);
  }
  sc->dt = dt;
  sc->dt_step = dt;
  sc->dt32 = (float)dt;
  if (dt_out) *dt_out = dt;
  if (g.glm) {
    double ch = p.c_h_fixed > 0.0 ? p.c_h_fixed : p.cfl_glm / (2.0 * g.d + 1.0) * g.dx / (g.D * dt);
    sc->ch = ch;
    sc->ch32 = (float)ch;
    const double tau = fmax(p.c_r / ch, 3.0 * dt);
    sc->kappa = 1.0 / tau;
    sc->kappa32 = (float)sc->kappa;
    if (p.c_h_fixed > 0.0 && !dt_in) {
      const double smax = __longlong_as_double((long long)sc->smax_bits);
      if (ch < smax) atomicOr(&sc->status, 4);
    }
  }
}

}  // namespace dgmhd
