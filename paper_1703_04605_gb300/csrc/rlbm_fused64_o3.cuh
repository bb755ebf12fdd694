// FP64 third-order equilibrium of a folded stencil, per reflection orbit (shared
// by the step, rlbm_fused64_o3.cu, and the init, rlbm_io_o3.cu).
#pragma once

#include "rlbm_fused64.cuh"
#include "rlbm_o3.cuh"

namespace rlbm {

// Parity classes of the centred monomials (kO3Mono order).
using O3EE = std::integer_sequence<int, 0, 1, 6, 7, 9, 10, 11, 17>;   // even in p_x and p_y
using O3OE = std::integer_sequence<int, 2, 4, 13, 15, 18>;            // odd in p_x only
using O3EO = std::integer_sequence<int, 3, 5, 14, 16, 19>;            // odd in p_y only
using O3OO = std::integer_sequence<int, 8, 12>;                       // odd in both

template <int... L>
__device__ __forceinline__ double sum64(std::integer_sequence<int, L...>, const double* w, const double (&e)[kO3Mono],
                                        double acc) {
  ((acc = fma(w[1 + L], e[L], acc)), ...);
  return acc;
}

__device__ __forceinline__ void deviations64(const FusedO364Params& p, const Macro<double>& o, double (&e)[kO3Mono]) {
  o3_deviations<double>(p.sc.mbar, p.c, o.n, o.U0, o.Ux, o.Uy, o.dU, o.dR, o.T - 1.0, o.T, o.R, e, p.sc.inv_m);
}

// E, X, Y, Z of orbit K (rlbm_fused64.cuh), dn the density above the reference.
template <class Def, int K>
__device__ __forceinline__ void orbit_equilibrium_o3(const double* w, const double (&e)[kO3Mono], double dn, double& E,
                                                     double& X, double& Y, double& Z) {
  constexpr int kind = Def::O.kind[K];
  E = sum64(O3EE{}, w, e, w[0] * dn);
  X = Y = Z = 0.0;
  if constexpr (kind == 2 || kind == 4) X = sum64(O3OE{}, w, e, 0.0);
  if constexpr (kind == 3 || kind == 4) Y = sum64(O3EO{}, w, e, 0.0);
  if constexpr (kind == 4) Z = sum64(O3OO{}, w, e, 0.0);
}

}  // namespace rlbm
