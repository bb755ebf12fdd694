// FP64 third-order equilibrium of a folded stencil, per reflection orbit (shared
// by the step, rlbm_fused64_o3.cu, and the init, rlbm_io_o3.cu).
#pragma once

#include "rlbm_fused64.cuh"
#include "rlbm_o3.cuh"

namespace rlbm {

// acc + sum of w[1 + W_k] e[E_k]
template <int... W, int... E>
__device__ __forceinline__ double sum64(MonoList<W...>, MonoList<E...>, const double* w, const double (&e)[kO3Mono],
                                        double acc) {
  ((acc = fma(w[1 + W], e[E], acc)), ...);
  return acc;
}

__device__ __forceinline__ void deviations64(const FusedO364Params& p, const Macro<double>& o, double (&e)[kO3Mono]) {
  o3_deviations<double>(p.sc.mbar, p.c, o.n, o.U0, o.Ux, o.Uy, o.dU, o.dR, o.T - 1.0, o.T, o.R, e, p.sc.inv_m);
}

// E, X, Y, Z (rlbm_fused64.cuh) of the orbits (a_x, a_y) with a_x >= a_y and of
// their exchanged ones, handed to use<K>(E, X, Y, Z); dn: the density above the
// reference.
template <class Def, int K, class Use>
__device__ __forceinline__ void orbit_equilibrium_o3(const double* w, const double (&e)[kO3Mono], double dn,
                                                     const Use& use) {
  constexpr int ax = Def::O.ax[K], ay = Def::O.ay[K], KX = exchanged_orbit<Def, K>();
  static_assert(KX >= 0, "full-symmetric groups are closed under exchange");
  const double both = sum64(O3Both{}, O3Both{}, w, e, w[0] * dn);
  double X = 0.0, Y = 0.0, Z = 0.0;
  if constexpr (ax != 0 && ay != 0) Z = sum64(O3OddXY{}, O3OddXY{}, w, e, 0.0);
  if constexpr (ax != 0) X = sum64(O3OddX{}, O3OddX{}, w, e, 0.0);
  if constexpr (ay != 0) Y = sum64(O3OddY{}, O3OddY{}, w, e, 0.0);
  use.template at<Def, K>(sum64(O3Even{}, O3Even{}, w, e, both), X, Y, Z);
  if constexpr (KX != K) {
    X = Y = 0.0;
    if constexpr (ay != 0) X = sum64(O3OddY{}, O3OddX{}, w, e, 0.0);
    if constexpr (ax != 0) Y = sum64(O3OddX{}, O3OddY{}, w, e, 0.0);
    use.template at<Def, KX>(sum64(O3EvenX{}, O3Even{}, w, e, both), X, Y, Z);
  }
}

// All orbits.
template <class Def, class P, class Use, int... Ks>
__device__ __forceinline__ void all_orbits_o3(MonoList<Ks...>, const P& p, const double (&e)[kO3Mono], double dn,
                                              const Use& use) {
  (
      [&] {
        if constexpr (Def::O.ax[Ks] >= Def::O.ay[Ks]) orbit_equilibrium_o3<Def, Ks>(p.ow[Ks], e, dn, use);
      }(),
      ...);
}

}  // namespace rlbm
