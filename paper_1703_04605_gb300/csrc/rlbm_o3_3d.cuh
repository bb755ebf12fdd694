// Device form of the thirty moment deviations of the third-order equilibrium
// on native 3D lattices (shared by rlbm_kernels3d.cu and rlbm_fused3d_o3.cu).
#pragma once

#include <utility>

#include "rlbm_o3_3d.h"

namespace rlbm {

// Site quantities of the third-order equilibrium (see rlbm_o3_3d.h and the
// 2D form in rlbm_o3.cuh): with h = m R + 4T, A3 = m^2 + 6 T h, B3 = -T h,
// the deviations from rest at T_R of the moments (per unit density) of
// t^a p^s1 ... p^sr are
//   r = 0:  a = 0: dR/m           a = 1: dU - c dR/m
//   r = 1:  a = 0: U_s            a = 1: U_s (h U0 - c)
//   r = 2:  a = 0: h U_s U_s' + d_ss' dT
//           a = 1: (A3 U0 - c h) U_s U_s' + d_ss' (T (h U0 - c) - (h_r - c))
//   r = 3:  A3 U_s U_s' U_s'' + T h (d_ss' U_s'' + d_ss'' U_s' + d_s's'' U_s)
// (Eq. 4-6, 28-29, 43-44; eta^ab = -delta_ab on the spatial indices).
template <typename R>
struct O3Site3 {
  R n, U[4], dU, dRm, dT, c, h, Th, Am, hU, sdev, q;   // dRm = dR/m
};

template <int A, int I, int J, int K, typename R>
__device__ __forceinline__ R o3dev3(const O3Site3<R>& s) {
  constexpr int r = I + J + K;
  constexpr int i1 = I > 0 ? 1 : (J > 0 ? 2 : 3);
  constexpr int i2 = I > 1 ? 1 : (I + J > 1 ? 2 : 3);
  constexpr int i3 = I > 2 ? 1 : (I + J > 2 ? 2 : 3);
  if constexpr (r == 0) {
    return A == 0 ? s.n * s.dRm : s.n * (s.dU - s.c * s.dRm);
  } else if constexpr (r == 1) {
    return A == 0 ? s.n * s.U[i1] : s.n * s.U[i1] * s.hU;
  } else if constexpr (r == 2) {
    const R uu = s.U[i1] * s.U[i2];
    if constexpr (A == 0) return s.n * (s.h * uu + (i1 == i2 ? s.dT : R(0)));
    else return s.n * (s.q * uu + (i1 == i2 ? s.sdev : R(0)));
  } else {
    R v = s.Am * s.U[i1] * s.U[i2] * s.U[i3];
    if constexpr (i1 == i2) v += s.Th * s.U[i3];
    if constexpr (i1 == i3) v += s.Th * s.U[i2];
    if constexpr (i2 == i3) v += s.Th * s.U[i1];
    return s.n * v;
  }
}

template <typename R, int... L>
__device__ __forceinline__ void o3_dev3_all(std::integer_sequence<int, L...>, const O3Site3<R>& s, R* e) {
  ((e[L] = o3dev3<kO3Exp3.e[L][0], kO3Exp3.e[L][1], kO3Exp3.e[L][2], kO3Exp3.e[L][3], R>(s)), ...);
}

}  // namespace rlbm
