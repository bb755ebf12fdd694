// FP64 site solve on native 3D lattices (rlbm_kernels3d.cu, rlbm_fused64_3d.cuh).
#pragma once

#include "rlbm_kernels.cuh"

namespace rlbm {

struct Macro3 {
  double n, U0, Ux, Uy, Uz, T, R, e;
};

// T from e/n = y (Eq. 28) by Newton iteration; returns T and R = K1/K2(m/T).
__device__ __forceinline__ void eos3(double y, const SiteConsts& sc, const double* __restrict__ rt64,
                                     double& T, double& R, unsigned& fl) {
  const double mb = sc.mbar;
  if (!(y > mb)) fl |= ERR_EOS;
  // g(T) = 3T + m R(m/T) - y is increasing and convex: Newton from the
  // non-relativistic estimate converges
  T = (y - mb) / (3.0 - 1.5 * (mb * mb) / (y * y));
#pragma unroll 1
  for (int it = 0; it < 40; ++it) {
    const double z = mb / T;
    R = ratio64(z, rt64, fl);
    const double dT = (3.0 * T + mb * R - y) / eos_slope<double>(R, z);
    T -= dT;
    if (!(T > 0.0)) {
      fl |= ERR_EOS;
      T = 1.0;
      break;
    }
    if (fabs(dT) < 1e-15 * T) break;
  }
  R = ratio64(mb / T, rt64, fl);
}

// Moments m = N0 Nx Ny Nz T00 T0x T0y T0z Txx Txy Txz Tyy Tyz Tzz -> n, U, T.
// Landau frame: Newton on v = U/U^0 for F(v) = T^0i - T^ij v_j - e v_i = 0
// with e = T^00 - T^0j v_j (the spatial rows of T^a_b U^b = e U^a).
__device__ __forceinline__ Macro3 solve3(const double* m, const SiteConsts& sc, const double* __restrict__ rt64,
                                         unsigned& fl) {
  const double T00 = m[4];
  const double T0[3] = {m[5], m[6], m[7]};
  const double Tij[3][3] = {{m[8], m[9], m[10]}, {m[9], m[11], m[12]}, {m[10], m[12], m[13]}};
  const double den = T00 + (m[8] + m[11] + m[13]) / 3.0;
  double v[3] = {T0[0] / den, T0[1] / den, T0[2] / den};
#pragma unroll 1
  for (int it = 0; it < 20; ++it) {
    const double e = T00 - T0[0] * v[0] - T0[1] * v[1] - T0[2] * v[2];
    double F[3], J[3][3];
#pragma unroll
    for (int a = 0; a < 3; ++a) {
      F[a] = T0[a] - Tij[a][0] * v[0] - Tij[a][1] * v[1] - Tij[a][2] * v[2] - e * v[a];
#pragma unroll
      for (int b = 0; b < 3; ++b) J[a][b] = -Tij[a][b] - (a == b ? e : 0.0) + v[a] * T0[b];
    }
    // J dv = F by Cramer's rule
    const double c00 = J[1][1] * J[2][2] - J[1][2] * J[2][1];
    const double c01 = J[1][2] * J[2][0] - J[1][0] * J[2][2];
    const double c02 = J[1][0] * J[2][1] - J[1][1] * J[2][0];
    const double det = J[0][0] * c00 + J[0][1] * c01 + J[0][2] * c02;
    const double id = 1.0 / det;
    const double d0 = (F[0] * c00 + J[0][1] * (F[2] * J[1][2] - F[1] * J[2][2]) +
                       J[0][2] * (F[1] * J[2][1] - F[2] * J[1][1])) * id;
    const double d1 = (J[0][0] * (F[1] * J[2][2] - F[2] * J[1][2]) + F[0] * c01 +
                       J[0][2] * (F[2] * J[1][0] - F[1] * J[2][0])) * id;
    const double d2 = (J[0][0] * (F[2] * J[1][1] - F[1] * J[2][1]) + J[0][1] * (F[1] * J[2][0] - F[2] * J[1][0]) +
                       F[0] * c02) * id;
    v[0] -= d0;
    v[1] -= d1;
    v[2] -= d2;
    if (fabs(d0) + fabs(d1) + fabs(d2) < 1e-15) break;
  }
  Macro3 o;
  const double v2 = v[0] * v[0] + v[1] * v[1] + v[2] * v[2];
  if (!(v2 < 1.0)) fl |= ERR_LANDAU;
  const double g = 1.0 / sqrt(1.0 - v2);
  o.U0 = g;
  o.Ux = g * v[0];
  o.Uy = g * v[1];
  o.Uz = g * v[2];
  o.e = T00 - T0[0] * v[0] - T0[1] * v[1] - T0[2] * v[2];
  o.n = g * (m[0] - v[0] * m[1] - v[1] * m[2] - v[2] * m[3]);
  if (!(o.n > 0.0)) fl |= ERR_DENSITY;
  eos3(o.e / o.n, sc, rt64, o.T, o.R, fl);
  return o;
}

}  // namespace rlbm
