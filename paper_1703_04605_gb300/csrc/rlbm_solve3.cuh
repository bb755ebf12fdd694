// Site solve of the compiled FP32 3D kernels (rlbm_fused3d.cu,
// rlbm_fused3d_o3.cu): the split arithmetic of split_solve (rlbm_fused.cuh)
// with three velocity components.
#pragma once

#include "rlbm_fused.cuh"

namespace rlbm {

struct SplitSite3 {
  float dg, U0, Ux, Uy, Uz, n, nd, Td, dR, R, T;
};

// M: deviation moments N0 Nx Ny Nz T00 T0x T0y T0z Txx Txy Txz Tyy Tyz Tzz;
// P: Fused3Params or Fused3O3Params.
template <class P>
__device__ __forceinline__ SplitSite3 split_solve3(const P& p, const float (&M)[14], unsigned& fl) {
  // Landau frame: FP32 Newton on the full moments
  float Mf[14];
#pragma unroll
  for (int k = 0; k < 14; ++k) Mf[k] = p.mref[k].hi + (p.mref[k].lo + M[k]);
  const float T00 = Mf[4];
  const float T0[3] = {Mf[5], Mf[6], Mf[7]};
  const float Tij[3][3] = {{Mf[8], Mf[9], Mf[10]}, {Mf[9], Mf[11], Mf[12]}, {Mf[10], Mf[12], Mf[13]}};
  float v[3];
  {
    const float iden = __fdividef(1.0f, T00 + (Mf[8] + Mf[11] + Mf[13]) * (1.0f / 3.0f));
    v[0] = T0[0] * iden;
    v[1] = T0[1] * iden;
    v[2] = T0[2] * iden;
  }
#pragma unroll 1
  for (int it = 0; it < 8; ++it) {
    const float e = T00 - T0[0] * v[0] - T0[1] * v[1] - T0[2] * v[2];
    float F[3], J[3][3];
#pragma unroll
    for (int a = 0; a < 3; ++a) {
      F[a] = T0[a] - Tij[a][0] * v[0] - Tij[a][1] * v[1] - Tij[a][2] * v[2] - e * v[a];
#pragma unroll
      for (int b = 0; b < 3; ++b) J[a][b] = -Tij[a][b] - (a == b ? e : 0.0f) + v[a] * T0[b];
    }
    const float c00 = J[1][1] * J[2][2] - J[1][2] * J[2][1];
    const float c01 = J[1][2] * J[2][0] - J[1][0] * J[2][2];
    const float c02 = J[1][0] * J[2][1] - J[1][1] * J[2][0];
    const float id = __fdividef(1.0f, J[0][0] * c00 + J[0][1] * c01 + J[0][2] * c02);
    const float d0 = (F[0] * c00 + J[0][1] * (F[2] * J[1][2] - F[1] * J[2][2]) +
                      J[0][2] * (F[1] * J[2][1] - F[2] * J[1][1])) * id;
    const float d1 = (J[0][0] * (F[1] * J[2][2] - F[2] * J[1][2]) + F[0] * c01 +
                      J[0][2] * (F[2] * J[1][0] - F[1] * J[2][0])) * id;
    const float d2 = (J[0][0] * (F[2] * J[1][1] - F[1] * J[2][1]) + J[0][1] * (F[1] * J[2][0] - F[2] * J[1][0]) +
                      F[0] * c02) * id;
    v[0] -= d0;
    v[1] -= d1;
    v[2] -= d2;
    // quadratic convergence: after a step below 1e-4 the error is of
    // order its square, below the FP32 rounding of v
    if (fabsf(d0) + fabsf(d1) + fabsf(d2) < 1e-4f) break;
  }
  const float v2 = v[0] * v[0] + v[1] * v[1] + v[2] * v[2];
  if (!(v2 < 1.0f)) fl |= ERR_LANDAU;
  const float sq = sqrtf(1.0f - v2);
  const float dg = __fdividef(v2, sq * (1.0f + sq));  // gamma - 1
  const float U0 = 1.0f + dg, Ux = U0 * v[0], Uy = U0 * v[1], Uz = U0 * v[2];
  // n = U.N = n_r + n_d, e/n = y_r + y_d from the deviation moments
  const float Xi = M[0] - v[0] * M[1] - v[1] * M[2] - v[2] * M[3];
  const float nd = fmaf(dg, p.nr.lo, fmaf(dg, Xi + p.nr.hi, Xi));
  const float n = p.nr.hi + (p.nr.lo + nd);
  if (!(n > 0.0f)) fl |= ERR_DENSITY;
  const float ed = M[4] - M[5] * v[0] - M[6] * v[1] - M[7] * v[2];
  const float yd = __fdividef(ed - fmaf(p.yr.hi, nd, p.yr.lo * nd), n);
  if (!(p.yr.hi + yd > p.mb)) fl |= ERR_EOS;
  // EOS: T = 1 + T_d solves 3 T_d + m (R(m/T) - R_r) = y_d; FP32 Newton ...
  float Td = yd / p.cv_r, slope = p.cv_r;
#pragma unroll 1
  for (int it = 0; it < 12; ++it) {
    const float T = 1.0f + Td;
    if (!(T > 0.0f)) {
      fl |= ERR_EOS;
      Td = 0.0f;
      break;
    }
    const float zz = __fdividef(p.mb, T);
    const float R32 = ratio32(zz, p.rt32, fl);
    slope = eos_slope<float>(R32, zz);
    const float step = __fdividef(3.0f * Td + p.mb * ((R32 - p.Rr.hi) - p.Rr.lo) - yd, slope);
    Td -= step;
    if (fabsf(step) < 1e-4f) break;   // the FP64 step below squares the remaining error
  }
  // ... and one FP64 Newton step: dR(Td) from the lattice's FP64 table in
  // Td, else from the R(zeta) table
  float dR;
  {
    double dR64;
    if (!dr_table64(Td, p.dr64, dR64)) dR64 = dr_from_zeta(Td, p.mb64, p.Rr64, p.rt64, fl);
    const double g64 = fma(3.0, (double)Td, fma(p.mb64, dR64, -(double)yd));
    const float step = __fdividef((float)g64, slope);
    Td -= step;
    // R at the corrected T to first order: d(dR)/dTd = (c_v - 3)/m, c_v = slope
    dR = fmaf((slope - 3.0f) * __fdividef(1.0f, p.mb), -step, (float)dR64);
  }
  const float R = p.Rr.hi + (p.Rr.lo + dR);
  const float T = 1.0f + Td;
  return SplitSite3{dg, U0, Ux, Uy, Uz, n, nd, Td, dR, R, T};
}

}  // namespace rlbm
