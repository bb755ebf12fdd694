// Third-order scheme on native 3D lattices (unfolded eleven-group stencils):
// the monomial basis shared by the host builder (rlbm_stencil.cpp) and the
// kernels (rlbm_kernels3d.cu), and the kernels' parameters.  Internal.
#pragma once

#include "rlbm_internal.h"

namespace rlbm {

// The thirty centred monomials t^a p_x^i p_y^j p_z^k (t = p0 - c, a <= 1,
// a + i + j + k <= 3) that span the polynomials of degree <= 3 on the mass
// shell, as (a, i, j, k), lowest degree first.
constexpr int kO3Mono3 = 30;
struct O3Exp3 {
  int e[kO3Mono3][4];
};
constexpr O3Exp3 kO3Exp3 = {{
    {0, 0, 0, 0}, {1, 0, 0, 0},                                     // 1, t
    {0, 1, 0, 0}, {0, 0, 1, 0}, {0, 0, 0, 1},                       // p_a
    {1, 1, 0, 0}, {1, 0, 1, 0}, {1, 0, 0, 1},                       // t p_a
    {0, 2, 0, 0}, {0, 0, 2, 0}, {0, 0, 0, 2},                       // p_a p_b
    {0, 1, 1, 0}, {0, 1, 0, 1}, {0, 0, 1, 1},
    {1, 2, 0, 0}, {1, 0, 2, 0}, {1, 0, 0, 2},                       // t p_a p_b
    {1, 1, 1, 0}, {1, 1, 0, 1}, {1, 0, 1, 1},
    {0, 3, 0, 0}, {0, 0, 3, 0}, {0, 0, 0, 3},                       // p_a p_b p_c
    {0, 2, 1, 0}, {0, 2, 0, 1}, {0, 1, 2, 0}, {0, 0, 2, 1},
    {0, 1, 0, 2}, {0, 0, 1, 2}, {0, 1, 1, 1}}};

// Per population i, the dual-basis row W3[i * kRowW3 + l] = w_i (G^-1 phi(p_i))_l
// of the thirty monomials (G their Gram matrix under the weights); the main
// table row (Step3Params::tab64) keeps the momentum products at 0..13, the
// rest-frame weight w_i K1/K2(mbar)/mbar at 14 and p^a/p^0 at 28..30.
constexpr int kRowW3 = 32;

struct Step3O3Params {
  Step3Params b;          // lattice, tables, reference moments, site constants
  double c;               // centring shift mbar K2/K1(mbar)
  const double* w64;      // [Q][kRowW3]
  const float* w32;       // [Q][kRowW3] (FP32 storage)
};

// Compiled FP32 third-order 3D step (rlbm_fused3d_o3.cu): as Fused3Params with
// eleven groups; ow[K]: rest weight and thirty dual-basis values of the
// representative (+n_x, +n_y, +n_z) of octant orbit K, as hi/lo pairs.
constexpr int kMaxOct3 = 40;
struct Fused3O3Params {
  int Nx, Ny, Nz;
  long long pitch, zstride, plane;   // elements; zstride = pitch * Ny
  float inv_tau, v0;
  float mb, cv_r, c, im;             // im = 1/m
  HL Rr, nr, yr;
  HL mref[14];
  double Rr64, mb64;
  HL gm[11][5];
  HL ow[kMaxOct3][kO3Mono3 + 1];
  const double* rt64;
  const float* rt32;
  const double* dr64;
  unsigned* err;
};

cudaError_t launch_fused3d_o3(const Fused3O3Params& p, const void* fin, void* fout, cudaStream_t s);

// FP64 arithmetic of the compiled 3D stencils (rlbm_fused64_3d.cu): the FP64
// step, and init and read-out of both storages (cur, other and prev as for
// launch_init2 and launch_moments2).  dxm, dym, dzm: displacement D at [D + 6]
// reduced modulo the lattice; mref, ref (n R) and nref: the reference state that
// FP32 storage subtracts.
struct C3Params {
  int Nx, Ny, Nz;
  long long pitch, zstride, plane;   // elements; zstride = pitch * Ny
  double inv_tau, v0;
  SiteConsts sc;
  double nref, ref;
  double mref[14];
  int dxm[13], dym[13], dzm[13];
  const double* rt64;
  const float* rt32;
  unsigned* err;
};
struct C3Params2 : C3Params {   // second order: group momenta and the constants gf3
  double gm[6][5], gf[6][10];
};
struct C3Params3 : C3Params {   // third order: dual basis of the octant representatives
  double c;
  double gm[11][5];
  double ow[kMaxOct3][kO3Mono3 + 1];
};
cudaError_t launch_step3c(int kind, const C3Params2& p, const void* fin, void* fout, cudaStream_t s);
cudaError_t launch_step3c(const C3Params3& p, const void* fin, void* fout, cudaStream_t s);
cudaError_t launch_init3c(int kind, bool f64, const C3Params2& p, Field3Ptrs f, void* cur, void* other,
                          cudaStream_t s);
cudaError_t launch_init3c(bool f64, const C3Params3& p, Field3Ptrs f, void* cur, void* other, cudaStream_t s);
cudaError_t launch_moments3c(int kind, bool f64, const C3Params2& p, const void* prev, const void* cur, MomentOut mo,
                             cudaStream_t s);
cudaError_t launch_moments3c(bool f64, const C3Params3& p, const void* prev, const void* cur, MomentOut mo,
                             cudaStream_t s);

cudaError_t launch_step3d_o3(rlbm_dtype dt, const Step3O3Params& p, const void* fin, void* fout, cudaStream_t s);
cudaError_t launch_init3d_o3(rlbm_dtype dt, const Step3O3Params& p, Field3Ptrs f, void* cur, void* prev,
                             cudaStream_t s);

}  // namespace rlbm
