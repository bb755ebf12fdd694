// Init and read-out of compiled 2D stencils, shared parts (rlbm_io2.cu,
// rlbm_io_o3.cu).  Both stay FP64, as the table-driven kernels they replace, but
// evaluate the equilibrium and the moment sums once a reflection orbit
// (rlbm_fused64.cuh), so that the FP64 pipe, which bounds them, has about a
// third to a fifth of the work; and the init writes S_0 alone: a read-out right
// after it reads S_0 in place (mark_unwritten) instead of pulling a shifted copy
// S_{-1}.
#pragma once

#include "rlbm_fused64.cuh"

namespace rlbm {

// Macros of an initial field in the form the site solve returns.
__device__ __forceinline__ Macro<double> macro_of_fields64(double n, double ux, double uy, double T,
                                                           const SiteConsts& sc, const double* __restrict__ rt64,
                                                           unsigned& fl) {
  const double v2 = ux * ux + uy * uy;
  if (!(v2 < 1.0)) fl |= ERR_LANDAU;
  if (!(n > 0.0)) fl |= ERR_DENSITY;
  if (!(T > 0.0)) fl |= ERR_EOS;
  const double s = 1.0 - v2, hs = 0.5 * s;
  double g = (double)rsqrtf((float)s);     // s >= 2^-53 where v2 < 1
  g = g * fma(-hs * g, g, 1.5);
  g = g * fma(-hs * g, g, 1.5);
  Macro<double> o;
  o.n = n;
  o.U0 = g;
  o.dU = g * g * v2 * rcp64(g + 1.0);
  o.Ux = g * ux;
  o.Uy = g * uy;
  o.T = T;
  o.zeta = T > 1e-30 && T < 1e30 ? sc.mbar * rcp64(T) : sc.mbar / T;
  o.R = ratio64(o.zeta, rt64, fl);
  o.dR = o.R - sc.Rr;
  o.F = fma(sc.mY, o.dR, 3.0 * (T - 1.0));
  o.G = fma(sc.mbar, o.dR, 4.0 * (T - 1.0));
  return o;
}

// The requested planes of a site from its moments and macros.
__device__ __forceinline__ void write_planes64(const MomentOut& mo, long long N, long long s, const double (&m)[9],
                                               const Macro<double>& o) {
  const double iU = rcp64(o.U0), vx = o.Ux * iU, vy = o.Uy * iU;
  double* out = mo.out;
  int plane = 0;
  if (mo.mask & RLBM_M_N) out[(plane++) * N + s] = o.n;
  if (mo.mask & RLBM_M_UX) out[(plane++) * N + s] = vx;
  if (mo.mask & RLBM_M_UY) out[(plane++) * N + s] = vy;
  if (mo.mask & RLBM_M_T) out[(plane++) * N + s] = o.T;
  if (mo.mask & RLBM_M_E) out[(plane++) * N + s] = m[3] - m[4] * vx - m[5] * vy;
  if (mo.mask & RLBM_M_NVEC) {
#pragma unroll
    for (int k = 0; k < 3; ++k) out[(plane++) * N + s] = m[k];
  }
  if (mo.mask & RLBM_M_TMN) {
#pragma unroll
    for (int k = 3; k < 9; ++k) out[(plane++) * N + s] = m[k];
  }
}

// Values of the members of orbit K to put (pairs: the partners of a BF16 word).
template <class Def, int K, class Put>
__device__ __forceinline__ void emit_orbit(const Put& put, double E, double X, double Y, double Z) {
  constexpr int kind = Def::O.kind[K];
  constexpr int i0 = Def::O.idx[K][0], i1 = Def::O.idx[K][1], i2 = Def::O.idx[K][2], i3 = Def::O.idx[K][3];
  if constexpr (kind == 1) {
    put.template one<Def, i0>(E);
  } else if constexpr (kind == 2) {
    put.template pair<Def, i0, i1>(E + X, E - X);
  } else if constexpr (kind == 3) {
    put.template pair<Def, i0, i2>(E + Y, E - Y);
  } else {
    const double EP = E + Z, EM = E - Z, XP = X + Y, XM = X - Y;
    put.template pair<Def, i0, i3>(EP + XP, EP - XP);
    put.template pair<Def, i1, i2>(EM - XM, EM + XM);
  }
}

template <typename S>
struct PutPlain {
  S* out;   // the site's element of plane 0
  size_t plane;
  template <class Def, int I>
  __device__ __forceinline__ void one(double v) const {
    __stcs(out + plane * I, (S)v);
  }
  template <class Def, int I, int J>
  __device__ __forceinline__ void pair(double a, double b) const {
    one<Def, I>(a);
    one<Def, J>(b);
  }
};

}  // namespace rlbm
