// Stencil-specialised FP64 step: parts shared by the second- and third-order
// kernels (rlbm_fused64.cu, rlbm_fused64_o3.cu).
//
// The FP64 pipe bounds these kernels (2 lanes a clock and SM on GB300, 64
// times fewer than FP32), so what counts is the number of FP64 instructions a
// site, and everything that need not be FP64 is kept off that pipe:
//
//  * moments from integer-weighted sums over reflection orbits, folded in
//    with one group momentum a sum: about 4 FP64 instructions a population
//    where nine products a population take 9;
//  * the site solve starts from FP32 iterates (Landau frame and temperature);
//    corrections with the FP64 residual and an FP32 inverse slope, mostly two,
//    go on until what is left is below FP64 rounding.  FP64 divisions and
//    square roots are an FP32 seed and two Newton corrections;
//  * where that does not settle (or a seed is not finite) the site falls back
//    to the all-FP64 iterations of solve_site_f64, so every state is treated,
//    and every error bit set, as there.
//
// Measured (M1, FP64): 256^2 272 -> 107 us a step against the table-driven
// step_f64_kernel, which other six-group stencils still take; third order
// (Q = 100) 504 -> 228 us against step_o3_kernel.  Lattices of few warps:
// rlbm_lanes64.cu.
// The populations are pulled twice (the second pull hits L1/L2) instead of
// being held in 116 registers: 128 registers, eight blocks of 64 threads an SM
// (65536 sites are 6.7 such blocks an SM; blocks of 128 left the SMs with four of
// them to finish 9 % later).
#pragma once

#include <utility>

#include "rlbm_kernels.cuh"
#include "rlbm_stencils.h"

namespace rlbm {

// 1/x from an FP32 seed (relative error 1e-7, squared twice); |x| in FP32's
// normal range.
__device__ __forceinline__ double rcp64(double x) {
  double r = (double)__frcp_rn((float)x);
  r = fma(r, fma(-x, r, 1.0), r);
  return fma(r, fma(-x, r, 1.0), r);
}

// The all-FP64 solve, out of line (rare).
static __device__ __noinline__ void solve_site_f64_cold(const double* m, const SiteConsts* sc,
                                                        const double* __restrict__ rt64, unsigned* fl,
                                                        Macro<double>* o) {
  *o = solve_site_f64(m, *sc, rt64, *fl);
}

// T and R = K1/K2(m/T) of 3 T + m R(m/T) = y (Eq. 28): FP32 Newton, then FP64
// corrections; iT = 1/T nearly.  False where it did not settle.
__device__ __forceinline__ bool eos_seeded(double y, const SiteConsts& sc, const double* __restrict__ rt64,
                                           const float* __restrict__ rt32, double& T, double& iT, double& R) {
  const double mb = sc.mbar;
  const double w = y - mb;
  bool ok = w > 1e-30 && w < 1e30;
  float last = 1.0f;
  {
    const float mbf = (float)mb, yf = (float)y;
    float Tf = __fdividef((float)w, 3.0f - 1.5f * __fdividef(mbf * mbf, yf * yf));
    unsigned fz = 0;
#pragma unroll 1
    for (int it = 0; it < 12; ++it) {
      const float z = __fdividef(mbf, Tf);
      const float Rf = ratio32(z, rt32, fz);
      const float dT = __fdividef(3.0f * Tf + mbf * (Rf - 1.0f) - (float)w, eos_slope<float>(Rf, z));
      if (!(Tf - dT > 0.0f)) break;
      Tf -= dT;
      // a step this short leaves an error of its square
      if (fabsf(dT) < 3e-4f * Tf) break;
    }
    ok = ok && Tf > 1e-30f && Tf < 1e30f;
    T = (double)Tf;
    float fiT = __frcp_rn(Tf);
    iT = (double)fiT;
    float dR = 0.0f, z32 = 0.0f;
#pragma unroll 1
    for (int it = 0; it < 4; ++it) {
      // iT is off by 1e-7 (the seed's rounding or the last step): two steps
      iT = fma(iT, fma(-T, iT, 1.0), iT);
      iT = fma(iT, fma(-T, iT, 1.0), iT);
      const double z = mb * iT;
      R = ratio64(z, rt64, fz);
      const double slope = eos_slope<double>(R, z);
      const float dT = (float)(fma(3.0, T, fma(mb, R, -y))) * __frcp_rn((float)slope);
      T -= (double)dT;
      last = fabsf(dT) * (float)iT;
      z32 = (float)z;
      // d R = R' dz, dz = z dT / T (T falls by dT), R' = (3 - slope) / z^2
      dR = (3.0f - (float)slope) * __frcp_rn(z32) * (dT * (float)iT);
      // the correction's slope is exact to FP32 rounding, so what is left is
      // 1e-7 of this step (and its square)
      if (last < 1e-9f) break;
    }
    R += (double)dR;
    ok = ok && last < 1e-9f && fz == 0;
  }
  return ok;
}

// Whether FP64 corrections of the Landau frame have settled, from the lengths of
// the last two.  Their inverse Jacobian is fixed, and off by up to about 1e-5 times
// gamma^2, so each is shorter than the one before by about that factor and d1 (d1/d0)
// is left: below 1e-17, a tenth of the rounding of v.  Or the last one is as short as
// the all-FP64 iterations ask for.  (NaN: not settled.)  A limit on d1 alone left up
// to 2e-13 at gamma = 8, where rounding leaves 2e-14.  At gamma below 1.2 one site
// in 200 takes a third correction.
__device__ __forceinline__ bool landau_settled(float d0, float d1) {
  return d1 < 1e-15f || d1 * d1 < 1e-17f * d0;
}

// Site solve of FP64 storage: m = N0 Nx Ny T00 T0x T0y Txx Txy Tyy.
__device__ __forceinline__ Macro<double> solve_site_f64_seeded(const double (&m)[9], const SiteConsts& sc,
                                                               const double* __restrict__ rt64,
                                                               const float* __restrict__ rt32, unsigned& fl) {
  // scaled by the power of two of T^00, so that FP32 holds any density
  const int ex = (int)((__double_as_longlong(m[3]) >> 52) & 0x7ff);
  const double scale = __longlong_as_double((long long)(2046 - ex) << 52);   // 2^(1023 - ex)
  double t[6];
#pragma unroll
  for (int k = 0; k < 6; ++k) t[k] = m[3 + k] * scale;   // T00 T0x T0y Txx Txy Tyy
  // 2^-465 .. 2^465, where the products of the all-FP64 Landau step neither
  // overflow nor underflow; it decides about states beyond
  bool ok = ex > 1023 - 465 && ex < 1023 + 465;
  float vx, vy, j11, j12, j21, j22;   // iterate, inverse Jacobian
  {
    float f[6];
#pragma unroll
    for (int k = 0; k < 6; ++k) f[k] = (float)t[k];
    const float iden = __fdividef(1.0f, f[0] + 0.5f * (f[3] + f[5]));
    vx = f[1] * iden;
    vy = f[2] * iden;
    j11 = j12 = j21 = j22 = 0.0f;
#pragma unroll 1
    for (int it = 0; it < 8; ++it) {
      const float e = f[0] - f[1] * vx - f[2] * vy;
      const float Fx = f[1] - f[3] * vx - f[4] * vy - e * vx;
      const float Fy = f[2] - f[4] * vx - f[5] * vy - e * vy;
      const float J11 = -f[3] - e + vx * f[1], J12 = -f[4] + vx * f[2];
      const float J21 = -f[4] + vy * f[1], J22 = -f[5] - e + vy * f[2];
      const float id = __fdividef(1.0f, J11 * J22 - J12 * J21);
      j11 = J22 * id;
      j12 = -J12 * id;
      j21 = -J21 * id;
      j22 = J11 * id;
      const float dx = j11 * Fx + j12 * Fy, dy = j21 * Fx + j22 * Fy;
      vx -= dx;
      vy -= dy;
      // the Jacobian of the last step is off by about its length
      if (fabsf(dx) + fabsf(dy) < 1e-5f) break;
    }
  }
  double Vx = vx, Vy = vy, e;
  float d0, d1 = 0.0f;   // lengths of the last two corrections
  auto correct = [&] {
    e = t[0] - t[1] * Vx - t[2] * Vy;
    const float Fx = (float)(t[1] - t[3] * Vx - t[4] * Vy - e * Vx);
    const float Fy = (float)(t[2] - t[4] * Vx - t[5] * Vy - e * Vy);
    const float dx = j11 * Fx + j12 * Fy, dy = j21 * Fx + j22 * Fy;
    Vx -= (double)dx;
    Vy -= (double)dy;
    d0 = d1;
    d1 = fabsf(dx) + fabsf(dy);
  };
  correct();
  correct();
#pragma unroll 1
  for (int it = 0; it < 4 && !landau_settled(d0, d1); ++it) correct();
  ok = ok && landau_settled(d0, d1);
  const double v2 = Vx * Vx + Vy * Vy;
  const double s = 1.0 - v2;
  ok = ok && s > 1e-6;
  double g = (double)rsqrtf((float)s);
  const double hs = 0.5 * s;
  g = g * fma(-hs * g, g, 1.5);
  g = g * fma(-hs * g, g, 1.5);
  Macro<double> o;
  o.U0 = g;
  o.dU = g * g * v2 * rcp64(g + 1.0);
  o.Ux = g * Vx;
  o.Uy = g * Vy;
  e = t[0] - t[1] * Vx - t[2] * Vy;          // energy density, scaled
  const double ns = g * ((m[0] - Vx * m[1] - Vy * m[2]) * scale);
  o.n = g * (m[0] - Vx * m[1] - Vy * m[2]);
  const double mb = sc.mbar;
  ok = ok && ns > 1e-30;
  const double rn = rcp64(ns);
  double y = e * rn;
  y = fma(rn, fma(-ns, y, e), y);            // e/n
  double T, iT, R;
  ok = eos_seeded(y, sc, rt64, rt32, T, iT, R) && ok;
  if (!ok) {
    // copies: passing the addresses of m or o would move them to local memory
    double mm[9];
#pragma unroll
    for (int k = 0; k < 9; ++k) mm[k] = m[k];
    Macro<double> c;
    unsigned f = 0;
    solve_site_f64_cold(mm, &sc, rt64, &f, &c);
    fl |= f;
    return c;
  }
  o.T = T;
  o.R = R;
  o.zeta = mb * iT;
  o.dR = R - sc.Rr;
  o.F = sc.mY * o.dR + 3.0 * (T - 1.0);
  o.G = mb * o.dR + 4.0 * (T - 1.0);
  return o;
}

// Displacements reduced modulo the lattice, for any lattice size: entry
// D + kMaxDisp is D mod N in [0, N).
constexpr int kMaxDisp = 6;

template <class Def, int K>
__host__ __device__ constexpr bool orbit_starts_group() {
  return K == 0 || Def::O.grp[K - 1] != Def::O.grp[K];
}
template <class Def, int K>
__host__ __device__ constexpr bool orbit_ends_group() {
  return K + 1 == Def::O.K || Def::O.grp[K + 1] != Def::O.grp[K];
}

// Where a site's populations are pulled from; mask 0: from the site itself (S_0
// read in place), -1: from x - n_i.
struct Pull64 {
  const double* fin;
  size_t plane;
  unsigned pitch;
  int x, y, Nx, Ny;
  const int *dxm, *dym;
  int mask;
};

template <class Def, int I>
__device__ __forceinline__ double pull64(const Pull64& q) {
  const unsigned xs = (unsigned)wrap_sub(q.x, q.dxm[Def::F.nx[I] + kMaxDisp] & q.mask, q.Nx);
  const unsigned ys = (unsigned)wrap_sub(q.y, q.dym[Def::F.ny[I] + kMaxDisp] & q.mask, q.Ny);
  return __ldg(q.fin + (ys * q.pitch + xs) + q.plane * I);
}

// FP32 planes, as FP64 values.
struct Pull32 {
  const float* fin;
  size_t plane;
  unsigned pitch;
  int x, y, Nx, Ny;
  const int *dxm, *dym;
  int mask;
};
template <class Def, int I>
__device__ __forceinline__ double pull64(const Pull32& q) {
  const unsigned xs = (unsigned)wrap_sub(q.x, q.dxm[Def::F.nx[I] + kMaxDisp] & q.mask, q.Nx);
  const unsigned ys = (unsigned)wrap_sub(q.y, q.dym[Def::F.ny[I] + kMaxDisp] & q.mask, q.Ny);
  return (double)__ldg(q.fin + (ys * q.pitch + xs) + q.plane * I);
}

// Sums of the current group, 1, n_x, n_y, n_x^2, n_x n_y, n_y^2, over one
// reflection orbit; at the end of a group they go into the moments with the
// group's momenta gm = P0, P0^2, Pv, P0 Pv, Pv^2.
template <class Def, int K, class Pull>
__device__ __forceinline__ void acc64_orbit(const Pull& q, const double (*gmt)[5], double (&s)[6], double (&M)[9]) {
  constexpr int kind = Def::O.kind[K], g = Def::O.grp[K], ax = Def::O.ax[K], ay = Def::O.ay[K];
  constexpr int i0 = Def::O.idx[K][0], i1 = Def::O.idx[K][1], i2 = Def::O.idx[K][2], i3 = Def::O.idx[K][3];
  if constexpr (orbit_starts_group<Def, K>()) {
#pragma unroll
    for (int k = 0; k < 6; ++k) s[k] = 0.0;
  }
  if constexpr (kind == 1) {
    s[0] += pull64<Def, i0>(q);
  } else if constexpr (kind == 2) {
    const double a = pull64<Def, i0>(q), b = pull64<Def, i1>(q);
    const double S = a + b;
    s[0] += S;
    s[1] = fma((double)ax, a - b, s[1]);
    s[3] = fma((double)(ax * ax), S, s[3]);
  } else if constexpr (kind == 3) {
    const double a = pull64<Def, i0>(q), b = pull64<Def, i2>(q);
    const double S = a + b;
    s[0] += S;
    s[2] = fma((double)ay, a - b, s[2]);
    s[5] = fma((double)(ay * ay), S, s[5]);
  } else {
    const double d0 = pull64<Def, i0>(q), d1 = pull64<Def, i1>(q), d2 = pull64<Def, i2>(q), d3 = pull64<Def, i3>(q);
    const double a = d0 + d1, b = d0 - d1, c = d2 + d3, w = d2 - d3;
    const double S = a + c;
    s[0] += S;
    s[1] = fma((double)ax, b + w, s[1]);
    s[2] = fma((double)ay, a - c, s[2]);
    s[3] = fma((double)(ax * ax), S, s[3]);
    s[4] = fma((double)(ax * ay), b - w, s[4]);
    s[5] = fma((double)(ay * ay), S, s[5]);
  }
  if constexpr (orbit_ends_group<Def, K>()) {
    const double* gm = gmt[g];
    M[0] = fma(gm[0], s[0], M[0]);
    M[3] = fma(gm[1], s[0], M[3]);
    M[1] = fma(gm[2], s[1], M[1]);
    M[2] = fma(gm[2], s[2], M[2]);
    M[4] = fma(gm[3], s[1], M[4]);
    M[5] = fma(gm[3], s[2], M[5]);
    M[6] = fma(gm[4], s[3], M[6]);
    M[7] = fma(gm[4], s[4], M[7]);
    M[8] = fma(gm[4], s[5], M[8]);
  }
}

template <class Def, class Pull, int... Ks>
__device__ __forceinline__ void acc64_all(std::integer_sequence<int, Ks...>, const Pull& q, const double (*gmt)[5],
                                          double (&M)[9]) {
  double s[6];
#pragma unroll
  for (int k = 0; k < 9; ++k) M[k] = 0.0;
  (acc64_orbit<Def, Ks>(q, gmt, s, M), ...);
}

// Relaxation weights U.p/(p0 tau) and destination of the collision.
struct Relax64 {
  double a0, ax, ay;
  double* out;
  size_t plane;
};

template <class Def, int I>
__device__ __forceinline__ void relax64(const Pull64& q, const Relax64& r, double om, double e) {
  const double v = pull64<Def, I>(q);
  __stcs(r.out + r.plane * I, fma(om, e - v, v));
}

// The members of reflection orbit K, with the equilibrium's parts E (even in
// n_x and n_y), X, Y (odd in one) and Z (odd in both).
template <class Def, int K>
__device__ __forceinline__ void relax64_orbit(const Pull64& q, const Relax64& r, double E, double X, double Y, double Z) {
  constexpr int kind = Def::O.kind[K], ax = Def::O.ax[K], ay = Def::O.ay[K];
  constexpr int i0 = Def::O.idx[K][0], i1 = Def::O.idx[K][1], i2 = Def::O.idx[K][2], i3 = Def::O.idx[K][3];
  if constexpr (kind == 1) {
    relax64<Def, i0>(q, r, r.a0, E);
  } else if constexpr (kind == 2) {
    relax64<Def, i0>(q, r, fma(-(double)ax, r.ax, r.a0), E + X);
    relax64<Def, i1>(q, r, fma((double)ax, r.ax, r.a0), E - X);
  } else if constexpr (kind == 3) {
    relax64<Def, i0>(q, r, fma(-(double)ay, r.ay, r.a0), E + Y);
    relax64<Def, i2>(q, r, fma((double)ay, r.ay, r.a0), E - Y);
  } else {
    const double EP = E + Z, EM = E - Z, XP = X + Y, XM = X - Y;
    const double op = fma(-(double)ax, r.ax, r.a0), om = fma((double)ax, r.ax, r.a0);
    relax64<Def, i0>(q, r, fma(-(double)ay, r.ay, op), EP + XP);   // (+, +)
    relax64<Def, i1>(q, r, fma(-(double)ay, r.ay, om), EM - XM);   // (-, +)
    relax64<Def, i2>(q, r, fma((double)ay, r.ay, op), EM + XM);    // (+, -)
    relax64<Def, i3>(q, r, fma((double)ay, r.ay, om), EP - XP);    // (-, -)
  }
}

// ------------------------------------------------ equilibrium, second order
// Equilibrium coefficients of one group from the projections r.
__device__ __forceinline__ void group_coeffs64(const double* a, const double (&r)[10], double (&c)[6]) {
  c[0] = fma(a[0], r[0], fma(a[1], r[1], fma(a[2], r[4], fma(a[3], r[7], a[4] * r[8]))));
  c[1] = fma(a[5], r[2], a[6] * r[5]);
  c[2] = fma(a[5], r[3], a[6] * r[6]);
  c[3] = a[7] * (r[7] - r[8]);
  c[4] = a[8] * r[7];
  c[5] = a[9] * r[9];
}

// n times the projections of App. B without their normalisations (in gf); ref:
// n R of the reference state that the storage subtracts (0: none).
__device__ __forceinline__ void projections64(const SiteConsts& sc, const Macro<double>& o, double ref,
                                              double (&r)[10]) {
  const double n = o.n, mr32 = fma(sc.mbar, o.R, 4.0 * o.T);
  const double nm = n * mr32, h = n * fma(mr32, o.dU, o.G);
  const double yy = nm * o.Uy * o.Uy;
  r[0] = n * o.R - ref;
  r[1] = n * (o.dU - sc.k21 * o.dR);
  r[2] = n * o.Ux;
  r[3] = n * o.Uy;
  r[4] = n * (o.F + o.dU * (fma(2.0, mr32, sc.cb00_1) + o.dU * mr32));
  r[5] = h * o.Ux;
  r[6] = h * o.Uy;
  r[7] = yy;
  r[8] = fma(-2.0 * nm * o.Ux, o.Ux, yy);
  r[9] = nm * o.Ux * o.Uy;
}

}  // namespace rlbm
