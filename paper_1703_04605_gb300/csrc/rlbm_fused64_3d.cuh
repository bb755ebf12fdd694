// FP64 arithmetic of the compiled stencils on native 3D lattices: the FP64 step,
// and the init and read-out of FP64 and FP32 storage (rlbm_fused64_3d.cu).  As
// rlbm_fused64.cuh in two dimensions, the FP64 pipe bounds all three: moment sums
// and equilibrium once an octant orbit (+-n_x, +-n_y, +-n_z), a site solve that
// starts from FP32 iterates, and an init that writes S_0 alone.
#pragma once

#include "rlbm_fused64.cuh"
#include "rlbm_o3_3d.cuh"
#include "rlbm_site3.cuh"

namespace rlbm {

// Site state: the macros and their deviations from rest at T_R.
struct Mac3 {
  double n, U0, Ux, Uy, Uz, T, R, dU, dR, e;
};

static __device__ __noinline__ void solve3_cold(const double* m, const SiteConsts* sc, const double* __restrict__ rt64,
                                                unsigned* fl, Macro3* o) {
  *o = solve3(m, *sc, rt64, *fl);
}

// m = N0 Nx Ny Nz T00 T0x T0y T0z Txx Txy Txz Tyy Tyz Tzz; see
// solve_site_f64_seeded for the scheme.
__device__ __forceinline__ Mac3 solve3_seeded(const double (&m)[14], const SiteConsts& sc,
                                              const double* __restrict__ rt64, const float* __restrict__ rt32,
                                              unsigned& fl) {
  const int ex = (int)((__double_as_longlong(m[4]) >> 52) & 0x7ff);
  const double scale = __longlong_as_double((long long)(2046 - ex) << 52);
  double t[10];
#pragma unroll
  for (int k = 0; k < 10; ++k) t[k] = m[4 + k] * scale;
  // 2^-310 .. 2^310: beyond, the all-FP64 solve's 3 x 3 determinant may leave the range
  bool ok = ex > 1023 - 310 && ex < 1023 + 310;
  float v[3], J[3][3];   // iterate, inverse Jacobian
  {
    float f[10];
#pragma unroll
    for (int k = 0; k < 10; ++k) f[k] = (float)t[k];
    const float S[3][3] = {{f[4], f[5], f[6]}, {f[5], f[7], f[8]}, {f[6], f[8], f[9]}};
    const float id0 = __fdividef(1.0f, f[0] + (f[4] + f[7] + f[9]) * (1.0f / 3.0f));
#pragma unroll
    for (int a = 0; a < 3; ++a) v[a] = f[1 + a] * id0;
#pragma unroll 1
    for (int it = 0; it < 8; ++it) {
      const float e = f[0] - f[1] * v[0] - f[2] * v[1] - f[3] * v[2];
      float F[3], A[3][3];
#pragma unroll
      for (int a = 0; a < 3; ++a) {
        F[a] = f[1 + a] - S[a][0] * v[0] - S[a][1] * v[1] - S[a][2] * v[2] - e * v[a];
#pragma unroll
        for (int b = 0; b < 3; ++b) A[a][b] = -S[a][b] - (a == b ? e : 0.0f) + v[a] * f[1 + b];
      }
      J[0][0] = A[1][1] * A[2][2] - A[1][2] * A[2][1];
      J[1][0] = A[1][2] * A[2][0] - A[1][0] * A[2][2];
      J[2][0] = A[1][0] * A[2][1] - A[1][1] * A[2][0];
      J[0][1] = A[0][2] * A[2][1] - A[0][1] * A[2][2];
      J[1][1] = A[0][0] * A[2][2] - A[0][2] * A[2][0];
      J[2][1] = A[0][1] * A[2][0] - A[0][0] * A[2][1];
      J[0][2] = A[0][1] * A[1][2] - A[0][2] * A[1][1];
      J[1][2] = A[0][2] * A[1][0] - A[0][0] * A[1][2];
      J[2][2] = A[0][0] * A[1][1] - A[0][1] * A[1][0];
      const float id = __fdividef(1.0f, A[0][0] * J[0][0] + A[0][1] * J[1][0] + A[0][2] * J[2][0]);
      float len = 0.0f;
#pragma unroll
      for (int a = 0; a < 3; ++a) {
#pragma unroll
        for (int b = 0; b < 3; ++b) J[a][b] *= id;
        const float d = J[a][0] * F[0] + J[a][1] * F[1] + J[a][2] * F[2];
        v[a] -= d;
        len += fabsf(d);
      }
      if (len < 1e-5f) break;
    }
  }
  double V[3] = {v[0], v[1], v[2]}, e;
  float d0, d1 = 0.0f;   // lengths of the last two corrections
  auto correct = [&] {
    e = t[0] - t[1] * V[0] - t[2] * V[1] - t[3] * V[2];
    float F[3];
    F[0] = (float)(t[1] - t[4] * V[0] - t[5] * V[1] - t[6] * V[2] - e * V[0]);
    F[1] = (float)(t[2] - t[5] * V[0] - t[7] * V[1] - t[8] * V[2] - e * V[1]);
    F[2] = (float)(t[3] - t[6] * V[0] - t[8] * V[1] - t[9] * V[2] - e * V[2]);
    d0 = d1;
    d1 = 0.0f;
#pragma unroll
    for (int a = 0; a < 3; ++a) {
      const float d = J[a][0] * F[0] + J[a][1] * F[1] + J[a][2] * F[2];
      V[a] -= (double)d;
      d1 += fabsf(d);
    }
  };
  correct();
  correct();
#pragma unroll 1
  for (int it = 0; it < 4 && !landau_settled(d0, d1); ++it) correct();
  ok = ok && landau_settled(d0, d1);
  const double v2 = V[0] * V[0] + V[1] * V[1] + V[2] * V[2];
  const double s = 1.0 - v2, hs = 0.5 * s;
  ok = ok && s > 1e-6;
  double g = (double)rsqrtf((float)s);
  g = g * fma(-hs * g, g, 1.5);
  g = g * fma(-hs * g, g, 1.5);
  Mac3 o;
  o.U0 = g;
  o.dU = g * g * v2 * rcp64(g + 1.0);
  o.Ux = g * V[0];
  o.Uy = g * V[1];
  o.Uz = g * V[2];
  o.e = m[4] - m[5] * V[0] - m[6] * V[1] - m[7] * V[2];
  o.n = g * (m[0] - V[0] * m[1] - V[1] * m[2] - V[2] * m[3]);
  const double ns = o.n * scale, es = o.e * scale;
  ok = ok && ns > 1e-30;
  const double rn = rcp64(ns);
  double y = es * rn;
  y = fma(rn, fma(-ns, y, es), y);
  double iT;
  ok = eos_seeded(y, sc, rt64, rt32, o.T, iT, o.R) && ok;
  if (!ok) {
    double mm[14];
#pragma unroll
    for (int k = 0; k < 14; ++k) mm[k] = m[k];
    Macro3 c;
    unsigned f = 0;
    solve3_cold(mm, &sc, rt64, &f, &c);
    fl |= f;
    o.n = c.n;
    o.U0 = c.U0;
    o.Ux = c.Ux;
    o.Uy = c.Uy;
    o.Uz = c.Uz;
    o.T = c.T;
    o.R = c.R;
    o.e = c.e;
    o.dU = (c.Ux * c.Ux + c.Uy * c.Uy + c.Uz * c.Uz) / (c.U0 + 1.0);
  }
  o.dR = o.R - sc.Rr;
  return o;
}

// The site state of an initial field.
__device__ __forceinline__ Mac3 mac3_of_fields(double n, double ux, double uy, double uz, double T,
                                               const SiteConsts& sc, const double* __restrict__ rt64, unsigned& fl) {
  const double v2 = ux * ux + uy * uy + uz * uz;
  if (!(v2 < 1.0)) fl |= ERR_LANDAU;
  if (!(n > 0.0)) fl |= ERR_DENSITY;
  if (!(T > 0.0)) fl |= ERR_EOS;
  const double s = 1.0 - v2, hs = 0.5 * s;
  double g = (double)rsqrtf((float)s);
  g = g * fma(-hs * g, g, 1.5);
  g = g * fma(-hs * g, g, 1.5);
  Mac3 o;
  o.n = n;
  o.U0 = g;
  o.dU = g * g * v2 * rcp64(g + 1.0);
  o.Ux = g * ux;
  o.Uy = g * uy;
  o.Uz = g * uz;
  o.T = T;
  o.R = ratio64(T > 1e-30 && T < 1e30 ? sc.mbar * rcp64(T) : sc.mbar / T, rt64, fl);
  o.dR = o.R - sc.Rr;
  o.e = 0.0;
  return o;
}

// ------------------------------------------------------------------ octants
template <class D, int K>
__host__ __device__ constexpr int octant_comps() {
  return (D::O.ax[K] ? 1 : 0) | (D::O.ay[K] ? 2 : 0) | (D::O.az[K] ? 4 : 0);
}

// A site's place; dxm, dym, dzm: displacements reduced modulo the lattice; mask 0:
// read in place, -1: pulled.
template <typename S>
struct Pull3 {
  const S* fin;
  size_t plane;
  unsigned zs, pitch;
  int x, y, z, Nx, Ny, Nz;
  const int *dxm, *dym, *dzm;
  int mask;
};

template <class D, int I, typename S>
__device__ __forceinline__ double pull3d(const Pull3<S>& q) {
  const unsigned xs = (unsigned)wrap_sub(q.x, q.dxm[D::U.nx[I] + kMaxDisp] & q.mask, q.Nx);
  const unsigned ys = (unsigned)wrap_sub(q.y, q.dym[D::U.ny[I] + kMaxDisp] & q.mask, q.Ny);
  const unsigned zs = (unsigned)wrap_sub(q.z, q.dzm[D::U.nz[I] + kMaxDisp] & q.mask, q.Nz);
  return (double)__ldg(q.fin + (zs * q.zs + ys * q.pitch + xs) + q.plane * I);
}

// In place: v[s] -> sum over t of (-1)^(popcount(s & t)) v[t] over the bits C.
template <int C>
__device__ __forceinline__ void wht64(double (&v)[8]) {
#pragma unroll
  for (int b = 1; b < 8; b <<= 1) {
    if (!(C & b)) continue;
#pragma unroll
    for (int s = 0; s < 8; ++s) {
      if ((s & b) || (s & ~C)) continue;
      const double a = v[s], c = v[s | b];
      v[s] = a + c;
      v[s | b] = a - c;
    }
  }
}

template <class D, int K, typename S, int... T>
__device__ __forceinline__ void pull_octant(std::integer_sequence<int, T...>, const Pull3<S>& q, double (&v)[8]) {
  (
      [&] {
        if constexpr ((T & ~octant_comps<D, K>()) == 0) {
          constexpr int I = D::O.idx[K][T];
          v[T] = pull3d<D, I>(q);
        }
      }(),
      ...);
}

// Group sums 1, n_a, n_a^2, n_x n_y, n_x n_z, n_y n_z over one octant orbit; at
// the end of a group into M with the group's momenta.
template <class D, int K, typename S>
__device__ __forceinline__ void acc_octant(const Pull3<S>& q, const double (*gmt)[5], double (&s)[10], double (&M)[14]) {
  constexpr int C = octant_comps<D, K>(), g = D::O.grp[K], ax = D::O.ax[K], ay = D::O.ay[K], az = D::O.az[K];
  if constexpr (K == 0 || D::O.grp[K > 0 ? K - 1 : 0] != g) {
#pragma unroll
    for (int k = 0; k < 10; ++k) s[k] = 0.0;
  }
  double v[8];
  pull_octant<D, K>(std::make_integer_sequence<int, 8>{}, q, v);
  wht64<C>(v);
  s[0] += v[0];
  if constexpr (C & 1) s[1] = fma((double)ax, v[1], s[1]);
  if constexpr (C & 2) s[2] = fma((double)ay, v[2], s[2]);
  if constexpr (C & 4) s[3] = fma((double)az, v[4], s[3]);
  if constexpr (C & 1) s[4] = fma((double)(ax * ax), v[0], s[4]);
  if constexpr (C & 2) s[5] = fma((double)(ay * ay), v[0], s[5]);
  if constexpr (C & 4) s[6] = fma((double)(az * az), v[0], s[6]);
  if constexpr ((C & 3) == 3) s[7] = fma((double)(ax * ay), v[3], s[7]);
  if constexpr ((C & 5) == 5) s[8] = fma((double)(ax * az), v[5], s[8]);
  if constexpr ((C & 6) == 6) s[9] = fma((double)(ay * az), v[6], s[9]);
  if constexpr (K + 1 == D::O.K || D::O.grp[K + 1] != g) {
    const double* gm = gmt[g];
    M[0] = fma(gm[0], s[0], M[0]);
    M[4] = fma(gm[1], s[0], M[4]);
#pragma unroll
    for (int a = 0; a < 3; ++a) {
      M[1 + a] = fma(gm[2], s[1 + a], M[1 + a]);
      M[5 + a] = fma(gm[3], s[1 + a], M[5 + a]);
    }
    M[8] = fma(gm[4], s[4], M[8]);     // xx
    M[9] = fma(gm[4], s[7], M[9]);     // xy
    M[10] = fma(gm[4], s[8], M[10]);   // xz
    M[11] = fma(gm[4], s[5], M[11]);   // yy
    M[12] = fma(gm[4], s[9], M[12]);   // yz
    M[13] = fma(gm[4], s[6], M[13]);   // zz
  }
}

template <class D, typename S, int... Ks>
__device__ __forceinline__ void acc_octants(std::integer_sequence<int, Ks...>, const Pull3<S>& q,
                                            const double (*gmt)[5], double (&M)[14]) {
  double s[10];
#pragma unroll
  for (int k = 0; k < 14; ++k) M[k] = 0.0;
  (acc_octant<D, Ks>(q, gmt, s, M), ...);
}

// -------------------------------------------------------------- equilibrium
// Second order (App. A/B per group, as rlbm_fused3d.cu): class sums of orbit K in v.
struct Eq3Second {
  double r[14], c[9];
  __device__ __forceinline__ void prepare(const C3Params2& p, const Mac3& o) {
    const double n = o.n, mr32 = fma(p.sc.mbar, o.R, 4.0 * o.T), nm = n * mr32;
    const double F = fma(p.sc.mY, o.dR, 3.0 * (o.T - 1.0)), G = fma(p.sc.mbar, o.dR, 4.0 * (o.T - 1.0));
    r[0] = n * o.R - p.ref;
    r[1] = n * (o.dU - p.sc.k21 * o.dR);
    r[2] = n * o.Ux;
    r[3] = n * o.Uy;
    r[4] = n * o.Uz;
    r[5] = n * (F + o.dU * (fma(2.0, mr32, p.sc.cb00_1) + o.dU * mr32));
    const double h = n * fma(mr32, o.dU, G);
    r[6] = h * o.Ux;
    r[7] = h * o.Uy;
    r[8] = h * o.Uz;
    const double yy = o.Uy * o.Uy, zz = o.Uz * o.Uz;
    r[9] = nm * (yy - zz);
    r[10] = nm * fma(-2.0 * o.Ux, o.Ux, yy + zz);
    r[11] = nm * o.Ux * o.Uz;
    r[12] = nm * o.Uy * o.Uz;
    r[13] = nm * o.Ux * o.Uy;
  }
  template <class D, int K>
  __device__ __forceinline__ void orbit(const C3Params2& p, double (&v)[8]) {
    constexpr int C = octant_comps<D, K>(), g = D::O.grp[K], ax = D::O.ax[K], ay = D::O.ay[K], az = D::O.az[K];
    if constexpr (K == 0 || D::O.grp[K > 0 ? K - 1 : 0] != g) {
      const double* a = p.gf[g];
      c[0] = fma(a[0], r[0], fma(a[1], r[1], fma(a[2], r[5], fma(a[3], r[9], a[4] * r[10]))));
#pragma unroll
      for (int b = 0; b < 3; ++b) c[1 + b] = fma(a[5], r[2 + b], a[6] * r[6 + b]);
      const double k9 = a[7] * r[9], k10 = a[8] * r[10];
      c[4] = fma(-3.0, k10, k9);    // q_xx
      c[5] = 2.0 * k9;              // q_yy
      c[6] = a[9] * r[13];          // q_xy
      c[7] = a[9] * r[11];          // q_xz
      c[8] = a[9] * r[12];          // q_yz
    }
    v[0] = c[0];
    if constexpr (C & 1) v[0] = fma((double)(ax * ax), c[4], v[0]);
    if constexpr (C & 2) v[0] = fma((double)(ay * ay), c[5], v[0]);
    if constexpr (C & 1) v[1] = (double)ax * c[1];
    if constexpr (C & 2) v[2] = (double)ay * c[2];
    if constexpr (C & 4) v[4] = (double)az * c[3];
    if constexpr ((C & 3) == 3) v[3] = (double)(ax * ay) * c[6];
    if constexpr ((C & 5) == 5) v[5] = (double)(ax * az) * c[7];
    if constexpr ((C & 6) == 6) v[6] = (double)(ay * az) * c[8];
    if constexpr (C == 7) {
      // no part odd in all three: two additions fewer than the full transform
      const double p0 = v[0] + v[1], m0 = v[0] - v[1], p1 = v[2] + v[3], m1 = v[2] - v[3];
      const double p2 = v[4] + v[5], m2 = v[4] - v[5], w = v[6];
      const double a0 = p0 + p1, a1 = m0 + m1, a2 = p0 - p1, a3 = m0 - m1;
      const double b0 = p2 + w, b1 = m2 + w, b2 = p2 - w, b3 = m2 - w;
      v[0] = a0 + b0;
      v[1] = a1 + b1;
      v[2] = a2 + b2;
      v[3] = a3 + b3;
      v[4] = a0 - b0;
      v[5] = a1 - b1;
      v[6] = a2 - b2;
      v[7] = a3 - b3;
    } else {
      wht64<C>(v);
    }
  }
};

// Parity class of monomial l of kO3Exp3: bits set where odd in p_x, p_y, p_z.
__host__ __device__ constexpr int parity_class3(int l) {
  return (kO3Exp3.e[l][1] & 1) | ((kO3Exp3.e[l][2] & 1) << 1) | ((kO3Exp3.e[l][3] & 1) << 2);
}

// Third order: the thirty dual-basis products by parity class.
struct Eq3Third {
  double e[kO3Mono3], dn;
  __device__ __forceinline__ void prepare(const C3Params3& p, const Mac3& o) {
    const double dT = o.T - 1.0, m = p.sc.mbar;
    O3Site3<double> s;
    s.n = o.n;
    s.U[0] = o.U0;
    s.U[1] = o.Ux;
    s.U[2] = o.Uy;
    s.U[3] = o.Uz;
    s.dU = o.dU;
    s.dT = dT;
    s.dRm = o.dR * p.sc.inv_m;
    s.c = p.c;
    s.h = fma(m, o.R, 4.0 * o.T);
    s.Th = o.T * s.h;
    s.Am = fma(6.0, s.Th, m * m);
    s.hU = fma(s.h, o.U0, -p.c);
    s.sdev = fma(dT, s.hU, fma(s.h, o.dU, fma(m, o.dR, 4.0 * dT)));
    s.q = fma(s.Am, o.U0, -p.c * s.h);
    o3_dev3_all<double>(std::make_integer_sequence<int, kO3Mono3>{}, s, e);
    dn = o.n - p.nref;
  }
  template <int CLS, int... L>
  __device__ __forceinline__ double sum(std::integer_sequence<int, L...>, const double* w, double acc) const {
    (
        [&] {
          if constexpr (parity_class3(L) == CLS) acc = fma(w[1 + L], e[L], acc);
        }(),
        ...);
    return acc;
  }
  template <int C, int... T>
  __device__ __forceinline__ void classes(std::integer_sequence<int, T...>, const double* w, double (&v)[8]) const {
    using L = std::make_integer_sequence<int, kO3Mono3>;
    (
        [&] {
          if constexpr ((T & ~C) == 0) v[T] = sum<T>(L{}, w, T == 0 ? w[0] * dn : 0.0);
        }(),
        ...);
  }
  template <class D, int K>
  __device__ __forceinline__ void orbit(const C3Params3& p, double (&v)[8]) {
    constexpr int C = octant_comps<D, K>();
    classes<C>(std::make_integer_sequence<int, 8>{}, p.ow[K], v);
    wht64<C>(v);
  }
};

template <class P>
struct EqOf;
template <>
struct EqOf<C3Params2> {
  using type = Eq3Second;
};
template <>
struct EqOf<C3Params3> {
  using type = Eq3Third;
};

}  // namespace rlbm
