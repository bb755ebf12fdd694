// Octant orbits in FP32 (rlbm_fused3d.cu, rlbm_fused3d_o3.cu): pull, moment sums
// and relaxation of the populations (+-n_x, +-n_y, +-n_z) of a group together.
// Cfg: the stencil (Cfg::D), threads a block (TB) and how many of the populations
// pulled from other planes (n_z != 0) stay in shared memory between the moment
// pass and the collision pass (KEEP; their lines have left L1 by then); the
// others are pulled again.
#pragma once

#include "rlbm_solve3.cuh"

namespace rlbm {

// the components that orbit K has (bits)
template <class D, int K>
__host__ __device__ constexpr int comps() {
  return (D::O.ax[K] ? 1 : 0) | (D::O.ay[K] ? 2 : 0) | (D::O.az[K] ? 4 : 0);
}

// slot of population i in shared memory, -1: pulled again
template <class Cfg>
__host__ __device__ constexpr int keep_slot(int i) {
  using D = typename Cfg::D;
  if (D::U.nz[i] == 0 && !Cfg::KEEP_PLANE) return -1;
  int n = 0;
  for (int j = 0; j < i; ++j) n += (D::U.nz[j] != 0 || Cfg::KEEP_PLANE) ? 1 : 0;
  return n < Cfg::KEEP ? n : -1;
}

struct Src3 {
  float* keep;
  const float* fin;
  size_t plane;
  unsigned zs, pitch;
  int x, y, z, Nx, Ny, Nz;
};

template <class D, int I>
__device__ __forceinline__ float pull3(const Src3& q) {
  constexpr int DX = D::U.nx[I], DY = D::U.ny[I], DZ = D::U.nz[I];
  const unsigned idx = (unsigned)wrap_c<DZ>(q.z, q.Nz) * q.zs + (unsigned)wrap_c<DY>(q.y, q.Ny) * q.pitch +
                       (unsigned)wrap_c<DX>(q.x, q.Nx);
  return __ldg(q.fin + idx + q.plane * I);
}

// In place: v[s] -> sum over members t of (-1)^(popcount(s & t)) v[t], over the bits C.
template <int C>
__device__ __forceinline__ void wht(float (&v)[8]) {
#pragma unroll
  for (int b = 1; b < 8; b <<= 1) {
    if (!(C & b)) continue;
#pragma unroll
    for (int s = 0; s < 8; ++s) {
      if ((s & b) || (s & ~C)) continue;
      const float a = v[s], c = v[s | b];
      v[s] = a + c;
      v[s | b] = a - c;
    }
  }
}

template <class Cfg, int K, int... S>
__device__ __forceinline__ void pull_orbit(std::integer_sequence<int, S...>, const Src3& q, float (&v)[8]) {
  using D = typename Cfg::D;
  (
      [&] {
        if constexpr ((S & ~comps<D, K>()) == 0) {
          constexpr int I = D::O.idx[K][S], slot = keep_slot<Cfg>(I);
          v[S] = pull3<D, I>(q);
          if constexpr (slot >= 0) q.keep[slot * Cfg::TB] = v[S];
        }
      }(),
      ...);
}

// group sums: 1, n_x, n_y, n_z, n_x^2, n_y^2, n_z^2, n_x n_y, n_x n_z, n_y n_z
template <class Cfg, int K, class P>
__device__ __forceinline__ void acc_orbit3(const Src3& q, const P& p, float (&s)[10], float (&M)[14]) {
  using D = typename Cfg::D;
  constexpr int C = comps<D, K>(), g = D::O.grp[K], ax = D::O.ax[K], ay = D::O.ay[K], az = D::O.az[K];
  if constexpr (K == 0 || D::O.grp[K > 0 ? K - 1 : 0] != g) {
#pragma unroll
    for (int k = 0; k < 10; ++k) s[k] = 0.0f;
  }
  float v[8];
  pull_orbit<Cfg, K>(std::make_integer_sequence<int, 8>{}, q, v);
  wht<C>(v);
  s[0] += v[0];
  if constexpr (C & 1) s[1] = fmaf((float)ax, v[1], s[1]);
  if constexpr (C & 2) s[2] = fmaf((float)ay, v[2], s[2]);
  if constexpr (C & 4) s[3] = fmaf((float)az, v[4], s[3]);
  if constexpr (C & 1) s[4] = fmaf((float)(ax * ax), v[0], s[4]);
  if constexpr (C & 2) s[5] = fmaf((float)(ay * ay), v[0], s[5]);
  if constexpr (C & 4) s[6] = fmaf((float)(az * az), v[0], s[6]);
  if constexpr ((C & 3) == 3) s[7] = fmaf((float)(ax * ay), v[3], s[7]);
  if constexpr ((C & 5) == 5) s[8] = fmaf((float)(ax * az), v[5], s[8]);
  if constexpr ((C & 6) == 6) s[9] = fmaf((float)(ay * az), v[6], s[9]);
  if constexpr (K + 1 == D::O.K || D::O.grp[K + 1] != g) {
    const HL* gm = p.gm[g];   // P0, P0^2, Pv, P0 Pv, Pv^2
    M[0] = hl_fma(gm[0], s[0], M[0]);
    M[4] = hl_fma(gm[1], s[0], M[4]);
#pragma unroll
    for (int a = 0; a < 3; ++a) {
      M[1 + a] = hl_fma(gm[2], s[1 + a], M[1 + a]);
      M[5 + a] = hl_fma(gm[3], s[1 + a], M[5 + a]);
    }
    M[8] = hl_fma(gm[4], s[4], M[8]);     // xx
    M[9] = hl_fma(gm[4], s[7], M[9]);     // xy
    M[10] = hl_fma(gm[4], s[8], M[10]);   // xz
    M[11] = hl_fma(gm[4], s[5], M[11]);   // yy
    M[12] = hl_fma(gm[4], s[9], M[12]);   // yz
    M[13] = hl_fma(gm[4], s[6], M[13]);   // zz
  }
}

template <class Cfg, class P, int... Ks>
__device__ __forceinline__ void acc_all3(std::integer_sequence<int, Ks...>, const Src3& q, const P& p, float (&M)[14]) {
  float s[10];
#pragma unroll
  for (int k = 0; k < 14; ++k) M[k] = 0.0f;
  (acc_orbit3<Cfg, Ks>(q, p, s, M), ...);
}

template <class Cfg, int K, int S>
__device__ __forceinline__ void relax_member3(const Src3& q, float e, float a0, float ax, float ay, float az,
                                              float* __restrict__ out) {
  using D = typename Cfg::D;
  constexpr int I = D::O.idx[K][S];
  constexpr int nx = D::U.nx[I], ny = D::U.ny[I], nz = D::U.nz[I];
  float om = a0;   // (U0 - v0 n_i.U)/tau
  if constexpr (nx != 0) om = fmaf(-(float)nx, ax, om);
  if constexpr (ny != 0) om = fmaf(-(float)ny, ay, om);
  if constexpr (nz != 0) om = fmaf(-(float)nz, az, om);
  constexpr int slot = keep_slot<Cfg>(I);
  float v;
  if constexpr (slot >= 0) v = q.keep[slot * Cfg::TB];
  else v = pull3<D, I>(q);
  __stcs(out + q.plane * I, fmaf(om, e - v, v));
}

template <class Cfg, int K, int... S>
__device__ __forceinline__ void relax_orbit3(std::integer_sequence<int, S...>, const Src3& q, const float (&v)[8],
                                             float a0, float ax, float ay, float az, float* __restrict__ out) {
  using D = typename Cfg::D;
  (
      [&] {
        if constexpr ((S & ~comps<D, K>()) == 0) relax_member3<Cfg, K, S>(q, v[S], a0, ax, ay, az, out);
      }(),
      ...);
}

}  // namespace rlbm
