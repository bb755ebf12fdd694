// Stencil-specialised FP32 third-order step on native 3D lattices (the unfolded
// eleven-group stencil of m = 5, 159 populations).  Split arithmetic of the
// other compiled FP32 kernels (stored d_i = f_i - nref wr_i, integer-weighted
// sums, hi/lo constants, one FP64 step of the equation of state).
//
// Per octant orbit (+-n_x, +-n_y, +-n_z) the moment sums come from the
// Walsh-Hadamard sums of its members, and the equilibrium
//   f^eq_i - nref wr_i = n_d wr_i + sum_l e_l W_il
// from eight parity class sums: 31 products an orbit of up to eight members,
// where the table-driven kernel evaluates 31 a population and reads 188 bytes of
// table for it.  96 x 80 x 64: 1006 -> 181 us a step, half of the copy bandwidth;
// issue and latency bound (16 warps an SM).
#include "rlbm_o3_3d.cuh"
#include "rlbm_solve3.cuh"

namespace rlbm {
namespace {

using D3 = Stencil3O3M5;

// Parity classes of the monomials kO3Exp3: bit 0, 1, 2 set where odd in p_x, p_y, p_z.
__host__ __device__ constexpr int parity3(int l) {
  return (kO3Exp3.e[l][1] & 1) | ((kO3Exp3.e[l][2] & 1) << 1) | ((kO3Exp3.e[l][3] & 1) << 2);
}

// the components that orbit K has (bits)
template <int K>
__host__ __device__ constexpr int comps() {
  return (D3::O.ax[K] ? 1 : 0) | (D3::O.ay[K] ? 2 : 0) | (D3::O.az[K] ? 4 : 0);
}

// Threads a block, and the populations that stay in shared memory between the
// two passes: KEEP_MAX of those from other planes (n_z != 0), whose lines have
// left L1 by the second pass; the others are pulled again.  90 of them (23 KB a
// block) leave room for eight blocks, 16 warps an SM.  Measured at 96 x 80 x 64:
// none kept 244 us a step, 60 184 us, 90 181 us, all 114 of other planes (seven
// blocks) 203 us, all 159 (five blocks) 245 us; 249-266 us at 128 threads with
// none kept; the table-driven kernel 1006 us.
constexpr int TB = 64;
constexpr int KEEP_MAX = 90;
__host__ __device__ constexpr int keep_slot(int i) {
  if (D3::U.nz[i] == 0) return -1;
  int n = 0;
  for (int j = 0; j < i; ++j) n += D3::U.nz[j] != 0 ? 1 : 0;
  return n < KEEP_MAX ? n : -1;
}

struct Src3 {
  float* keep;
  const float* fin;
  size_t plane;
  unsigned zs, pitch;
  int x, y, z, Nx, Ny, Nz;
};

template <int I>
__device__ __forceinline__ float pull3(const Src3& q) {
  constexpr int DX = D3::U.nx[I], DY = D3::U.ny[I], DZ = D3::U.nz[I];
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

template <int K, int... S>
__device__ __forceinline__ void pull_orbit(std::integer_sequence<int, S...>, const Src3& q, float (&v)[8]) {
  (
      [&] {
        if constexpr ((S & ~comps<K>()) == 0) {
          constexpr int I = D3::O.idx[K][S], slot = keep_slot(I);
          v[S] = pull3<I>(q);
          if constexpr (slot >= 0) q.keep[slot * TB] = v[S];
        }
      }(),
      ...);
}

// group sums: 1, n_x, n_y, n_z, n_x^2, n_y^2, n_z^2, n_x n_y, n_x n_z, n_y n_z
template <int K>
__device__ __forceinline__ void acc_orbit3(const Src3& q, const Fused3O3Params& p, float (&s)[10], float (&M)[14]) {
  constexpr int C = comps<K>(), g = D3::O.grp[K], ax = D3::O.ax[K], ay = D3::O.ay[K], az = D3::O.az[K];
  if constexpr (K == 0 || D3::O.grp[K > 0 ? K - 1 : 0] != g) {
#pragma unroll
    for (int k = 0; k < 10; ++k) s[k] = 0.0f;
  }
  float v[8];
  pull_orbit<K>(std::make_integer_sequence<int, 8>{}, q, v);
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
  if constexpr (K + 1 == D3::O.K || D3::O.grp[K + 1] != g) {
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

template <int... Ks>
__device__ __forceinline__ void acc_all3(std::integer_sequence<int, Ks...>, const Src3& q, const Fused3O3Params& p,
                                         float (&M)[14]) {
  float s[10];
#pragma unroll
  for (int k = 0; k < 14; ++k) M[k] = 0.0f;
  (acc_orbit3<Ks>(q, p, s, M), ...);
}

template <int CLS, int... L>
__device__ __forceinline__ float class3(std::integer_sequence<int, L...>, const HL* w, const float* e, float acc) {
  (
      [&] {
        if constexpr (parity3(L) == CLS) acc = hl_fma(w[1 + L], e[L], acc);
      }(),
      ...);
  return acc;
}

template <int K, int... S>
__device__ __forceinline__ void classes3(std::integer_sequence<int, S...>, const HL* w, const float* e, float nd,
                                         float (&v)[8]) {
  using L = std::make_integer_sequence<int, kO3Mono3>;
  (
      [&] {
        if constexpr ((S & ~comps<K>()) == 0) v[S] = class3<S>(L{}, w, e, S == 0 ? hl(w[0], nd) : 0.0f);
      }(),
      ...);
}

template <int K, int S>
__device__ __forceinline__ void relax_member3(const Src3& q, float e, float a0, float ax, float ay, float az,
                                              float* __restrict__ out) {
  constexpr int I = D3::O.idx[K][S];
  constexpr int nx = D3::U.nx[I], ny = D3::U.ny[I], nz = D3::U.nz[I];
  float om = a0;   // (U0 - v0 n_i.U)/tau
  if constexpr (nx != 0) om = fmaf(-(float)nx, ax, om);
  if constexpr (ny != 0) om = fmaf(-(float)ny, ay, om);
  if constexpr (nz != 0) om = fmaf(-(float)nz, az, om);
  constexpr int slot = keep_slot(I);
  float v;
  if constexpr (slot >= 0) v = q.keep[slot * TB];
  else v = pull3<I>(q);
  __stcs(out + q.plane * I, fmaf(om, e - v, v));
}

template <int K, int... S>
__device__ __forceinline__ void relax_orbit3(std::integer_sequence<int, S...>, const Src3& q, const float (&v)[8],
                                             float a0, float ax, float ay, float az, float* __restrict__ out) {
  (
      [&] {
        if constexpr ((S & ~comps<K>()) == 0) relax_member3<K, S>(q, v[S], a0, ax, ay, az, out);
      }(),
      ...);
}

template <int K>
__device__ __forceinline__ void collide_orbit3(const Src3& q, const Fused3O3Params& p, const float* e, float nd,
                                               float a0, float ax, float ay, float az, float* __restrict__ out) {
  using S8 = std::make_integer_sequence<int, 8>;
  float v[8];
  classes3<K>(S8{}, p.ow[K], e, nd, v);
  wht<comps<K>()>(v);   // class sums -> the members' equilibria
  relax_orbit3<K>(S8{}, q, v, a0, ax, ay, az, out);
}

template <int... Ks>
__device__ __forceinline__ void collide_all3(std::integer_sequence<int, Ks...>, const Src3& q,
                                             const Fused3O3Params& p, const float* e, float nd, float a0, float ax,
                                             float ay, float az, float* __restrict__ out) {
  (collide_orbit3<Ks>(q, p, e, nd, a0, ax, ay, az, out), ...);
}

__global__ void __launch_bounds__(TB, 8) fused3d_o3_kernel(const __grid_constant__ Fused3O3Params p,
                                                            const float* __restrict__ fin, float* __restrict__ fout) {
  static_assert(D3::O.K <= kMaxOct3, "orbit constants exceed Fused3O3Params::ow");
  const int nsite = p.Nx * p.Ny * p.Nz;   // < 2^31 (checked at creation)
  const int site = (int)(blockIdx.x * blockDim.x + threadIdx.x);
  unsigned fl = 0;
  __shared__ float kept[KEEP_MAX * TB];
  if (site < nsite) {
    const int r = site / p.Nx;
    const int x = site - r * p.Nx;
    const int z = r / p.Ny;
    const int y = r - z * p.Ny;
    Src3 q{kept + threadIdx.x, fin, (size_t)(unsigned)p.plane, (unsigned)p.zstride, (unsigned)p.pitch, x, y, z, p.Nx, p.Ny, p.Nz};
    using Orb = std::make_integer_sequence<int, D3::O.K>;
    float M[14];
    acc_all3(Orb{}, q, p, M);
    const SplitSite3 o = split_solve3(p, M, fl);
    // e_l = n dmu_l in the small quantities dU, dT, dR, U_a
    float e[kO3Mono3];
    {
      O3Site3<float> s;
      const float h = fmaf(p.mb, o.R, 4.0f * o.T), dh = fmaf(p.mb, o.dR, 4.0f * o.Td);
      s.n = o.n;
      s.U[0] = o.U0;
      s.U[1] = o.Ux;
      s.U[2] = o.Uy;
      s.U[3] = o.Uz;
      s.dU = o.dg;
      s.dT = o.Td;
      s.dRm = o.dR * p.im;
      s.c = p.c;
      s.h = h;
      s.Th = o.T * h;
      s.Am = fmaf(6.0f, s.Th, p.mb * p.mb);
      s.hU = fmaf(h, o.U0, -p.c);
      s.sdev = fmaf(o.Td, s.hU, fmaf(h, o.dg, dh));
      s.q = fmaf(s.Am, o.U0, -p.c * h);
      o3_dev3_all<float>(std::make_integer_sequence<int, kO3Mono3>{}, s, e);
    }
    const float w = p.v0 * p.inv_tau;
    float* out = fout + ((unsigned)z * (unsigned)p.zstride + (unsigned)y * (unsigned)p.pitch + (unsigned)x);
    // the second pass pulls again: hide that its addresses are the first's, or
    // the compiler keeps 159 of them (or the values) across the site solve
    asm volatile("" : "+r"(q.x), "+r"(q.y), "+r"(q.z));
    collide_all3(Orb{}, q, p, e, o.nd, o.U0 * p.inv_tau, w * o.Ux, w * o.Uy, w * o.Uz, out);
  }
  report(fl, p.err);
}

}  // namespace

cudaError_t launch_fused3d_o3(const Fused3O3Params& p, const void* fin, void* fout, cudaStream_t s) {
  const unsigned grid = (unsigned)(((long long)p.Nx * p.Ny * p.Nz + TB - 1) / TB);
  fused3d_o3_kernel<<<grid, TB, 0, s>>>(p, static_cast<const float*>(fin), static_cast<float*>(fout));
  return cudaGetLastError();
}

}  // namespace rlbm
