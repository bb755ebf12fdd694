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
#include "rlbm_octants.cuh"

namespace rlbm {
namespace {

using D3 = Stencil3O3M5;

// Parity classes of the monomials kO3Exp3: bit 0, 1, 2 set where odd in p_x, p_y, p_z.
__host__ __device__ constexpr int parity3(int l) {
  return (kO3Exp3.e[l][1] & 1) | ((kO3Exp3.e[l][2] & 1) << 1) | ((kO3Exp3.e[l][3] & 1) << 2);
}

// Threads a block, and the populations that stay in shared memory between the
// two passes: KEEP of those from other planes (n_z != 0), whose lines have
// left L1 by the second pass; the others are pulled again.  90 of them (23 KB a
// block) leave room for eight blocks, 16 warps an SM.  Measured at 96 x 80 x 64:
// none kept 244 us a step, 60 184 us, 90 181 us, all 114 of other planes (seven
// blocks) 203 us, all 159 (five blocks) 245 us; 249-266 us at 128 threads with
// none kept; the table-driven kernel 1006 us.
struct Cfg3O3 {
  using D = D3;
  static constexpr int TB = 64, BLOCKS = 8, KEEP = 90;
  static constexpr bool KEEP_PLANE = false;
};

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
        if constexpr ((S & ~comps<D3, K>()) == 0) v[S] = class3<S>(L{}, w, e, S == 0 ? hl(w[0], nd) : 0.0f);
      }(),
      ...);
}

template <int K>
__device__ __forceinline__ void collide_orbit3(const Src3& q, const Fused3O3Params& p, const float* e, float nd,
                                               float a0, float ax, float ay, float az, float* __restrict__ out) {
  using S8 = std::make_integer_sequence<int, 8>;
  float v[8];
  classes3<K>(S8{}, p.ow[K], e, nd, v);
  wht<comps<D3, K>()>(v);   // class sums -> the members' equilibria
  relax_orbit3<Cfg3O3, K>(S8{}, q, v, a0, ax, ay, az, out);
}

template <int... Ks>
__device__ __forceinline__ void collide_all3(std::integer_sequence<int, Ks...>, const Src3& q,
                                             const Fused3O3Params& p, const float* e, float nd, float a0, float ax,
                                             float ay, float az, float* __restrict__ out) {
  (collide_orbit3<Ks>(q, p, e, nd, a0, ax, ay, az, out), ...);
}

__global__ void __launch_bounds__(Cfg3O3::TB, Cfg3O3::BLOCKS) fused3d_o3_kernel(const __grid_constant__ Fused3O3Params p,
                                                            const float* __restrict__ fin, float* __restrict__ fout) {
  static_assert(D3::O.K <= kMaxOct3, "orbit constants exceed Fused3O3Params::ow");
  const int nsite = p.Nx * p.Ny * p.Nz;   // < 2^31 (checked at creation)
  const int site = (int)(blockIdx.x * blockDim.x + threadIdx.x);
  unsigned fl = 0;
  __shared__ float kept[Cfg3O3::KEEP * Cfg3O3::TB];
  if (site < nsite) {
    const int r = site / p.Nx;
    const int x = site - r * p.Nx;
    const int z = r / p.Ny;
    const int y = r - z * p.Ny;
    Src3 q{kept + threadIdx.x, fin, (size_t)(unsigned)p.plane, (unsigned)p.zstride, (unsigned)p.pitch, x, y, z, p.Nx, p.Ny, p.Nz};
    using Orb = std::make_integer_sequence<int, D3::O.K>;
    float M[14];
    acc_all3<Cfg3O3>(Orb{}, q, p, M);
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
  const unsigned grid = (unsigned)(((long long)p.Nx * p.Ny * p.Nz + Cfg3O3::TB - 1) / Cfg3O3::TB);
  fused3d_o3_kernel<<<grid, Cfg3O3::TB, 0, s>>>(p, static_cast<const float*>(fin), static_cast<float*>(fout));
  return cudaGetLastError();
}

}  // namespace rlbm
