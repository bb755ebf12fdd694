// Stencil-specialised FP32 step for 3D lattices (the unfolded stencil known at
// compile time).  Same step and split arithmetic as the 2D kernel of
// rlbm_fused.cuh (Eq. 16-20, 28, 49): stored values d_i = f_i - r_i; group
// sums with exact integer weights; group constants as hi/lo FP32 pairs; FP32
// Landau frame (Newton on the three velocity components) and FP32 EOS
// iterations with one FP64 Newton step of the EOS.
//
// Equilibrium per group g (|n|^2 constant in a group, so the n_z^2 term of the
// App. A polynomials folds into the others):
//   f^eq_i - r_i = alpha + beta . n + q_xx n_x^2 + q_yy n_y^2 + q_xy n_x n_y
//                  + q_xz n_x n_z + q_yz n_y n_z.
// Two passes over the populations, an octant orbit at a time (rlbm_octants.cuh):
// pull and sum, then relax and store, so only the sums of one group and its
// coefficients live in registers; values stay in shared memory between the
// passes or are pulled again (Cfg3).
#include "rlbm_octants.cuh"

namespace rlbm {
namespace {

// Threads a block, resident blocks and kept populations per stencil, measured
// at 160^3 (fraction of the copy bandwidth; in brackets the kernel without
// octant orbits): all values kept where they fit beside enough warps, else 60
// of those from other planes, at five blocks of 96 registers.
//   M1  (Q = 96):  all, 2 x 256 threads 0.764; 4 x 128 0.747; 60, 5 x 128 0.730 [0.680]
//   G16 (Q = 57):  all, 5 x 128 0.822; 4 x 128 0.783 [0.739]
//   E5  (Q = 133): 60, 5 x 128 0.711; 60, 4 x 128 0.704; all, 4 x 128 0.612 [0.567]
//   S2  (Q = 86):  60, 5 x 128 0.774; all, 4 x 128 0.753 [0.652]
template <class S>
struct Cfg3 {   // E5, S2
  using D = S;
  static constexpr int TB = 128, BLOCKS = 5, KEEP = 60;
  static constexpr bool KEEP_PLANE = false;
};
template <>
struct Cfg3<Stencil3M1> {
  using D = Stencil3M1;
  static constexpr int TB = 256, BLOCKS = 2, KEEP = D::Q;
  static constexpr bool KEEP_PLANE = true;
};
template <>
struct Cfg3<Stencil3G16> {
  using D = Stencil3G16;
  static constexpr int TB = 128, BLOCKS = 5, KEEP = D::Q;
  static constexpr bool KEEP_PLANE = true;
};

// Lattices of at most 200 sites an SM: blocks of 64 threads, so that the sites are
// on all of the SMs.  Such a step is bound by the latency of one pass, and
// by the loads that an SM's warps share.  us a step, Cfg3's block / 64 threads:
// 17^3 M1 10.3 / 8.2, E5 12.3 / 11.9; 23^3 M1 10.3 / 8.2; 27^3 G16 8.2 / 6.2, S2 9.3 /
// 8.2; 31^3 S2 10.3 / 9.3, E5 14.4 / 12.6 (32 threads: 12.3, but 17^3 12.3).  Above, at
// 33^3, M1 loses (10.3 / 12.3) and the others are even.
template <class C>
struct Small3 : C {
  static constexpr int TB = 64, BLOCKS = C::BLOCKS * C::TB / 64;
};
constexpr long long kSmall3 = 200;   // sites an SM

// The projections of App. B at a site, without their normalisations (in p.gf).
struct Proj3 {
  float r0, r1, r5, r9, r10, r11, r12, r13, h;
  float rU[3], U[3];
};

// Class sums of octant orbit K (bits of the odd directions): the group polynomial
// alpha + beta.n + q_xx n_x^2 + .. split by parity; c: the group's coefficients
// alpha, beta_a, q_xx, q_yy, q_xy, q_xz, q_yz.
template <class D, int K>
__device__ __forceinline__ void classes3(const Fused3Params& p, const Proj3& w, float (&c)[9], float (&v)[8]) {
  constexpr int C = comps<D, K>(), g = D::O.grp[K], ax = D::O.ax[K], ay = D::O.ay[K], az = D::O.az[K];
  if constexpr (K == 0 || D::O.grp[K > 0 ? K - 1 : 0] != g) {
    const HL* a = p.gf[g];
    float al = hl(a[0], w.r0);
    al = hl_fma(a[1], w.r1, al);
    al = hl_fma(a[2], w.r5, al);
    al = hl_fma(a[3], w.r9, al);
    al = hl_fma(a[4], w.r10, al);
    c[0] = al;
#pragma unroll
    for (int b = 0; b < 3; ++b) c[1 + b] = hl_fma(a[5], w.rU[b], hl(a[6], w.h * w.U[b]));
    const float k9 = hl(a[7], w.r9), k10 = hl(a[8], w.r10);
    c[4] = fmaf(-3.0f, k10, k9);    // q_xx
    c[5] = 2.0f * k9;               // q_yy
    c[6] = hl(a[9], w.r13);         // q_xy
    c[7] = hl(a[9], w.r11);         // q_xz
    c[8] = hl(a[9], w.r12);         // q_yz
  }
  v[0] = c[0];
  if constexpr (C & 1) v[0] = fmaf((float)(ax * ax), c[4], v[0]);
  if constexpr (C & 2) v[0] = fmaf((float)(ay * ay), c[5], v[0]);
  if constexpr (C & 1) v[1] = (float)ax * c[1];
  if constexpr (C & 2) v[2] = (float)ay * c[2];
  if constexpr (C & 4) v[4] = (float)az * c[3];
  if constexpr ((C & 3) == 3) v[3] = (float)(ax * ay) * c[6];
  if constexpr ((C & 5) == 5) v[5] = (float)(ax * az) * c[7];
  if constexpr ((C & 6) == 6) v[6] = (float)(ay * az) * c[8];
  if constexpr (C == 7) {
    // no part odd in all three
    const float p0 = v[0] + v[1], m0 = v[0] - v[1], p1 = v[2] + v[3], m1 = v[2] - v[3];
    const float p2 = v[4] + v[5], m2 = v[4] - v[5], u = v[6];
    const float a0 = p0 + p1, a1 = m0 + m1, a2 = p0 - p1, a3 = m0 - m1;
    const float b0 = p2 + u, b1 = m2 + u, b2 = p2 - u, b3 = m2 - u;
    v[0] = a0 + b0;
    v[1] = a1 + b1;
    v[2] = a2 + b2;
    v[3] = a3 + b3;
    v[4] = a0 - b0;
    v[5] = a1 - b1;
    v[6] = a2 - b2;
    v[7] = a3 - b3;
  } else {
    wht<C>(v);
  }
}

template <class Cfg, int... Ks>
__device__ __forceinline__ void collide_all3(std::integer_sequence<int, Ks...>, const Src3& q, const Fused3Params& p,
                                             const Proj3& w, float a0, float ax, float ay, float az,
                                             float* __restrict__ out) {
  float c[9];
  (
      [&] {
        float v[8];
        classes3<typename Cfg::D, Ks>(p, w, c, v);
        relax_orbit3<Cfg, Ks>(std::make_integer_sequence<int, 8>{}, q, v, a0, ax, ay, az, out);
      }(),
      ...);
}

template <class Cfg>
__global__ void __launch_bounds__(Cfg::TB, Cfg::BLOCKS) fused3d_kernel(const __grid_constant__ Fused3Params p,
                                                                       const float* __restrict__ fin,
                                                                       float* __restrict__ fout) {
  using D = typename Cfg::D;
  // Nx Ny Nz < 2^31 (checked at creation): 32-bit site arithmetic
  const int nsite = p.Nx * p.Ny * p.Nz;
  const int site = (int)(blockIdx.x * blockDim.x + threadIdx.x);
  unsigned fl = 0;
  // the thread's kept populations: column threadIdx.x of a [KEEP][TB] array
  extern __shared__ float kept[];
  if (site < nsite) {
    const int r = site / p.Nx;
    const int x = site - r * p.Nx;
    const int z = r / p.Ny;
    const int y = r - z * p.Ny;
    Src3 q{kept + threadIdx.x, fin, (size_t)(unsigned)p.plane, (unsigned)p.zstride, (unsigned)p.pitch,
           x, y, z, p.Nx, p.Ny, p.Nz};
    using Orb = std::make_integer_sequence<int, D::O.K>;
    // deviation moments N0 Nx Ny Nz T00 T0x T0y T0z Txx Txy Txz Tyy Tyz Tzz
    float M[14];
    acc_all3<Cfg>(Orb{}, q, p, M);
    const SplitSite3 o = split_solve3(p, M, fl);
    const float n = o.n, mr32 = fmaf(p.mb, o.R, 4.0f * o.T);          // mbar K3/K2(zeta)
    const float F = fmaf(p.mY, o.dR, 3.0f * o.Td), G = fmaf(p.mb, o.dR, 4.0f * o.Td);
    const float nm = n * mr32, yy = o.Uy * o.Uy, zz = o.Uz * o.Uz;
    Proj3 w;
    w.r0 = fmaf(p.nr.hi, o.dR, fmaf(p.nr.lo, o.dR, o.nd * o.R));   // n R - n_r R_r
    w.r1 = n * (o.dg - p.k21 * o.dR);
    w.r5 = n * (F + o.dg * fmaf(2.0f, mr32, p.cb00_1) + o.dg * o.dg * mr32);
    w.h = n * fmaf(mr32, o.dg, G);
    w.r9 = nm * (yy - zz);
    w.r10 = nm * (yy + zz - 2.0f * o.Ux * o.Ux);
    w.r11 = nm * o.Ux * o.Uz;
    w.r12 = nm * o.Uy * o.Uz;
    w.r13 = nm * o.Ux * o.Uy;
    w.rU[0] = n * o.Ux;
    w.rU[1] = n * o.Uy;
    w.rU[2] = n * o.Uz;
    w.U[0] = o.Ux;
    w.U[1] = o.Uy;
    w.U[2] = o.Uz;
    const float wv = p.v0 * p.inv_tau;
    float* out = fout + ((unsigned)z * (unsigned)p.zstride + (unsigned)y * (unsigned)p.pitch + (unsigned)x);
    // where the second pass pulls again, its addresses are not the first's for
    // the compiler, which would keep all of them across the site solve
    if constexpr (Cfg::KEEP < D::Q) asm volatile("" : "+r"(q.x), "+r"(q.y), "+r"(q.z));
    collide_all3<Cfg>(Orb{}, q, p, w, o.U0 * p.inv_tau, wv * o.Ux, wv * o.Uy, wv * o.Uz, out);
  }
  report(fl, p.err);
}

template <class Cfg>
constexpr int smem_of = Cfg::KEEP * Cfg::TB * (int)sizeof(float);

template <class Cfg>
cudaError_t launch_fused3d_cfg(const Fused3Params& p, const void* fin, void* fout, cudaStream_t s) {
  const unsigned grid = (unsigned)(((long long)p.Nx * p.Ny * p.Nz + Cfg::TB - 1) / Cfg::TB);
  fused3d_kernel<Cfg><<<grid, Cfg::TB, smem_of<Cfg>, s>>>(p, static_cast<const float*>(fin), static_cast<float*>(fout));
  return cudaGetLastError();
}

template <class Cfg>
cudaError_t launch_fused3d_impl(bool small, const Fused3Params& p, const void* fin, void* fout, cudaStream_t s) {
  if (small) return launch_fused3d_cfg<Small3<Cfg>>(p, fin, fout, s);
  return launch_fused3d_cfg<Cfg>(p, fin, fout, s);
}

// The opt-in to more shared memory than a kernel gets by default (48 KB: only M1's
// blocks of 256 threads need it).  It belongs to the current device, so every
// context asks for it when it is created; nothing is remembered between contexts.
template <class Cfg>
cudaError_t prepare_cfg() {
  if (smem_of<Cfg> <= 48 * 1024) return cudaSuccess;
  return cudaFuncSetAttribute(fused3d_kernel<Cfg>, cudaFuncAttributeMaxDynamicSharedMemorySize, smem_of<Cfg>);
}
template <class Cfg>
cudaError_t prepare_impl(bool small) {
  return small ? prepare_cfg<Small3<Cfg>>() : prepare_cfg<Cfg>();
}

}  // namespace

bool fused3d_small(long long nsite) { return nsite <= kSmall3 * sm_count(); }

cudaError_t prepare_fused3d(int kind, bool small) {
  switch (kind) {
    case 1: return prepare_impl<Cfg3<Stencil3M1>>(small);
    case 2: return prepare_impl<Cfg3<Stencil3G16>>(small);
    case 3: return prepare_impl<Cfg3<Stencil3E5>>(small);
    default: return prepare_impl<Cfg3<Stencil3S2>>(small);
  }
}

cudaError_t launch_fused3d(int kind, bool small, const Fused3Params& p, const void* fin, void* fout, cudaStream_t s) {
  switch (kind) {
    case 1: return launch_fused3d_impl<Cfg3<Stencil3M1>>(small, p, fin, fout, s);
    case 2: return launch_fused3d_impl<Cfg3<Stencil3G16>>(small, p, fin, fout, s);
    case 3: return launch_fused3d_impl<Cfg3<Stencil3E5>>(small, p, fin, fout, s);
    default: return launch_fused3d_impl<Cfg3<Stencil3S2>>(small, p, fin, fout, s);
  }
}

}  // namespace rlbm
