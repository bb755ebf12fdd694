// Stencil-specialised FP64 step of the second-order stencils (storage f_i, all
// arithmetic FP64; see rlbm_fused64.cuh).  Equilibrium of a group's populations:
//   f^eq_i = mult (c0 + c1 n_x + c2 n_y + c3 n_x^2 + c4 n_y^2 + c5 n_x n_y),
// the App. A/B expansion folded per group (the constants gf of StencilBuild),
// evaluated once a reflection orbit.
#include "rlbm_fused64.cuh"

namespace rlbm {
namespace {

template <class Def, int K>
__device__ __forceinline__ void collide64_orbit(const Fused64Params& p, const double (&r)[10], double (&c)[6],
                                                const Pull64& q, const Relax64& rx) {
  constexpr int g = Def::O.grp[K], ax = Def::O.ax[K], ay = Def::O.ay[K];
  constexpr double m = (double)Def::O.mult[K];
  if constexpr (orbit_starts_group<Def, K>()) {
    group_coeffs64(p.gf[g], r, c);
  }
  double E = m == 1.0 ? c[0] : m * c[0];
  if constexpr (ax != 0) E = fma(m * (double)(ax * ax), c[3], E);
  if constexpr (ay != 0) E = fma(m * (double)(ay * ay), c[4], E);
  relax64_orbit<Def, K>(q, rx, E, (m * (double)ax) * c[1], (m * (double)ay) * c[2], (m * (double)(ax * ay)) * c[5]);
}

template <class Def, int... Ks>
__device__ __forceinline__ void collide64_all(std::integer_sequence<int, Ks...>, const Fused64Params& p,
                                              const double (&r)[10], const Pull64& q, const Relax64& rx) {
  double c[6];
  (collide64_orbit<Def, Ks>(p, r, c, q, rx), ...);
}

template <class Def>
__global__ void __launch_bounds__(64, 8) fused_f64_kernel(const __grid_constant__ Fused64Params p,
                                                           const double* __restrict__ fin, double* __restrict__ fout) {
  static_assert(Def::halo <= kMaxDisp, "displacement tables hold kMaxDisp");
  const int s = blockIdx.x * blockDim.x + threadIdx.x;
  unsigned fl = 0;
  if (s < p.Nx * p.Ny) {
    int x, y;
    site_of(s, p.Nx, x, y);
    const Pull64 q{fin, (size_t)p.plane, (unsigned)p.pitch, x, y, p.Nx, p.Ny, p.dxm, p.dym, -1};
    using Orb = std::make_integer_sequence<int, Def::O.K>;
    double M[9];
    acc64_all<Def>(Orb{}, q, p.gm, M);
    const Macro<double> o = solve_site_f64_seeded(M, p.sc, p.rt64, p.rt32, fl);
    double r[10];
    projections64(p.sc, o, 0.0, r);
    const double wv = p.v0 * p.inv_tau;
    const Relax64 rx{o.U0 * p.inv_tau, wv * o.Ux, wv * o.Uy, fout + ((unsigned)y * (unsigned)p.pitch + (unsigned)x),
                     (size_t)p.plane};
    collide64_all<Def>(Orb{}, p, r, q, rx);
  }
  report(fl, p.err);
}

template <class Def>
cudaError_t launch64(const Fused64Params& p, const void* fin, void* fout, cudaStream_t s) {
  const long long nsite = (long long)p.Nx * p.Ny;
  fused_f64_kernel<Def><<<(unsigned)((nsite + 63) / 64), 64, 0, s>>>(p, static_cast<const double*>(fin),
                                                                     static_cast<double*>(fout));
  return cudaGetLastError();
}

}  // namespace

cudaError_t launch_fused_f64(int kind, const Fused64Params& p, const void* fin, void* fout, cudaStream_t s) {
  if (kind == 1) return launch64<StencilM1>(p, fin, fout, s);
  if (kind == 2) return launch64<StencilG16>(p, fin, fout, s);
  if (kind == 3) return launch64<StencilE5>(p, fin, fout, s);
  return launch64<StencilS2>(p, fin, fout, s);
}

}  // namespace rlbm
