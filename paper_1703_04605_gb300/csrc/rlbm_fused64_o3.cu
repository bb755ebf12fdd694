// Stencil-specialised FP64 third-order step (storage f_i, all arithmetic FP64;
// rlbm_fused64.cuh).  Equilibrium f^eq_i = n wr_i + sum_l e_l W_il, e_l = n dmu_l
// (rlbm_o3.cuh), summed once a reflection orbit over the parity classes of the
// twenty monomials (as rlbm_fused_o3.cu): 21 FP64 instructions a quartet of
// populations instead of 84.
#include "rlbm_fused64_o3.cuh"

namespace rlbm {
namespace {

struct RelaxUse {
  const Pull64& q;
  const Relax64& rx;
  template <class Def, int K>
  __device__ __forceinline__ void at(double E, double X, double Y, double Z) const {
    relax64_orbit<Def, K>(q, rx, E, X, Y, Z);
  }
};

// Six blocks of 64 threads an SM (168 registers): the sets of Q = 99 and 100 spill at
// most 12 bytes so, those of Q = 133-149 164 to 628.  Measured on Q = 100 (256^2
// 228 us a step).
template <class Def>
__global__ void __launch_bounds__(64, 6) fused_f64_o3_kernel(const __grid_constant__ FusedO364Params p,
                                                             const double* __restrict__ fin,
                                                             double* __restrict__ fout) {
  static_assert(Def::halo <= kMaxDisp && Def::O.K <= kMaxOrbO3, "table sizes");
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
    double e[kO3Mono];
    deviations64(p, o, e);
    const double wv = p.v0 * p.inv_tau;
    const Relax64 rx{o.U0 * p.inv_tau, wv * o.Ux, wv * o.Uy, fout + ((unsigned)y * (unsigned)p.pitch + (unsigned)x),
                     (size_t)p.plane};
    all_orbits_o3<Def>(Orb{}, p, e, o.n, RelaxUse{q, rx});
  }
  report(fl, p.err);
}

template <class Def>
cudaError_t launch64(const FusedO364Params& p, const void* fin, void* fout, cudaStream_t s) {
  const long long nsite = (long long)p.Nx * p.Ny;
  fused_f64_o3_kernel<Def><<<(unsigned)((nsite + 63) / 64), 64, 0, s>>>(p, static_cast<const double*>(fin),
                                                                        static_cast<double*>(fout));
  return cudaGetLastError();
}

}  // namespace

cudaError_t launch_fused_f64_o3(int kind, const FusedO364Params& p, const void* fin, void* fout, cudaStream_t s) {
  switch (kind) {
    case 5: return launch64<StencilO3M5>(p, fin, fout, s);
    case 6: return launch64<StencilO3D>(p, fin, fout, s);
    case 7: return launch64<StencilO3E>(p, fin, fout, s);
    case 8: return launch64<StencilO3A>(p, fin, fout, s);
    case 9: return launch64<StencilO3B>(p, fin, fout, s);
    default: return launch64<StencilO3C>(p, fin, fout, s);
  }
}

}  // namespace rlbm
