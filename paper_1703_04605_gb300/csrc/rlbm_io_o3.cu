// Init and read-out of the compiled third-order stencils on 2D lattices, FP64 and
// FP32 storage (rlbm_io.cuh).
#include "rlbm_fused64_o3.cuh"
#include "rlbm_io.cuh"

namespace rlbm {
namespace {

template <class Put>
struct EmitUse {
  const Put& put;
  template <class Def, int K>
  __device__ __forceinline__ void at(double E, double X, double Y, double Z) const {
    emit_orbit<Def, K>(put, E, X, Y, Z);
  }
};

template <class Def, typename S>
__global__ void __launch_bounds__(128) init_o3c_kernel(const __grid_constant__ IoO3Params p, FieldPtrs fd,
                                                       S* __restrict__ cur, S* __restrict__ other) {
  const int s = blockIdx.x * blockDim.x + threadIdx.x;
  unsigned fl = 0;
  if (s < p.b.Nx * p.b.Ny) {
    int x, y;
    site_of(s, p.b.Nx, x, y);
    const Macro<double> o = macro_of_fields64(fd.n[s], fd.ux[s], fd.uy[s], fd.T[s], p.b.sc, p.b.rt64, fl);
    double e[kO3Mono];
    deviations64(p.b, o, e);
    const PutPlain<S> put{cur + ((unsigned)y * (unsigned)p.b.pitch + (unsigned)x), (size_t)p.b.plane};
    all_orbits_o3<Def>(std::make_integer_sequence<int, Def::O.K>{}, p.b, e, o.n - p.nref, EmitUse<PutPlain<S>>{put});
    if (s == 0) mark_unwritten(other);
  }
  report(fl, p.b.err);
}

template <typename S>
struct PullOf;
template <>
struct PullOf<double> {
  using type = Pull64;
};
template <>
struct PullOf<float> {
  using type = Pull32;
};

template <class Def, typename S>
__global__ void __launch_bounds__(64, 8) moments_o3c_kernel(const __grid_constant__ IoO3Params p,
                                                            const S* __restrict__ prev,
                                                            const S* __restrict__ cur, MomentOut mo) {
  const int s = blockIdx.x * blockDim.x + threadIdx.x;
  unsigned fl = 0;
  const long long N = (long long)p.b.Nx * p.b.Ny;
  if (s < N) {
    int x, y;
    site_of(s, p.b.Nx, x, y);
    double m[9];
    const bool here = is_unwritten(prev);
    const typename PullOf<S>::type q{here ? cur : prev, (size_t)p.b.plane, (unsigned)p.b.pitch, x, y, p.b.Nx, p.b.Ny,
                                     p.b.dxm, p.b.dym, here ? 0 : -1};
    acc64_all<Def>(std::make_integer_sequence<int, Def::O.K>{}, q, p.b.gm, m);
#pragma unroll
    for (int k = 0; k < 9; ++k) m[k] += p.mref[k];
    const Macro<double> o = solve_site_f64_seeded(m, p.b.sc, p.b.rt64, p.b.rt32, fl);
    write_planes64(mo, N, s, m, o);
  }
  report(fl, p.b.err);
}

template <class Def>
cudaError_t init3(bool f64, const IoO3Params& p, FieldPtrs f, void* cur, void* other, cudaStream_t s) {
  const unsigned grid = (unsigned)(((long long)p.b.Nx * p.b.Ny + 127) / 128);
  if (f64) init_o3c_kernel<Def, double><<<grid, 128, 0, s>>>(p, f, static_cast<double*>(cur), static_cast<double*>(other));
  else init_o3c_kernel<Def, float><<<grid, 128, 0, s>>>(p, f, static_cast<float*>(cur), static_cast<float*>(other));
  return cudaGetLastError();
}

template <class Def>
cudaError_t moments3(bool f64, const IoO3Params& p, const void* prev, const void* cur, MomentOut mo,
                     cudaStream_t s) {
  const unsigned grid = (unsigned)(((long long)p.b.Nx * p.b.Ny + 63) / 64);
  if (f64)
    moments_o3c_kernel<Def, double><<<grid, 64, 0, s>>>(p, static_cast<const double*>(prev),
                                                        static_cast<const double*>(cur), mo);
  else
    moments_o3c_kernel<Def, float><<<grid, 64, 0, s>>>(p, static_cast<const float*>(prev),
                                                       static_cast<const float*>(cur), mo);
  return cudaGetLastError();
}

}  // namespace

cudaError_t launch_init_o3c(int kind, bool f64, const IoO3Params& p, FieldPtrs f, void* cur, void* other,
                            cudaStream_t s) {
  switch (kind) {
    case 5: return init3<StencilO3M5>(f64, p, f, cur, other, s);
    case 6: return init3<StencilO3D>(f64, p, f, cur, other, s);
    case 7: return init3<StencilO3E>(f64, p, f, cur, other, s);
    case 8: return init3<StencilO3A>(f64, p, f, cur, other, s);
    case 9: return init3<StencilO3B>(f64, p, f, cur, other, s);
    default: return init3<StencilO3C>(f64, p, f, cur, other, s);
  }
}

cudaError_t launch_moments_o3c(int kind, bool f64, const IoO3Params& p, const void* prev, const void* cur,
                               MomentOut mo, cudaStream_t s) {
  switch (kind) {
    case 5: return moments3<StencilO3M5>(f64, p, prev, cur, mo, s);
    case 6: return moments3<StencilO3D>(f64, p, prev, cur, mo, s);
    case 7: return moments3<StencilO3E>(f64, p, prev, cur, mo, s);
    case 8: return moments3<StencilO3A>(f64, p, prev, cur, mo, s);
    case 9: return moments3<StencilO3B>(f64, p, prev, cur, mo, s);
    default: return moments3<StencilO3C>(f64, p, prev, cur, mo, s);
  }
}

}  // namespace rlbm
