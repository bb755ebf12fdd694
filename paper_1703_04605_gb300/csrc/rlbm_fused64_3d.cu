// FP64 step, and init and read-out in FP64 and FP32 storage, of the compiled
// stencils on native 3D lattices (rlbm_fused64_3d.cuh).
#include "rlbm_fused64_3d.cuh"

namespace rlbm {
namespace {

template <class P>
__device__ __forceinline__ bool site_of3(const P& p, int& x, int& y, int& z, int& s) {
  s = (int)(blockIdx.x * blockDim.x + threadIdx.x);   // Nx Ny Nz < 2^31
  const int r = s / p.Nx;
  x = s - r * p.Nx;
  z = r / p.Ny;
  y = r - z * p.Ny;
  return s < p.Nx * p.Ny * p.Nz;
}

template <class P, typename S>
__device__ __forceinline__ Pull3<S> pull_of(const P& p, const S* fin, int x, int y, int z, int mask = -1) {
  return Pull3<S>{fin, (size_t)p.plane, (unsigned)p.zstride, (unsigned)p.pitch, x, y, z, p.Nx, p.Ny, p.Nz,
                  p.dxm, p.dym, p.dzm, mask};
}

struct Relax3 {
  double a0, a[3];
  double* out;
};

template <class D, int I>
__device__ __forceinline__ void relax3(const Pull3<double>& q, const Relax3& r, double e) {
  constexpr int nx = D::U.nx[I], ny = D::U.ny[I], nz = D::U.nz[I];
  double om = r.a0;
  if constexpr (nx != 0) om = fma(-(double)nx, r.a[0], om);
  if constexpr (ny != 0) om = fma(-(double)ny, r.a[1], om);
  if constexpr (nz != 0) om = fma(-(double)nz, r.a[2], om);
  const double v = pull3d<D, I>(q);
  __stcs(r.out + q.plane * I, fma(om, e - v, v));
}

template <class D, int K, class P, class Eq, int... T>
__device__ __forceinline__ void relax_octant(std::integer_sequence<int, T...>, const P& p, Eq& eq,
                                             const Pull3<double>& q, const Relax3& r) {
  double v[8];
  eq.template orbit<D, K>(p, v);
  (
      [&] {
        if constexpr ((T & ~octant_comps<D, K>()) == 0) {
          constexpr int I = D::O.idx[K][T];
          relax3<D, I>(q, r, v[T]);
        }
      }(),
      ...);
}

template <class D, class P, class Eq, int... Ks>
__device__ __forceinline__ void relax_octants(std::integer_sequence<int, Ks...>, const P& p, Eq& eq,
                                              const Pull3<double>& q, const Relax3& r) {
  (relax_octant<D, Ks>(std::make_integer_sequence<int, 8>{}, p, eq, q, r), ...);
}

template <class D, class P>
__global__ void __launch_bounds__(64, D::Q <= 90 ? 8 : 6) step3c_kernel(const __grid_constant__ P p, const double* __restrict__ fin,
                                                       double* __restrict__ fout) {
  static_assert(D::U.halo <= kMaxDisp, "displacement tables hold kMaxDisp");
  int x, y, z, s;
  unsigned fl = 0;
  if (site_of3(p, x, y, z, s)) {
    Pull3<double> q = pull_of(p, fin, x, y, z);
    using Orb = std::make_integer_sequence<int, D::O.K>;
    double M[14];
    acc_octants<D>(Orb{}, q, p.gm, M);
    const Mac3 o = solve3_seeded(M, p.sc, p.rt64, p.rt32, fl);
    typename EqOf<P>::type eq;
    eq.prepare(p, o);
    const double w = p.v0 * p.inv_tau;
    const Relax3 r{o.U0 * p.inv_tau, {w * o.Ux, w * o.Uy, w * o.Uz},
                   fout + ((unsigned)z * (unsigned)p.zstride + (unsigned)y * (unsigned)p.pitch + (unsigned)x)};
    // the second pass pulls again: hide that its addresses are the first's, or
    // the compiler keeps all of them across the site solve
    asm volatile("" : "+r"(q.x), "+r"(q.y), "+r"(q.z));
    relax_octants<D>(Orb{}, p, eq, q, r);
  }
  report(fl, p.err);
}

template <class D, int K, class P, class Eq, typename S, int... T>
__device__ __forceinline__ void put_octant(std::integer_sequence<int, T...>, const P& p, Eq& eq, S* out) {
  double v[8];
  eq.template orbit<D, K>(p, v);
  (
      [&] {
        if constexpr ((T & ~octant_comps<D, K>()) == 0) {
          constexpr int I = D::O.idx[K][T];
          __stcs(out + (size_t)p.plane * I, (S)v[T]);
        }
      }(),
      ...);
}

template <class D, class P, class Eq, typename S, int... Ks>
__device__ __forceinline__ void put_octants(std::integer_sequence<int, Ks...>, const P& p, Eq& eq, S* out) {
  (put_octant<D, Ks>(std::make_integer_sequence<int, 8>{}, p, eq, out), ...);
}

template <class D, class P, typename S>
__global__ void __launch_bounds__(64, 8) init3c_kernel(const __grid_constant__ P p, Field3Ptrs f, S* __restrict__ cur,
                                                      S* __restrict__ other) {
  int x, y, z, s;
  unsigned fl = 0;
  if (site_of3(p, x, y, z, s)) {
    const Mac3 o = mac3_of_fields(f.n[s], f.ux[s], f.uy[s], f.uz[s], f.T[s], p.sc, p.rt64, fl);
    typename EqOf<P>::type eq;
    eq.prepare(p, o);
    put_octants<D>(std::make_integer_sequence<int, D::O.K>{}, p, eq,
                   cur + ((unsigned)z * (unsigned)p.zstride + (unsigned)y * (unsigned)p.pitch + (unsigned)x));
    if (s == 0) mark_unwritten(other);
  }
  report(fl, p.err);
}

template <class D, class P, typename S>
__global__ void __launch_bounds__(64, 8) moments3c_kernel(const __grid_constant__ P p, const S* __restrict__ prev,
                                                          const S* __restrict__ cur, MomentOut mo) {
  int x, y, z, s;
  unsigned fl = 0;
  if (site_of3(p, x, y, z, s)) {
    const long long N = (long long)p.Nx * p.Ny * p.Nz;
    double m[14];
    const bool here = is_unwritten(prev);
    acc_octants<D>(std::make_integer_sequence<int, D::O.K>{}, pull_of(p, here ? cur : prev, x, y, z, here ? 0 : -1),
                   p.gm, m);
#pragma unroll
    for (int k = 0; k < 14; ++k) m[k] += p.mref[k];
    const Mac3 o = solve3_seeded(m, p.sc, p.rt64, p.rt32, fl);
    const double iU = rcp64(o.U0);
    double* out = mo.out;
    long long plane = 0;
    if (mo.mask & RLBM_M_N) out[(plane++) * N + s] = o.n;
    if (mo.mask & RLBM_M_UX) out[(plane++) * N + s] = o.Ux * iU;
    if (mo.mask & RLBM_M_UY) out[(plane++) * N + s] = o.Uy * iU;
    if (mo.mask & RLBM_M_T) out[(plane++) * N + s] = o.T;
    if (mo.mask & RLBM_M_E) out[(plane++) * N + s] = o.e;
    if (mo.mask & RLBM_M_NVEC) {
#pragma unroll
      for (int k = 0; k < 4; ++k) out[(plane++) * N + s] = m[k];
    }
    if (mo.mask & RLBM_M_TMN) {
#pragma unroll
      for (int k = 4; k < 14; ++k) out[(plane++) * N + s] = m[k];
    }
    if (mo.mask & RLBM_M_UZ) out[(plane++) * N + s] = o.Uz * iU;
  }
  report(fl, p.err);
}

template <class P>
unsigned grid64(const P& p) {
  return (unsigned)(((long long)p.Nx * p.Ny * p.Nz + 63) / 64);
}

template <class D, class P>
cudaError_t step3c(const P& p, const void* fin, void* fout, cudaStream_t s) {
  step3c_kernel<D, P><<<grid64(p), 64, 0, s>>>(p, static_cast<const double*>(fin), static_cast<double*>(fout));
  return cudaGetLastError();
}

template <class D, class P>
cudaError_t init3c(bool f64, const P& p, Field3Ptrs f, void* cur, void* other, cudaStream_t s) {
  if (f64)
    init3c_kernel<D, P, double><<<grid64(p), 64, 0, s>>>(p, f, static_cast<double*>(cur), static_cast<double*>(other));
  else
    init3c_kernel<D, P, float><<<grid64(p), 64, 0, s>>>(p, f, static_cast<float*>(cur), static_cast<float*>(other));
  return cudaGetLastError();
}

template <class D, class P>
cudaError_t moments3c(bool f64, const P& p, const void* prev, const void* cur, MomentOut mo, cudaStream_t s) {
  if (f64)
    moments3c_kernel<D, P, double><<<grid64(p), 64, 0, s>>>(p, static_cast<const double*>(prev),
                                                            static_cast<const double*>(cur), mo);
  else
    moments3c_kernel<D, P, float><<<grid64(p), 64, 0, s>>>(p, static_cast<const float*>(prev),
                                                           static_cast<const float*>(cur), mo);
  return cudaGetLastError();
}

}  // namespace

cudaError_t launch_step3c(int kind, const C3Params2& p, const void* fin, void* fout, cudaStream_t s) {
  switch (kind) {
    case 1: return step3c<Stencil3M1>(p, fin, fout, s);
    case 2: return step3c<Stencil3G16>(p, fin, fout, s);
    case 3: return step3c<Stencil3E5>(p, fin, fout, s);
    default: return step3c<Stencil3S2>(p, fin, fout, s);
  }
}
cudaError_t launch_step3c(const C3Params3& p, const void* fin, void* fout, cudaStream_t s) {
  return step3c<Stencil3O3M5>(p, fin, fout, s);
}

cudaError_t launch_init3c(int kind, bool f64, const C3Params2& p, Field3Ptrs f, void* cur, void* other, cudaStream_t s) {
  switch (kind) {
    case 1: return init3c<Stencil3M1>(f64, p, f, cur, other, s);
    case 2: return init3c<Stencil3G16>(f64, p, f, cur, other, s);
    case 3: return init3c<Stencil3E5>(f64, p, f, cur, other, s);
    default: return init3c<Stencil3S2>(f64, p, f, cur, other, s);
  }
}
cudaError_t launch_init3c(bool f64, const C3Params3& p, Field3Ptrs f, void* cur, void* other, cudaStream_t s) {
  return init3c<Stencil3O3M5>(f64, p, f, cur, other, s);
}

cudaError_t launch_moments3c(int kind, bool f64, const C3Params2& p, const void* prev, const void* cur, MomentOut mo,
                             cudaStream_t s) {
  switch (kind) {
    case 1: return moments3c<Stencil3M1>(f64, p, prev, cur, mo, s);
    case 2: return moments3c<Stencil3G16>(f64, p, prev, cur, mo, s);
    case 3: return moments3c<Stencil3E5>(f64, p, prev, cur, mo, s);
    default: return moments3c<Stencil3S2>(f64, p, prev, cur, mo, s);
  }
}
cudaError_t launch_moments3c(bool f64, const C3Params3& p, const void* prev, const void* cur, MomentOut mo,
                             cudaStream_t s) {
  return moments3c<Stencil3O3M5>(f64, p, prev, cur, mo, s);
}

}  // namespace rlbm
