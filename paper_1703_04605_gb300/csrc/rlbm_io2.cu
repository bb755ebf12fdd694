// Init and read-out of the compiled second-order stencils, FP64 and
// BF16-deviation storage (rlbm_io.cuh; FP32 storage: rlbm_fused.cuh).
#include "rlbm_fused.cuh"
#include "rlbm_io.cuh"

namespace rlbm {
namespace {

// BF16-deviation storage: the values f - r = d + ref of a source site, ref from
// its coefficient word (bf_ref of rlbm_fused.cuh).  Every term is exact in FP32, and
// their sum is carried as an FP32 number and its rounding error, two conversions and
// one addition of the FP64 pipe, which bounds the read-out, in place of five and
// four.  The error itself can take more than 24 bits where a coefficient is far
// smaller than the sum; its own rounding is then carried too, so that nothing is
// lost that an FP64 sum keeps.  Read-out of the 4096^2 flow 17.2 -> 18.0 ms with that,
// of the 2048^2 blast (large parts nearly at rest) 5.2 -> 6.1 ms; carried always
// 20.9 and 6.4 ms.
struct PullBF {
  const unsigned short* fin;
  const uint2* cin;
  size_t plane;
  unsigned pitch;
  int x, y, Nx, Ny;
  const int *dxm, *dym;
  int mask;
};

template <class Def, int I>
__device__ __forceinline__ double pull64(const PullBF& q) {
  constexpr int nx = Def::F.nx[I], ny = Def::F.ny[I], g = Def::F.grp[I], mult = Def::F.mult[I];
  constexpr int word = Def::B.word[I], half = Def::B.half[I];
  const unsigned xs = (unsigned)wrap_sub(q.x, q.dxm[nx + kMaxDisp] & q.mask, q.Nx);
  const unsigned ys = (unsigned)wrap_sub(q.y, q.dym[ny + kMaxDisp] & q.mask, q.Ny);
  const unsigned idx = ys * q.pitch + xs;
  const uint2 c = __ldg(q.cin + idx + q.plane * g);
  const unsigned h = __ldg(q.fin + 2 * (size_t)idx + half + 2 * q.plane * word);
  float s = (float)mult * bf_lo(c.x), t[3] = {0.0f, 0.0f, 0.0f}, e, f = 0.0f;
  if constexpr (nx * nx + ny * ny != 0) s = ex_two_sum(s, (float)(mult * (nx * nx + ny * ny)) * bf_hi(c.y), t[0]);
  if constexpr (ny != 0) s = ex_two_sum(s, (float)(mult * ny) * bf_lo(c.y), t[1]);
  if constexpr (nx != 0) s = ex_two_sum(s, (float)(mult * nx) * bf_hi(c.x), t[2]);
  s = ex_two_sum(s, __uint_as_float(h << 16), e);
  // whether a coefficient left anything (the sign of a zero does not count)
  if (((__float_as_uint(t[0]) | __float_as_uint(t[1]) | __float_as_uint(t[2])) << 1) != 0u) {
#pragma unroll
    for (int k = 0; k < 3; ++k) {
      float u;
      e = ex_two_sum(e, t[k], u);
      f += u;
    }
    return ((double)s + (double)e) + (double)f;
  }
  return (double)s + (double)e;
}

// The bfloat16 nearest to a double, in integer arithmetic: the FP64 pipe, which
// bounds the init, has no part in it.  The double is cut to an FP32 bit pattern
// whose last bit stands for anything cut off (round to odd), so that the second
// rounding is the only one.  Outside FP32's normal range the conversion decides.
__device__ __forceinline__ unsigned short bf16_nearest(double v) {
  const unsigned hi = (unsigned)__double2hiint(v), lo = (unsigned)__double2loint(v);
  const unsigned e = ((hi >> 20) & 0x7ffu) - 896u;   // FP32 exponent field
  if (e - 1u >= 253u) return __bfloat16_as_ushort(__double2bfloat16(v));
  const unsigned f = (hi & 0x80000000u) | (e << 23) | ((hi & 0xfffffu) << 3) | (lo >> 29) | ((lo & 0x1fffffffu) != 0u);
  return __bfloat16_as_ushort(__float2bfloat16_rn(__uint_as_float(f)));
}

// Puts deviations from the site's own reference.
struct PutBF {
  unsigned* out;   // the site's word of word plane 0
  size_t plane;
  template <class Def, int I>
  __device__ __forceinline__ void one(double v) const {
    constexpr int word = Def::B.word[I], half = Def::B.half[I];
    unsigned short* w = reinterpret_cast<unsigned short*>(out + plane * word);
    __stcs(w + half, bf16_nearest(v));
  }
  template <class Def, int I, int J>
  __device__ __forceinline__ void pair(double a, double b) const {
    static_assert(Def::B.word[I] == Def::B.word[J] && Def::B.half[I] == 0, "orbit partners share a word");
    constexpr int word = Def::B.word[I];
    __stcs(out + plane * word, (unsigned)bf16_nearest(a) | ((unsigned)bf16_nearest(b) << 16));
  }
};

// c: the group's equilibrium coefficients, for BF16-deviation storage less those
// of the reference (rounded to bfloat16), so that the orbits' values are the
// deviations themselves.
template <class Def, int K, class Put>
__device__ __forceinline__ void init_orbit(const Io2Params& p, const double (&r)[10], double (&c)[6], const Put& put,
                                           uint2* cout) {
  constexpr int g = Def::O.grp[K], ax = Def::O.ax[K], ay = Def::O.ay[K];
  constexpr double m = (double)Def::O.mult[K];
  if constexpr (orbit_starts_group<Def, K>()) {
    group_coeffs64(p.b.gf[g], r, c);
    if constexpr (std::is_same<Put, PutBF>::value) {
      uint2 cq;
      cq.x = bf_pack((float)c[0], (float)c[1]);
      cq.y = bf_pack((float)c[2], (float)(0.5 * (c[3] + c[4])));
      __stcs(cout + put.plane * g, cq);
      const double q = (double)bf_hi(cq.y);
      c[0] -= (double)bf_lo(cq.x);
      c[1] -= (double)bf_hi(cq.x);
      c[2] -= (double)bf_lo(cq.y);
      c[3] -= q;
      c[4] -= q;
    }
  }
  double E = m == 1.0 ? c[0] : m * c[0];
  if constexpr (ax != 0) E = fma(m * (double)(ax * ax), c[3], E);
  if constexpr (ay != 0) E = fma(m * (double)(ay * ay), c[4], E);
  emit_orbit<Def, K>(put, E, (m * (double)ax) * c[1], (m * (double)ay) * c[2], (m * (double)(ax * ay)) * c[5]);
}

template <class Def, class Put, int... Ks>
__device__ __forceinline__ void init_all(std::integer_sequence<int, Ks...>, const Io2Params& p, const double (&r)[10],
                                         const Put& put, uint2* cout) {
  double c[6];
  (init_orbit<Def, Ks>(p, r, c, put, cout), ...);
}

template <class Def, bool BF>
__global__ void __launch_bounds__(128) init2_kernel(const __grid_constant__ Io2Params p, FieldPtrs fd,
                                                    void* __restrict__ cur, uint2* __restrict__ ccur,
                                                    void* __restrict__ other) {
  const int s = blockIdx.x * blockDim.x + threadIdx.x;
  unsigned fl = 0;
  if (s < p.b.Nx * p.b.Ny) {
    int x, y;
    site_of(s, p.b.Nx, x, y);
    const Macro<double> o = macro_of_fields64(fd.n[s], fd.ux[s], fd.uy[s], fd.T[s], p.b.sc, p.b.rt64, fl);
    double r[10];
    projections64(p.b.sc, o, p.ref, r);
    const unsigned here = (unsigned)y * (unsigned)p.b.pitch + (unsigned)x;
    using Orb = std::make_integer_sequence<int, Def::O.K>;
    if constexpr (BF) {
      const PutBF put{static_cast<unsigned*>(cur) + here, (size_t)p.b.plane};
      init_all<Def>(Orb{}, p, r, put, ccur + here);
      if (s == 0) mark_unwritten(static_cast<uint2*>(other));
    } else {
      const PutPlain<double> put{static_cast<double*>(cur) + here, (size_t)p.b.plane};
      init_all<Def>(Orb{}, p, r, put, nullptr);
      if (s == 0) mark_unwritten(static_cast<double*>(other));
    }
  }
  report(fl, p.b.err);
}

template <class Def, bool BF>
__global__ void __launch_bounds__(64, 8) moments2_kernel(const __grid_constant__ Io2Params p,
                                                         const void* __restrict__ prev,
                                                         const uint2* __restrict__ cprev,
                                                         const void* __restrict__ cur,
                                                         const uint2* __restrict__ ccur, MomentOut mo) {
  const int s = blockIdx.x * blockDim.x + threadIdx.x;
  unsigned fl = 0;
  const long long N = (long long)p.b.Nx * p.b.Ny;
  if (s < N) {
    int x, y;
    site_of(s, p.b.Nx, x, y);
    double m[9];
    using Orb = std::make_integer_sequence<int, Def::O.K>;
    if constexpr (BF) {
      const bool here = is_unwritten(cprev);
      acc64_all<Def>(Orb{},
                     PullBF{static_cast<const unsigned short*>(here ? cur : prev), here ? ccur : cprev,
                            (size_t)p.b.plane, (unsigned)p.b.pitch, x, y, p.b.Nx, p.b.Ny, p.b.dxm, p.b.dym,
                            here ? 0 : -1},
                     p.b.gm, m);
    } else {
      const bool here = is_unwritten(static_cast<const double*>(prev));
      acc64_all<Def>(Orb{},
                     Pull64{static_cast<const double*>(here ? cur : prev), (size_t)p.b.plane, (unsigned)p.b.pitch, x,
                            y, p.b.Nx, p.b.Ny, p.b.dxm, p.b.dym, here ? 0 : -1},
                     p.b.gm, m);
    }
#pragma unroll
    for (int k = 0; k < 9; ++k) m[k] += p.mref[k];
    const Macro<double> o = solve_site_f64_seeded(m, p.b.sc, p.b.rt64, p.b.rt32, fl);
    write_planes64(mo, N, s, m, o);
  }
  report(fl, p.b.err);
}

template <class Def>
cudaError_t init2(bool bf, const Io2Params& p, FieldPtrs f, void* cur, void* ccur, void* other, cudaStream_t s) {
  const unsigned grid = (unsigned)(((long long)p.b.Nx * p.b.Ny + 127) / 128);
  if (bf) init2_kernel<Def, true><<<grid, 128, 0, s>>>(p, f, cur, static_cast<uint2*>(ccur), other);
  else init2_kernel<Def, false><<<grid, 128, 0, s>>>(p, f, cur, nullptr, other);
  return cudaGetLastError();
}

template <class Def>
cudaError_t moments2(bool bf, const Io2Params& p, const void* prev, const void* cprev, const void* cur,
                     const void* ccur, MomentOut mo, cudaStream_t s) {
  const unsigned grid = (unsigned)(((long long)p.b.Nx * p.b.Ny + 63) / 64);
  if (bf) moments2_kernel<Def, true><<<grid, 64, 0, s>>>(p, prev, static_cast<const uint2*>(cprev), cur,
                                                           static_cast<const uint2*>(ccur), mo);
  else moments2_kernel<Def, false><<<grid, 64, 0, s>>>(p, prev, nullptr, cur, nullptr, mo);
  return cudaGetLastError();
}

}  // namespace

cudaError_t launch_init2(int kind, bool bf, const Io2Params& p, FieldPtrs f, void* cur, void* ccur, void* other,
                         cudaStream_t s) {
  if (kind == 1) return init2<StencilM1>(bf, p, f, cur, ccur, other, s);
  if (kind == 2) return init2<StencilG16>(bf, p, f, cur, ccur, other, s);
  if (kind == 3) return init2<StencilE5>(bf, p, f, cur, ccur, other, s);
  return init2<StencilS2>(bf, p, f, cur, ccur, other, s);
}

cudaError_t launch_moments2(int kind, bool bf, const Io2Params& p, const void* prev, const void* cprev,
                            const void* cur, const void* ccur, MomentOut mo, cudaStream_t s) {
  if (kind == 1) return moments2<StencilM1>(bf, p, prev, cprev, cur, ccur, mo, s);
  if (kind == 2) return moments2<StencilG16>(bf, p, prev, cprev, cur, ccur, mo, s);
  if (kind == 3) return moments2<StencilE5>(bf, p, prev, cprev, cur, ccur, mo, s);
  return moments2<StencilS2>(bf, p, prev, cprev, cur, ccur, mo, s);
}

}  // namespace rlbm
