// FP64 step of small 2D lattices (any second- or third-order stencil): L lanes a
// site, one warp a block.
//
// An FP64 instruction of a warp holds its SM sub-partition's FP64 unit for 64
// cycles (half a lane a clock) however few warps there are, so a lattice with
// fewer warps than the GPU has sub-partitions (4 an SM) takes as long as one
// warp's FP64 instructions: 741 x 64 cycles in fused_f64_kernel, 23 us.  Here
// the populations of a site are spread over L lanes (table rows in place of
// compile-time constants), their moments summed by shuffles, the site solve
// repeated on every lane: about 308 FP64 instructions a warp at L = 16, 391 at
// L = 8, 566 at L = 4 (Q = 58).  L is the largest of 32, 16, 8 and 4 that gives
// no more warps than sub-partitions (lanes64_for); a lattice with more sites than
// that holds at L = 4 is faster with a lane a site.  Measured, us a step, M1
// (Q = 58): 64 sites 14.0, 800 19.7, 2432 24.5, 4864 28.1 against 30.8 for
// fused_f64_kernel up to 9728 (800 x 1 on step_f64_kernel: 77); third order
// (Q = 100) 64 sites 22.2, 800 23.3, 2432 33.7, 4864 48.1 against 55.3.  What is
// left is the solve's serial FP64 chain and the latency of one pass over memory.
#include "rlbm_fused64.cuh"
#include "rlbm_o3.cuh"
#include "rlbm_pdl.cuh"

namespace rlbm {
namespace {

// Two consecutive FP64 table entries.
__device__ __forceinline__ double2 ld2(const double* p) { return __ldg(reinterpret_cast<const double2*>(p)); }

__device__ __forceinline__ const double* source(const LanesParams& p, const double* fin, int i, int x, int y) {
  const unsigned xs = (unsigned)wrap_sub(x, __ldg(p.shift + i), p.Nx);
  const unsigned ys = (unsigned)wrap_sub(y, __ldg(p.shift + p.Q + i), p.Ny);
  return fin + (ys * (unsigned)p.pitch + xs) + (size_t)p.plane * i;
}

// Equilibrium of one population: second order sum_k n b^(k) (w_i J_k), third
// order n wr_i + sum_l e_l W_il; row: the population's table row.
struct Eq2 {
  double b[NJ];
  __device__ __forceinline__ void prepare(const LanesParams& p, const Macro<double>& o) {
    projections<double>(o, p.sc, b);
  }
  __device__ __forceinline__ double at(const double* row) const {
    double f = 0.0;
#pragma unroll
    for (int k = 0; k < NJ; k += 2) {
      const double2 c = ld2(row + 10 + k);
      f = fma(b[k], c.x, f);
      f = fma(b[k + 1], c.y, f);
    }
    return f;
  }
};
struct Eq3 {
  double e[kO3Mono], n;
  __device__ __forceinline__ void prepare(const LanesParams& p, const Macro<double>& o) {
    o3_deviations<double>(p.sc.mbar, p.c, o.n, o.U0, o.Ux, o.Uy, o.dU, o.dR, o.T - 1.0, o.T, o.R, e, p.sc.inv_m);
    n = o.n;
  }
  __device__ __forceinline__ double at(const double* row) const {
    double f = n * __ldg(row + 9);
#pragma unroll
    for (int l = 0; l < kO3Mono; l += 2) {
      const double2 c = ld2(row + 10 + l);
      f = fma(e[l], c.x, f);
      f = fma(e[l + 1], c.y, f);
    }
    return f;
  }
};

// Into L1, while the previous step finishes: the population table, and the
// R(zeta) slices around T_R, where most temperatures lie.
__device__ __forceinline__ void prefetch_l1(const void* a) { asm volatile("prefetch.global.L1 [%0];" : : "l"(a)); }
__device__ __forceinline__ void prefetch_tables(const LanesParams& p, int entries) {
  for (int k = (int)threadIdx.x * 16; k < entries; k += 32 * 16) prefetch_l1(p.tab + k);   // 128-byte lines
  const long long bits = __double_as_longlong(p.sc.mbar);
  const int e = (int)((bits >> 52) & 0x7ff) - 1023, j = (int)((bits >> 49) & 7);
  const int idx = (e - RT_EMIN) * RT_SEG + j;
  const int k = min(max(idx - 3, 0), RT_NSEG - 7) + (int)threadIdx.x;   // seven slices, a lane each
  if (threadIdx.x < 7) {
    prefetch_l1(p.rt64 + k * RT_NC64);
    prefetch_l1(p.rt32 + k * RT_NC32);
  }
}

// Eq2: rows of kRowLanes2 (p^a/p^0 at 20, 21); Eq3: rows of kRowO3 (at 30, 31).
template <int L, class Eq>
__global__ void __launch_bounds__(32) lanes64_kernel(const __grid_constant__ LanesParams p,
                                                     const double* __restrict__ fin, double* __restrict__ fout) {
  constexpr bool third = std::is_same<Eq, Eq3>::value;
  constexpr int ROW = third ? kRowO3 : kRowLanes2;
  const int lane = (int)threadIdx.x % L;
  const int nsite = p.Nx * p.Ny;
  const int s0 = (int)(blockIdx.x * (32 / L)) + (int)threadIdx.x / L;
  // lanes past the end repeat the last site without storing, so that every
  // lane takes part in the sums over lanes
  const bool live = s0 < nsite;
  const int site = live ? s0 : nsite - 1;
  unsigned fl = 0;
  int x, y;
  site_of(site, p.Nx, x, y);
  prefetch_tables(p, p.Q * ROW);
  pdl_wait();
  double m[9];
#pragma unroll
  for (int k = 0; k < 9; ++k) m[k] = 0.0;
#pragma unroll 4
  for (int i = lane; i < p.Q; i += L) {
    const double f = ld_pop(source(p, fin, i, x, y));
    const double* row = p.tab + i * ROW;
#pragma unroll
    for (int k = 0; k < 8; k += 2) {
      const double2 c = ld2(row + k);
      m[k] = fma(f, c.x, m[k]);
      m[k + 1] = fma(f, c.y, m[k + 1]);
    }
    m[8] = fma(f, __ldg(row + 8), m[8]);
  }
#pragma unroll
  for (int k = 0; k < 9; ++k) {
#pragma unroll
    for (int h = 1; h < L; h <<= 1) m[k] += __shfl_xor_sync(0xffffffffu, m[k], h);
  }
  const Macro<double> o = solve_site_f64_seeded(m, p.sc, p.rt64, p.rt32, fl);
  Eq eq;
  eq.prepare(p, o);
  const double a0 = o.U0 * p.inv_tau, ax = o.Ux * p.inv_tau, ay = o.Uy * p.inv_tau;
  double* out = fout + ((unsigned)y * (unsigned)p.pitch + (unsigned)x);
  if (live) {
#pragma unroll 4
    for (int i = lane; i < p.Q; i += L) {
      const double f = ld_pop(source(p, fin, i, x, y));
      const double* row = p.tab + i * ROW;
      const double e = eq.at(row);
      const double2 v = ld2(row + (third ? 30 : 20));
      const double om = fma(-ay, v.y, fma(-ax, v.x, a0));
      __stcs(out + (size_t)p.plane * i, fma(om, e - f, f));
    }
  }
  report(fl, p.err);
}

template <class Eq>
cudaError_t launch(const LanesParams& p, int L, const double* fin, double* fout, cudaStream_t s) {
  const long long nsite = (long long)p.Nx * p.Ny;
  const unsigned grid = (unsigned)((nsite * L + 31) / 32);
  switch (L) {
    case 4: return launch_pdl(lanes64_kernel<4, Eq>, grid, 32, s, p, fin, fout);
    case 8: return launch_pdl(lanes64_kernel<8, Eq>, grid, 32, s, p, fin, fout);
    case 16: return launch_pdl(lanes64_kernel<16, Eq>, grid, 32, s, p, fin, fout);
    default: return launch_pdl(lanes64_kernel<32, Eq>, grid, 32, s, p, fin, fout);
  }
}

}  // namespace

cudaError_t launch_lanes64(const LanesParams& p, int L, const void* fin, void* fout, cudaStream_t s) {
  const double* f = static_cast<const double*>(fin);
  double* g = static_cast<double*>(fout);
  return p.third ? launch<Eq3>(p, L, f, g, s) : launch<Eq2>(p, L, f, g, s);
}

}  // namespace rlbm
