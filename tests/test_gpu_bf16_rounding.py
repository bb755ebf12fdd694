"""The BF16 init's rounding of a double to the nearest bfloat16 (ties to even), as
compiled for the device: ties and their neighbours, double-rounding traps, zeros,
subnormal and overflowing values, infinities and NaN, against the rounding done
exactly by powers of two."""
import ctypes as C
import os
import subprocess

import numpy as np
import pytest

pytestmark = pytest.mark.gpu

SOURCE = r"""
#include "rlbm_io2.cu"
namespace rlbm {
namespace {
__global__ void round_all(const double* v, unsigned short* o, int n) {
  const int i = blockIdx.x * blockDim.x + threadIdx.x;
  if (i < n) o[i] = bf16_nearest(v[i]);
}
}  // namespace
}  // namespace rlbm
extern "C" int round_bf16(const double* v, unsigned short* o, int n) {
  double* dv = nullptr;
  unsigned short* dout = nullptr;
  cudaError_t e = cudaMalloc(&dv, n * sizeof(double));
  if (e == cudaSuccess) e = cudaMalloc(&dout, n * sizeof(unsigned short));
  if (e == cudaSuccess) e = cudaMemcpy(dv, v, n * sizeof(double), cudaMemcpyHostToDevice);
  if (e == cudaSuccess) {
    rlbm::round_all<<<(n + 127) / 128, 128>>>(dv, dout, n);
    e = cudaMemcpy(o, dout, n * sizeof(unsigned short), cudaMemcpyDeviceToHost);
  }
  cudaFree(dv);
  cudaFree(dout);
  return (int)e;
}
"""


def _nearest(v):
    """bfloat16 bits: 8 significant bits, exponents from -126, by exact scaling and rint."""
    with np.errstate(invalid="ignore", over="ignore", divide="ignore"):
        a = np.abs(v)
        ex = np.maximum(np.frexp(a)[1] - 1, -126)
        step = np.ldexp(1.0, ex - 7)
        r = np.rint(a / step) * step
        r = np.where(r >= 2.0 ** 128, np.inf, r)
        bits = (r.astype(np.float32).view(np.uint32) >> 16).astype(np.uint16)
    return bits | np.where(np.signbit(v), 0x8000, 0).astype(np.uint16)


def test_rounding(tmp_path):
    from paper_1703_04605_gb300 import build as B
    src, lib = tmp_path / "round.cu", tmp_path / "round.so"
    src.write_text(SOURCE)
    subprocess.run([B._nvcc(), *B.GENCODE, "-O3", "-std=c++17", "-shared", "-Xcompiler", "-fPIC", "-I", B.CSRC, "-I",
                    os.path.join(B.ROOT, "include"), str(src), "-o", str(lib)], check=True, capture_output=True)
    rng = np.random.default_rng(1)
    k = np.arange(-133, 129)
    base = np.ldexp(1.0 + rng.integers(0, 256, k.size) / 256.0, k)          # every other one a tie
    near = [base * (1 + s * 2.0 ** -b) for s in (-1, 1) for b in (24, 25, 33, 40, 52)]
    small = np.ldexp(rng.integers(0, 4096, 500) / 16.0, -133)                # subnormal, ties among them
    edges = np.array([0.0, 2.0 ** -1074, 2.0 ** -134, 2.0 ** -134 * (1 + 2.0 ** -52), 2.0 ** -126, 2.0 ** -126 * (1 - 2.0 ** -53),
                      255.5 * 2.0 ** 120, np.nextafter(255.5 * 2.0 ** 120, 0), 2.0 ** 128, 1e300, np.inf])
    v = np.concatenate([base, *near, small, edges, np.ldexp(rng.uniform(1, 2, 20000), rng.integers(-140, 130, 20000))])
    v = np.concatenate([v, -v])
    out = np.empty(v.size + 1, np.uint16)
    full = np.append(v, np.nan)
    f = C.CDLL(str(lib)).round_bf16
    assert f(full.ctypes.data_as(C.c_void_p), out.ctypes.data_as(C.c_void_p), C.c_int(full.size)) == 0
    want = _nearest(v)
    bad = np.nonzero(out[:-1] != want)[0]
    assert bad.size == 0, [(v[i].hex(), hex(out[i]), hex(want[i])) for i in bad[:8]]
    assert (out[-1] & 0x7fff) > 0x7f80
