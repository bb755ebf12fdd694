"""Chained step launches (each step comes up while the previous one ends): the
same results as single calls, bit for bit, and under stream capture."""
import numpy as np
import pytest

from gpu_common import smooth_fields
from paper_1703_04605_gb300 import workloads as W

pytestmark = pytest.mark.gpu

CASES = [("M1", "f32", (160, 96), 0), ("E5", "f32", (64, 48), 0), ("E5", "f32", (1100, 1000), 0),
         ("S2", "f32", (70, 33), 1), ("M1", "bf16dev", (90, 70), 0), ("M1", "f64", (40, 20), 0),
         ("O3", "f64", (40, 20), 0)]
ST = {"M1": W.STENCIL_M1, "E5": W.STENCIL_E5, "S2": W.STENCIL_S2, "O3": W.STENCIL_O3}


@pytest.fixture(scope="module", autouse=True)
def _built():
    from paper_1703_04605_gb300 import build
    build.build()


def _lattice(case, stream=None):
    from paper_1703_04605_gb300 import Lattice
    name, dtype, (Nx, Ny), ext = case
    st = ST[name]
    lat = Lattice(st["groups"], st["m"], 0.9, Nx, Ny, dtype=dtype, v0=st["v0"], stream=stream)
    if ext:
        lat.set_extended_sums(ext)
    f = smooth_fields(Nx, Ny, seed=3, dn=0.05, dT=0.05, du=0.05)
    lat.init(f["n"], f["ux"], f["uy"], f["T"])
    return lat


@pytest.mark.parametrize("case", CASES)
def test_chained_equals_single_and_captured(case):
    import torch
    with _lattice(case) as lat:
        for _ in range(24):
            lat.step(1)
            lat.sync()
        ref = lat.moments()
    with _lattice(case) as lat:
        lat.step(24)
        got = lat.moments()
    for k in ref:
        assert np.array_equal(ref[k], got[k]), k
    s = torch.cuda.Stream()
    with torch.cuda.stream(s), _lattice(case, s.cuda_stream) as lat:
        lat.step(4)          # kernels loaded before the capture
        lat.sync()
        g = torch.cuda.CUDAGraph()
        with torch.cuda.graph(g, stream=s):
            lat.step(4)
        for _ in range(5):
            g.replay()
        got = lat.moments()
    for k in ref:
        assert np.array_equal(ref[k], got[k]), k
