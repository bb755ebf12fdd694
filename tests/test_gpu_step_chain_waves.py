"""Chained step launches on lattices of many waves of blocks, where the next step's
blocks come up in the places of retiring ones: the same results as single calls, bit
for bit, on ragged lattices of every kernel form that is chained."""
import numpy as np
import pytest

from gpu_common import smooth_fields
from paper_1703_04605_gb300 import workloads as W

pytestmark = pytest.mark.gpu

ST = {"M1": W.STENCIL_M1, "G16": W.STENCIL_G16, "E5": W.STENCIL_E5, "S2": W.STENCIL_S2}
# E5 FP32 is chained up to 3 2^17 sites: the last lattice below that
CASES = [("M1", "f32", (1011, 777), 0), ("G16", "f32", (1011, 777), 0), ("M1", "bf16dev", (1011, 777), 0),
         ("E5", "bf16dev", (1011, 777), 0), ("S2", "f32", (1011, 777), 1), ("M1", "f32", (1011, 777), 2),
         ("E5", "f32", (627, 626), 0)]


@pytest.fixture(scope="module", autouse=True)
def _built():
    from paper_1703_04605_gb300 import build
    build.build()


@pytest.mark.parametrize("name,dtype,size,ext", CASES)
def test_waves(name, dtype, size, ext):
    from paper_1703_04605_gb300 import Lattice
    st, (Nx, Ny) = ST[name], size
    f = smooth_fields(Nx, Ny, seed=3, dn=0.05, dT=0.05, du=0.05)
    out = []
    for chained in (False, True):
        with Lattice(st["groups"], st["m"], 0.9, Nx, Ny, dtype=dtype, v0=st["v0"]) as lat:
            if ext:
                lat.set_extended_sums(ext)
            lat.init(f["n"], f["ux"], f["uy"], f["T"])
            if chained:
                lat.step(40)
            else:
                for _ in range(40):
                    lat.step(1)
                    lat.sync()
            out.append(lat.moments())
    for k in out[0]:
        assert np.array_equal(out[0][k], out[1][k]), k
