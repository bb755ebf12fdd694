"""Compiled FP32 third-order 3D kernel against the oracle where it can go wrong:
lattices exactly a halo (3) wide, sides below two halos, blocks of 64 with a
tail.  Tolerances of the FP32 third-order 3D path: n, T 1e-5, u 1e-4."""
import numpy as np
import pytest

from gpu_common import oracle_lattice
from paper_1703_04605_gb300 import workloads as W

pytestmark = pytest.mark.gpu

ST = W.STENCIL_O3


@pytest.fixture(scope="module", autouse=True)
def _built():
    from paper_1703_04605_gb300 import build
    build.build()


@pytest.mark.parametrize("shape", [(3, 3, 3), (3, 4, 5), (7, 3, 13), (12, 8, 9)])
def test_against_oracle(shape):
    from oracle import lattice as OL
    from paper_1703_04605_gb300 import Lattice3D
    rng = np.random.default_rng(sum(shape))
    f = {k: 0.05 * rng.uniform(-1, 1, shape) for k in ("n", "ux", "uy", "uz", "T")}
    f["n"] += 1.0
    f["T"] += 1.0
    st = oracle_lattice(ST, 0.9, shape[1:]).st
    o = OL.Lattice(st, 0.9, shape, two_d=False)
    o.init(f["n"], f["ux"], f["uy"], f["T"], f["uz"])
    o.step(4)
    ref = o.macros()
    Nz, Ny, Nx = shape
    with Lattice3D(ST["groups"], ST["m"], 0.9, Nx, Ny, Nz, dtype="f32", v0=ST["v0"]) as lat:
        lat.init(f["n"], f["ux"], f["uy"], f["uz"], f["T"])
        lat.step(4)
        got = lat.moments()
    umax = max(np.max(np.abs(ref[k])) for k in ("ux", "uy", "uz"))
    assert np.max(np.abs(got["n"] / ref["n"] - 1)) < 1e-5
    assert np.max(np.abs(got["T"] / ref["T"] - 1)) < 1e-5
    for k in ("ux", "uy", "uz"):
        assert np.max(np.abs(got[k] - ref[k])) / umax < 1e-4, k
