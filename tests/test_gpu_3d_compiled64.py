"""Compiled FP64 3D kernels (step, init, read-out; both orders) against the
oracle at the edges of their forms: a single site, sides below the halo, blocks
of 64 with a tail; the read-out right after the init (S_0 in place).
Tolerance: the FP64 path's 1e-12."""
import numpy as np
import pytest

from gpu_common import oracle_lattice
from paper_1703_04605_gb300 import workloads as W

pytestmark = pytest.mark.gpu

STENCILS = {"M1": W.STENCIL_M1, "G16": W.STENCIL_G16, "E5": W.STENCIL_E5, "S2": W.STENCIL_S2, "O3": W.STENCIL_O3}


@pytest.fixture(scope="module", autouse=True)
def _built():
    from paper_1703_04605_gb300 import build
    build.build()


@pytest.mark.parametrize("name", sorted(STENCILS))
@pytest.mark.parametrize("shape,steps", [((1, 1, 1), 2), ((2, 5, 3), 3), ((7, 8, 9), 3), ((4, 6, 5), 0)])
def test_against_oracle(name, shape, steps):
    from oracle import lattice as OL
    from paper_1703_04605_gb300 import Lattice3D
    st = STENCILS[name]
    rng = np.random.default_rng(sum(shape) + steps)
    f = {k: 0.05 * rng.uniform(-1, 1, shape) for k in ("n", "ux", "uy", "uz", "T")}
    f["n"] += 1.0
    f["T"] += 1.0
    o = OL.Lattice(oracle_lattice(st, 0.9, shape[1:]).st, 0.9, shape, two_d=False)
    o.init(f["n"], f["ux"], f["uy"], f["T"], f["uz"])
    o.step(steps)
    ref = o.macros()
    Nz, Ny, Nx = shape
    with Lattice3D(st["groups"], st["m"], 0.9, Nx, Ny, Nz, dtype="f64", v0=st["v0"]) as lat:
        lat.init(f["n"], f["ux"], f["uy"], f["uz"], f["T"])
        lat.step(steps)
        got = lat.moments()
    umax = max(np.max(np.abs(ref[k])) for k in ("ux", "uy", "uz"))
    for k in ("n", "T", "e"):
        assert np.max(np.abs(got[k] / ref[k] - 1)) < 1e-12, k
    for k in ("ux", "uy", "uz"):
        assert np.max(np.abs(got[k] - ref[k])) / umax < 1e-12, k
