"""FP32 3D step kernels on both sides of the rule that gives small lattices
smaller blocks (at most 200 sites an SM of 152): a single site, sides below the
halo, a block with a tail, the last lattice of the small blocks and the first of
the others, against the FP64 kernels.  Tolerance: the FP32 path's 1e-5."""
import numpy as np
import pytest

from paper_1703_04605_gb300 import workloads as W

pytestmark = pytest.mark.gpu

STENCILS = {"M1": W.STENCIL_M1, "G16": W.STENCIL_G16, "E5": W.STENCIL_E5, "S2": W.STENCIL_S2}
SHAPES = [(1, 1, 1), (3, 2, 7), (9, 11, 13), (25, 32, 38), (7, 43, 101)]   # .. 30400 | 30401


@pytest.fixture(scope="module", autouse=True)
def _built():
    from paper_1703_04605_gb300 import build
    build.build()


@pytest.mark.parametrize("name", sorted(STENCILS))
@pytest.mark.parametrize("shape", SHAPES)
def test_against_f64(name, shape):
    from paper_1703_04605_gb300 import Lattice3D
    st = STENCILS[name]
    rng = np.random.default_rng(sum(shape))
    f = {k: 0.05 * rng.uniform(-1, 1, shape) for k in ("n", "ux", "uy", "uz", "T")}
    f["n"] += 1.0
    f["T"] += 1.0
    Nz, Ny, Nx = shape
    got = {}
    for dtype in ("f32", "f64"):
        with Lattice3D(st["groups"], st["m"], 0.9, Nx, Ny, Nz, dtype=dtype, v0=st["v0"]) as lat:
            lat.init(f["n"], f["ux"], f["uy"], f["uz"], f["T"])
            lat.step(4)
            got[dtype] = lat.moments()
    umax = max(np.max(np.abs(got["f64"][k])) for k in ("ux", "uy", "uz"))
    for k in ("n", "T", "e"):
        assert np.max(np.abs(got["f32"][k] / got["f64"][k] - 1)) < 1e-5, k
    for k in ("ux", "uy", "uz"):
        assert np.max(np.abs(got["f32"][k] - got["f64"][k])) / umax < 1e-5, k
