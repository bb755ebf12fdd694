"""Compiled FP32 second-order 3D steps on lattices exactly a halo wide and a little
more, where every pull wraps: against the FP64 kernels, and the step kernel that
info() reports is the compiled one (below a halo: the table-driven one).
Tolerance: the FP32 path's 1e-5."""
import numpy as np
import pytest

from paper_1703_04605_gb300 import workloads as W

pytestmark = pytest.mark.gpu

STENCILS = {"M1": (W.STENCIL_M1, 1), "G16": (W.STENCIL_G16, 2), "E5": (W.STENCIL_E5, 3), "S2": (W.STENCIL_S2, 4)}


@pytest.fixture(scope="module", autouse=True)
def _built():
    from paper_1703_04605_gb300 import build
    build.build()


@pytest.mark.parametrize("name", sorted(STENCILS))
@pytest.mark.parametrize("extra", [(0, 0, 0), (0, 1, 5), (3, 0, 1), (-1, 0, 2)])
def test_against_f64(name, extra):
    from paper_1703_04605_gb300 import Lattice3D
    st, kernel = STENCILS[name]
    with Lattice3D(st["groups"], st["m"], 0.9, 1, 1, 1, dtype="f32", v0=st["v0"]) as lat:
        halo = lat.info()["halo"]
    shape = tuple(halo + d for d in extra)
    rng = np.random.default_rng(sum(shape))
    f = {k: 0.05 * rng.uniform(-1, 1, shape) for k in ("n", "ux", "uy", "uz", "T")}
    f["n"] += 1.0
    f["T"] += 1.0
    got = {}
    for dtype in ("f32", "f64"):
        with Lattice3D(st["groups"], st["m"], 0.9, shape[2], shape[1], shape[0], dtype=dtype, v0=st["v0"]) as lat:
            if dtype == "f32":
                assert lat.info()["kernel"] == (kernel if min(extra) >= 0 else 0)
            lat.init(f["n"], f["ux"], f["uy"], f["uz"], f["T"])
            lat.step(4)
            got[dtype] = lat.moments()
    umax = max(np.max(np.abs(got["f64"][k])) for k in ("ux", "uy", "uz"))
    for k in ("n", "T", "e"):
        assert np.max(np.abs(got["f32"][k] / got["f64"][k] - 1)) < 1e-5, k
    for k in ("ux", "uy", "uz"):
        assert np.max(np.abs(got["f32"][k] - got["f64"][k])) / umax < 1e-5, k
