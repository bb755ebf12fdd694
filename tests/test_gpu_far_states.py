"""FP64 site solve outside the range of its FP32-seeded path (T^00 beyond 2^+-465,
on 3D lattices 2^+-310), where the all-FP64 iterations take over: densities scaled by
a power of two, which scales every number of a run exactly, against the oracle at
density 1.  Above and below the several-lanes kernel's limit, both orders.
Tolerance: the FP64 path's 1e-12."""
import numpy as np
import pytest

from gpu_common import errors, oracle_lattice, run_gpu, run_oracle, smooth_fields
from paper_1703_04605_gb300 import workloads as W

pytestmark = pytest.mark.gpu

ST = {"M1": W.STENCIL_M1, "E5": W.STENCIL_E5, "O3": W.STENCIL_O3}


@pytest.fixture(scope="module", autouse=True)
def _built():
    from paper_1703_04605_gb300 import build
    build.build()


@pytest.mark.parametrize("name,shape", [("M1", (24, 20)), ("M1", (96, 77)), ("E5", (96, 77)), ("O3", (24, 20)),
                                        ("O3", (96, 77))])
def test_2d(name, shape):
    f = smooth_fields(shape[0], shape[1], seed=8, dn=0.05, dT=0.05, du=0.05)
    ref = run_oracle(ST[name], 1.2, f, 2)
    for scale in (2.0 ** -482, 2.0 ** 482):
        got, _ = run_gpu(ST[name], 1.2, dict(f, n=f["n"] * scale), "f64", 2)
        got["n"] = got["n"] / scale
        e = errors(got, ref)
        assert max(e.values()) < 1e-12, (scale, e)


@pytest.mark.parametrize("name", ["M1", "O3"])
def test_3d(name):
    from oracle import lattice as OL
    from paper_1703_04605_gb300 import Lattice3D
    st, shape = ST[name], (5, 6, 7)
    rng = np.random.default_rng(3)
    f = {k: 0.05 * rng.uniform(-1, 1, shape) for k in ("n", "ux", "uy", "uz", "T")}
    f["n"] += 1.0
    f["T"] += 1.0
    o = OL.Lattice(oracle_lattice(st, 0.9, shape[1:]).st, 0.9, shape, two_d=False)
    o.init(f["n"], f["ux"], f["uy"], f["T"], f["uz"])
    o.step(2)
    ref = o.macros()
    umax = max(np.max(np.abs(ref[k])) for k in ("ux", "uy", "uz"))
    for scale in (2.0 ** -320, 2.0 ** 320):
        with Lattice3D(st["groups"], st["m"], 0.9, 7, 6, 5, dtype="f64", v0=st["v0"]) as lat:
            lat.init(f["n"] * scale, f["ux"], f["uy"], f["uz"], f["T"])
            lat.step(2)
            got = lat.moments()
        assert np.max(np.abs(got["n"] / scale / ref["n"] - 1)) < 1e-12
        assert np.max(np.abs(got["T"] / ref["T"] - 1)) < 1e-12
        for k in ("ux", "uy", "uz"):
            assert np.max(np.abs(got[k] - ref[k])) / umax < 1e-12, k
