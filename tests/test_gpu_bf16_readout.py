"""BF16-deviation read-out: populations are decoded without loss where their terms
span many bits.  With u_y around 2^-43 and u_x around 2^-21, the coefficient that
carries u_y is 2^-43 of a population, and one that carries u_x takes up the bits
between.  Doubling u_y doubles that coefficient and leaves every other stored
number as it is, so the velocity read out doubles too, to the FP64 rounding of
numbers of its own size; 2^-20 leaves room for the solve's relative error."""
import numpy as np
import pytest

from paper_1703_04605_gb300 import workloads as W

pytestmark = pytest.mark.gpu

STENCILS = {"M1": W.STENCIL_M1, "G16": W.STENCIL_G16, "E5": W.STENCIL_E5, "S2": W.STENCIL_S2}


@pytest.fixture(scope="module", autouse=True)
def _built():
    from paper_1703_04605_gb300 import build
    build.build()


@pytest.mark.parametrize("name", sorted(STENCILS))
def test_small_velocity(name):
    import torch
    from paper_1703_04605_gb300 import Lattice
    st, shape = STENCILS[name], (24, 40)
    rng = np.random.default_rng(6)
    f = dict(n=rng.uniform(0.8, 1.2, shape), ux=2.0 ** rng.uniform(-22, -20, shape),
             uy=2.0 ** rng.uniform(-43, -42, shape), T=rng.uniform(0.9, 1.1, shape))
    got = []
    with Lattice(st["groups"], st["m"], 0.9, shape[1], shape[0], dtype="bf16dev", v0=st["v0"]) as lat:
        for k in (1.0, 2.0):
            lat.init_device(**{q: torch.tensor(v * (k if q == "uy" else 1.0), device="cuda") for q, v in f.items()})
            got.append(lat.moments()["uy"].copy())
    assert np.max(np.abs(got[1] / (2 * got[0]) - 1)) < 2.0 ** -20
