"""Compiled FP64 kernels against the FP64 oracle where they can go wrong:
lattices smaller than a halo, one warp, block-size and tile edges (the limits of
the several-lanes kernel are 608, 1216, 2432 and 4864 sites on 152 SMs), and states
far from the reference (extreme densities, cold and hot gas), where the site
solve leaves its FP32-seeded path.  Tolerance: the FP64 path's 1e-12."""
import numpy as np
import pytest

from gpu_common import errors, run_gpu, run_oracle, smooth_fields
from paper_1703_04605_gb300 import workloads as W

pytestmark = pytest.mark.gpu

STENCILS = {"M1": W.STENCIL_M1, "G16": W.STENCIL_G16, "E5": W.STENCIL_E5, "S2": W.STENCIL_S2}


@pytest.fixture(scope="module", autouse=True)
def _built():
    from paper_1703_04605_gb300 import build
    build.build()


@pytest.mark.parametrize("name", sorted(STENCILS))
@pytest.mark.parametrize("shape", [(1, 1), (2, 3), (31, 1), (33, 5), (96, 102), (160, 123)])
def test_shapes(name, shape):
    st = STENCILS[name]
    f = smooth_fields(shape[0], shape[1], seed=shape[0] + shape[1], du=0.3)
    got, _ = run_gpu(st, 0.9, f, "f64", 3)
    e = errors(got, run_oracle(st, 0.9, f, 3))
    assert max(e.values()) < 1e-12, e


@pytest.mark.parametrize("n,T", [(1e-30, 1.0), (1e30, 1.0), (1.0, 0.2), (1.0, 3.0), (1e40, 2.5)])
def test_far_states(n, T):
    st = W.STENCIL_M1
    f = smooth_fields(24, 20, seed=8, dn=0.02, dT=0.02, du=0.05)
    f["n"], f["T"] = f["n"] * n, f["T"] * T
    got, _ = run_gpu(st, 1.2, f, "f64", 2)
    e = errors(got, run_oracle(st, 1.2, f, 2))
    assert max(e.values()) < 1e-12, e


def test_density_below_the_solve_is_refused():
    # the Landau determinant of such a state underflows: ENONPHYS
    from paper_1703_04605_gb300 import RLBMError
    f = smooth_fields(24, 20, seed=8, dn=0.02, dT=0.02, du=0.05)
    f["n"] = f["n"] * 1e-200
    with pytest.raises(RLBMError):
        run_gpu(W.STENCIL_M1, 1.2, f, "f64", 2)


def test_nonphysical_state_is_reported():
    from paper_1703_04605_gb300 import Lattice, RLBMError
    import torch
    st = W.STENCIL_M1
    one = torch.ones(16, 16, dtype=torch.float64, device="cuda")
    T = one.clone()
    T[3, 4] = -0.5
    with Lattice(st["groups"], st["m"], 0.8, 16, 16, dtype="f64", v0=st["v0"]) as lat:
        lat.init_device(one, 0 * one, 0 * one, T)
        lat.step(2)
        with pytest.raises(RLBMError):
            lat.sync()


# at most and just above 608, 1216, 2432 and 4864 sites
@pytest.mark.parametrize("shape", [(19, 32), (87, 7), (64, 19), (1217, 1), (64, 38), (811, 3), (64, 76), (695, 7)])
def test_lane_counts(shape):
    st = W.STENCIL_S2
    f = smooth_fields(shape[0], shape[1], seed=shape[0], du=0.2)
    got, _ = run_gpu(st, 0.8, f, "f64", 2)
    e = errors(got, run_oracle(st, 0.8, f, 2))
    assert max(e.values()) < 1e-12, e


@pytest.mark.parametrize("shape", [(50, 16), (96, 77)])
def test_other_group_set(shape):
    # no compiled kernel: several lanes a site, and the table-driven kernel above that
    st = dict(groups=[1, 2, 3, 6, 7, 11], m=5.0, v0=0.3095)
    f = smooth_fields(shape[0], shape[1], seed=4, dn=0.05, dT=0.05, du=0.05)
    got, info = run_gpu(st, 0.9, f, "f64", 3)
    e = errors(got, run_oracle(st, 0.9, f, 3))
    assert max(e.values()) < 1e-12, e
