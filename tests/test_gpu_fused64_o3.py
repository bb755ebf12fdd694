"""Compiled FP64 third-order kernels against the oracle at the edges of their
forms: lattices smaller than a halo, small lattices on several lanes a site (up
to 4864 sites on 152 SMs), blocks with a tail.  Tolerance: the FP64
path's 1e-12."""
import pytest

from gpu_common import errors, run_gpu, run_oracle, smooth_fields
from paper_1703_04605_gb300 import stencils as S
from paper_1703_04605_gb300 import workloads as W

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module", autouse=True)
def _built():
    from paper_1703_04605_gb300 import build
    build.build()


@pytest.mark.parametrize("shape", [(1, 1), (2, 4), (9, 1), (33, 5), (96, 76), (96, 77)])
def test_shapes(shape):
    f = smooth_fields(shape[0], shape[1], seed=shape[0] + shape[1], dn=0.05, dT=0.05, du=0.08)
    got, _ = run_gpu(W.STENCIL_O3, 0.9, f, "f64", 2)
    e = errors(got, run_oracle(W.STENCIL_O3, 0.9, f, 2))
    assert max(e.values()) < 1e-12, e


@pytest.mark.parametrize("m", [2.0, 3.0, 4.0, 5.5, 8.0])
@pytest.mark.parametrize("shape", [(11, 9), (96, 77)])
def test_library_sets(m, shape):
    groups, mu = S.choose(m, order=3)
    from paper_1703_04605_gb300 import quadrature_window
    lo, hi, _ = quadrature_window(groups, mu)
    st = dict(groups=groups, m=mu, v0=0.5 * (lo + hi))
    f = smooth_fields(shape[0], shape[1], seed=5, dn=0.03, dT=0.03, du=0.05)
    got, _ = run_gpu(st, 1.1, f, "f64", 2)
    e = errors(got, run_oracle(st, 1.1, f, 2))
    assert max(e.values()) < 1e-12, e
