"""Read-out of a state whose steps have been captured but not replayed: what is
read follows what has run on the device.  An init writes S_0 alone, so the
read-out has to find out whether a step has overwritten the other buffer.  Bit
for bit against lattices without graphs, for every storage and order with such
an init."""
import numpy as np
import pytest

from gpu_common import smooth_fields
from paper_1703_04605_gb300 import workloads as W

pytestmark = pytest.mark.gpu

ST = {"M1": W.STENCIL_M1, "E5": W.STENCIL_E5, "O3": W.STENCIL_O3}
# stencil, storage, lattice: below and above the several-lanes kernel's limit in FP64
CASES2 = [("M1", "f64", (40, 20)), ("M1", "f64", (96, 80)), ("O3", "f64", (96, 80)), ("O3", "f32", (50, 40)),
          ("E5", "bf16dev", (50, 40)), ("M1", "f32", (50, 40))]
CASES3 = [("M1", "f64"), ("M1", "f32"), ("O3", "f64"), ("O3", "f32")]


@pytest.fixture(scope="module", autouse=True)
def _built():
    from paper_1703_04605_gb300 import build
    build.build()


def _same(a, b):
    for k in a:
        assert np.array_equal(a[k], b[k]), k


def _capture(s, call):
    import torch
    g = torch.cuda.CUDAGraph()
    with torch.cuda.graph(g, stream=s):
        call()
    return g


@pytest.mark.parametrize("name,dtype,size", CASES2)
def test_2d(name, dtype, size):
    import torch
    from paper_1703_04605_gb300 import Lattice
    st, (Nx, Ny) = ST[name], size
    dev = [{k: torch.tensor(v, device="cuda") for k, v in smooth_fields(Nx, Ny, seed=s, dn=0.05, dT=0.05, du=0.05).items()}
           for s in (1, 2)]
    s = torch.cuda.Stream()
    with torch.cuda.stream(s):
        def lattice():
            return Lattice(st["groups"], st["m"], 0.9, Nx, Ny, dtype=dtype, v0=st["v0"], stream=s.cuda_stream)
        ref = []
        for f in dev:
            with lattice() as lat:
                lat.init_device(**f)
                at0 = {k: v.copy() for k, v in lat.moments().items()}
                lat.step(2)
                ref.append((at0, lat.moments()))
        with lattice() as lat:
            lat.init_device(**dev[0])
            steps = _capture(s, lambda: lat.step(2))
            _same(ref[0][0], lat.moments())      # nothing has run yet
            steps.replay()
            _same(ref[0][1], lat.moments())
            again = _capture(s, lambda: lat.init_device(**dev[1]))
            steps = _capture(s, lambda: lat.step(2))
            again.replay()
            _same(ref[1][0], lat.moments())
            steps.replay()
            _same(ref[1][1], lat.moments())
            again.replay()
            _same(ref[1][0], lat.moments())


@pytest.mark.parametrize("name,dtype", CASES3)
def test_3d(name, dtype):
    import torch
    from paper_1703_04605_gb300 import Lattice3D
    st, shape = ST[name], (7, 8, 9)
    rng = np.random.default_rng(5)
    f = {k: 0.05 * rng.uniform(-1, 1, shape) for k in ("n", "ux", "uy", "uz", "T")}
    f["n"] += 1.0
    f["T"] += 1.0
    s = torch.cuda.Stream()
    with torch.cuda.stream(s):
        def lattice():
            return Lattice3D(st["groups"], st["m"], 0.9, 9, 8, 7, dtype=dtype, v0=st["v0"], stream=s.cuda_stream)
        with lattice() as lat:
            lat.init(**f)
            at0 = {k: v.copy() for k, v in lat.moments().items()}
            lat.step(2)
            at2 = lat.moments()
        with lattice() as lat:
            lat.init(**f)
            steps = _capture(s, lambda: lat.step(2))
            _same(at0, lat.moments())
            steps.replay()
            _same(at2, lat.moments())
