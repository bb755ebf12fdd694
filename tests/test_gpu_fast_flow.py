"""FP64 site solve in fast flows, where the Landau frame is ill conditioned: the
velocity of a read-out against the frame of its own moments T^ab, solved in
extended precision.  Tolerance 1e-15 gamma^2: rounding of the residual's six
products (6 2^-53 T^00; eight in 3D) through the inverse Jacobian (T^00 <= (e + P) gamma^2),
and of the velocity itself."""
import numpy as np
import pytest

from paper_1703_04605_gb300 import _abi as A
from paper_1703_04605_gb300 import workloads as W

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module", autouse=True)
def _built():
    from paper_1703_04605_gb300 import build
    build.build()


def _frame(T00, T0, S, v):
    """Newton iterations of T0_i - S_ij v_j - (T00 - T0.v) v_i = 0 from v, in long double."""
    d = len(v)
    v = [x.astype(np.longdouble) for x in v]
    for _ in range(6):
        e = T00 - sum(T0[a] * v[a] for a in range(d))
        F = [T0[a] - sum(S[a][b] * v[b] for b in range(d)) - e * v[a] for a in range(d)]
        # the Jacobian may be rounded: the iteration ends where F does
        J = np.empty(v[0].shape + (d, d))
        for a in range(d):
            for b in range(d):
                J[..., a, b] = (-S[a][b] - (e if a == b else 0) + v[a] * T0[b]).astype(float)
        dv = np.linalg.solve(J, np.stack([f.astype(float) for f in F], -1)[..., None])[..., 0]
        v = [v[a] - dv[..., a] for a in range(d)]
    return v


@pytest.mark.parametrize("name", ["M1", "O3"])
def test_frame_2d(name):
    import torch
    from paper_1703_04605_gb300 import Lattice
    st = {"M1": W.STENCIL_M1, "O3": W.STENCIL_O3}[name]
    Nx, Ny = 256, 200
    rng = np.random.default_rng(11)
    g, a = rng.uniform(3, 9, (Ny, Nx)), rng.uniform(0, 2 * np.pi, (Ny, Nx))
    v = np.sqrt(1 - 1 / g ** 2)
    f = dict(n=rng.uniform(0.5, 2, (Ny, Nx)), ux=v * np.cos(a), uy=v * np.sin(a), T=rng.uniform(0.3, 3, (Ny, Nx)))
    with Lattice(st["groups"], st["m"], 0.9, Nx, Ny, dtype="f64", v0=st["v0"]) as lat:
        lat.init_device(**{k: torch.tensor(x, device="cuda") for k, x in f.items()})
        m = lat.moments(A.M_UX | A.M_UY | A.M_TMN)
    t = {k: x.astype(np.longdouble) for k, x in m.items()}
    T00, T0 = t["T00"], [t["T0x"], t["T0y"]]
    S = [[t["Txx"], t["Txy"]], [t["Txy"], t["Tyy"]]]
    ref = _frame(T00, T0, S, [m["ux"], m["uy"]])
    err = sum(np.abs((m[k] - r).astype(float)) for k, r in zip(("ux", "uy"), ref))
    assert np.max(err / g ** 2) < 1e-15


@pytest.mark.parametrize("name", ["M1", "O3"])
def test_frame_3d(name):
    from paper_1703_04605_gb300 import Lattice3D
    st = {"M1": W.STENCIL_M1, "O3": W.STENCIL_O3}[name]
    shape = (32, 36, 44)
    rng = np.random.default_rng(12)
    g, d = rng.uniform(3, 9, shape), rng.normal(size=(3,) + shape)
    v = np.sqrt(1 - 1 / g ** 2) * d / np.sqrt((d * d).sum(0))
    names = ("ux", "uy", "uz")
    with Lattice3D(st["groups"], st["m"], 0.9, shape[2], shape[1], shape[0], dtype="f64", v0=st["v0"]) as lat:
        lat.init(n=rng.uniform(0.5, 2, shape), T=rng.uniform(0.3, 3, shape), **dict(zip(names, v)))
        m = lat.moments(A.M_UX | A.M_UY | A.M_UZ | A.M_TMN)
    t = {k: x.astype(np.longdouble) for k, x in m.items()}
    S = [[t["T" + "".join(sorted(a + b))] for b in "xyz"] for a in "xyz"]
    ref = _frame(t["T00"], [t["T0" + a] for a in "xyz"], S, [m[k] for k in names])
    err = sum(np.abs((m[k] - r).astype(float)) for k, r in zip(names, ref))
    assert np.max(err / g ** 2) < 1e-15
