"""Diagnostics of FP64 lattices at the ends of the range: densities beyond what FP32 holds, and velocities that
overflow in the quotient by a tiny density, by both entry points against NumPy on the lattice's fields."""
import ctypes as C
import math

import numpy as np
import pytest

from paper_1002_3028_gb300 import inputs as I

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu

W9 = np.array([4 / 9] + [1 / 9] * 4 + [1 / 36] * 4).reshape(9, 1, 1)
E9 = np.array([(0, 0), (1, 0), (0, 1), (-1, 0), (0, -1), (1, 1), (-1, 1), (-1, -1), (1, -1)], dtype=float)


@pytest.fixture(scope="module")
def lbm():
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_1002_3028_gb300 import lbm as L

    L.lib()
    return L


def lattice(lbm, rho0, nx=70, nr=40):
    """Smooth flow of density rho0 (1 + a few percent), T = 1."""
    lat = lbm.Lattice(I.LatticeConfig(nx=nx, nr=nr, rho0=rho0, axisym=False), "f64", device="cuda:0")
    rng = np.random.default_rng(2)
    rho = 1 + 0.05 * rng.random((nr, nx))
    ux, ur = 0.05 * rng.standard_normal((2, nr, nx))
    eu = E9[:, 0].reshape(9, 1, 1) * ux + E9[:, 1].reshape(9, 1, 1) * ur
    f = rho0 * (W9 * rho * (1 + 3 * eu))
    return lat, f, np.full((4, nr, nx), 0.25)


def both(lbm, lat):
    stream = C.c_void_p(int(torch.cuda.current_stream().cuda_stream))
    for fn in (lbm.lib().lbm_diagnostics, lbm.lib().lbm_diagnostics_noalloc):
        d = lbm.Diag()
        rc = fn(lat.handle, C.byref(d), stream)
        yield rc, d.as_dict()


# each quantity rounds a few times in FP64, and the sums over 2800 nodes of one sign once per node
REL = 1e-12


@pytest.mark.parametrize("rho0", [1e-200, 1e-40, 3e-39, 1e-30, 1.0, 1e30, 1e38, 3e38, 1e39, 1e150])
def test_densities_beyond_fp32(lbm, rho0):
    lat, f, g = lattice(lbm, rho0)
    lat.set_state(f, g)
    rho, ux, ur, T = lat.fields().cpu().numpy()
    speed = np.hypot(ux, ur).max()
    assert 0.1 < speed < 1.0
    for rc, d in both(lbm, lat):
        assert rc == 0 and d["nonfinite"] == 0
        assert d["mass"] == pytest.approx(rho.sum(), rel=REL)
        assert d["max_speed"] == pytest.approx(speed, rel=REL)


@pytest.mark.parametrize("rho0", [1e-40, 1e39])
def test_residual_beyond_fp32(lbm, rho0):
    lat, f, g = lattice(lbm, rho0)
    lat.set_state(f, g)
    _, ux, ur, _ = lat.fields().cpu().numpy()
    lat.step(1)
    _, vx, vr, _ = lat.fields().cpu().numpy()
    diff = np.hypot(vx - ux, vr - ur)
    speed = np.hypot(vx, vr)
    assert np.isfinite(speed).all()
    for rc, d in both(lbm, lat):
        assert rc == 0
        assert d["residual_max"] == pytest.approx(diff.max() / speed.max(), rel=1e-10)
        assert d["residual_l2"] == pytest.approx(math.sqrt((diff ** 2).sum() / (speed ** 2).sum()), rel=1e-10)


@pytest.mark.parametrize("rho0", [1e-300, 1e-150])
def test_a_velocity_that_overflows_is_counted(lbm, rho0):
    """Momentum 2e200 at three nodes without a change of their density: above 1.8e308 over 1e-300 only."""
    lat, f, g = lattice(lbm, rho0)
    for i, j in ((10, 7), (33, 20), (60, 31)):
        f[1, j, i - 1], f[3, j, i + 1] = 1e200, -1e200
    lat.set_state(f, g)
    rho, ux, ur, T = lat.fields().cpu().numpy()
    bad = ~(np.isfinite(rho) & (rho > 0) & np.isfinite(ux) & np.isfinite(ur) & np.isfinite(T))
    assert bad.sum() == 3
    for rc, d in both(lbm, lat):
        assert d["nonfinite"] == bad.sum() and rc == -4
        assert d["mass"] == pytest.approx(rho[~bad].sum(), rel=REL)
        assert d["max_speed"] == pytest.approx(np.hypot(ux, ur)[~bad].max(), rel=REL)
