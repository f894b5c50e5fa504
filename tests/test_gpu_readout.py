"""Reading a state out: FP64 populations formed in integer arithmetic (csrc/lbm_readout.cuh) have
the bits of the FP64 sum, and checkpoints copied in wide or narrow words hold the same values."""
import numpy as np
import pytest

from paper_1002_3028_gb300 import inputs as I

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu

W9 = [4 / 9] + [1 / 9] * 4 + [1 / 36] * 4


@pytest.fixture(scope="module")
def lbm():
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_1002_3028_gb300 import lbm as L

    L.lib()
    return L


def deviations(shape, seed):
    """Deviations of every size and sign: around the constants' binade edges, up to several times
    the constants, down to far below their last place, and exact zeros."""
    rng = np.random.default_rng(seed)
    mag = np.exp(rng.uniform(np.log(1e-25), np.log(8.0), shape))
    v = mag * rng.choice([-1.0, 1.0], shape)
    v[rng.random(shape) < 0.05] = 0.0
    near = rng.random(shape) < 0.2
    edges = np.array([0.5, 0.25, 0.125, 0.0625, 0.03125, 0.015625])
    c = np.array(W9 + [0.25] * 4).reshape(13, 1, 1)
    v = np.where(near, rng.choice(edges, shape) - c + 1e-7 * rng.standard_normal(shape), v)
    return v


@pytest.mark.parametrize("rho0,T0", [(1.0, 1.0), (1.0, 0.7), (1.3, 1.0)])
@pytest.mark.parametrize("storage,pattern", [("f32", "ab"), ("f16", "ab"), ("bf16", "ab"), ("f32", "aa"), ("f16s", "ab")])
@pytest.mark.parametrize("size", [(300, 41), (33, 3)], ids=lambda s: f"{s[0]}x{s[1]}")
def test_fp64_populations_are_the_fp64_sums(lbm, size, storage, pattern, rho0, T0):
    nx, nr = size
    cfg = I.LatticeConfig(nx=nx, nr=nr, rho0=rho0, T0=T0)
    lat = lbm.Lattice(cfg, storage, device="cuda:0", pattern=pattern)
    c = np.array([w * rho0 for w in W9] + [0.25 * T0] * 4).reshape(13, 1, 1)
    a = c + deviations((13, nr, nx), 5)
    lat.set_state(a[:9], a[9:])
    f, g = lat.get_state()
    got = torch.cat([f, g]).cpu().numpy()
    planes = lat.save()[0]
    if storage == "f16s":  # the stored values are not deviations from rest: one FP32 rounding from them
        assert np.all(np.abs(got - a) <= 2e-3 * np.abs(a - c) + 2e-2)
        assert np.array_equal(got, (got - c).astype(np.float32).astype(np.float64) + c) or rho0 != 1.0
        return
    want = planes.cpu().double().numpy() + c
    if rho0 == 1.0:
        assert np.array_equal(got, want)
    else:  # the product w rho0 rounds, or is fused into the sum
        assert np.allclose(got, want, rtol=0, atol=4e-16 * 8)


@pytest.mark.parametrize("storage", ["f64", "f32", "f16", "f16s"])
@pytest.mark.parametrize("nx", [1, 7, 64, 130, 301, 520])
@pytest.mark.parametrize("pattern,steps", [("ab", 3), ("aa", 2), ("aa", 3)])
def test_checkpoints_of_every_row_alignment(lbm, nx, storage, pattern, steps):
    if storage == "f16s" and pattern == "aa":
        pytest.skip("moment-split storage has no AA pattern")
    w = I.jet_workload(nx=nx, nr=11)
    a, b = (lbm.Lattice.from_workload(w, storage, device="cuda:0", pattern=pattern) for _ in range(2))
    a.step(steps)
    planes, step = a.save()
    b.restore(planes, step)
    assert torch.equal(a.fields(), b.fields())
    a.step(2)
    b.step(2)
    assert torch.equal(a.save()[0], b.save()[0])


@pytest.mark.parametrize("storage,pattern,steps", [("f64", "ab", 1), ("f32", "ab", 1), ("bf16", "ab", 1), ("f16s", "ab", 1),
                                                   ("f32", "aa", 1), ("f16", "aa", 2)])
@pytest.mark.parametrize("size", [(3, 3), (33, 9), (64, 8), (65, 17), (258, 40)], ids=lambda s: f"{s[0]}x{s[1]}")
def test_fields_are_the_moments_of_the_streamed_populations(lbm, size, storage, pattern, steps):
    """Inside the lattice, where every population comes from a node of the state."""
    nx, nr = size
    lat = lbm.Lattice.from_workload(I.jet_workload(nx=nx, nr=nr), storage, device="cuda:0", pattern=pattern)
    lat.step(steps)
    f, g = lat.get_state()
    e9 = [(0, 0), (1, 0), (0, 1), (-1, 0), (0, -1), (1, 1), (-1, 1), (-1, -1), (1, -1)]
    pull = lambda p, e: torch.roll(p, (e[1], e[0]), (0, 1))
    f, g = [pull(p, e) for p, e in zip(f, e9)], [pull(p, e) for p, e in zip(g, e9[1:5])]
    rho = sum(f)
    want = torch.stack([rho, sum(p * e[0] for p, e in zip(f, e9)) / rho, sum(p * e[1] for p, e in zip(f, e9)) / rho, sum(g)])
    inside = (slice(None), slice(1, -1), slice(1, -1))
    eps = 2.0 ** -53 if storage == "f64" else 2.0 ** -24
    scale = max(1.0, float(want.abs().max()))
    for dtype in (torch.float64, torch.float32):
        got = lat.fields(dtype=dtype).double()
        # 13 terms of at most the largest value, each sum rounded once, and the quotient's
        assert (got - want)[inside].abs().max() <= 16 * (eps if dtype == torch.float64 else max(eps, 2.0 ** -24)) * scale
