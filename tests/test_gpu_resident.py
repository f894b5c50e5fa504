"""Lattices kept on the chip (csrc/lbm_resident.cuh): a launch of many steps gives the bits of
one-step launches, which the step kernel runs, at the edges of tiles and of the plan."""
import pytest

from paper_1002_3028_gb300 import inputs as I

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu

BOUNDARIES = {
    "jet": dict(),
    "pipe": dict(bc_top="wall"),
    "substrate": dict(bc_out="wall"),
    "inner_wall": dict(bc_top="wall", bc_bottom="wall", r0=3.0, bc_out="wall"),
}


@pytest.fixture(scope="module")
def lbm():
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_1002_3028_gb300 import lbm as L

    L.lib()
    return L


def pair(lbm, nx, nr, storage, bounds, seed=3):
    cfg = I.LatticeConfig(nx=nx, nr=nr, T_top=1.2, T_bottom=1.5, T_out=0.8, noise_amp=1e-3, seed=seed,
                          **BOUNDARIES[bounds])
    u_in, T_in = I.jet_profiles(nr, max(1.0, nr / 3.0), 0.06, 1.0, 4.0)
    nu, al = I.power_law_tables(64, 0.8, 4.0, nu_max=0.2)
    w = I.Workload("tiles", cfg, u_in, T_in, nu, al, 0.8, 4.0)
    w9 = [4 / 9] + [1 / 9] * 4 + [1 / 36] * 4
    f, g = I.random_state(nx, nr, w9, [0.3] * 4, 0.04, seed)
    lats = [lbm.Lattice.from_workload(w, storage) for _ in range(2)]
    for lat in lats:
        lat.set_state(f, g, 5)
    return lats


def same(a, b):
    assert a.check() == 0 and b.check() == 0
    assert a.step_count == b.step_count
    assert torch.equal(a.save()[0], b.save()[0]) and torch.equal(a.fields(), b.fields())
    da, db = a.diagnostics(), b.diagnostics()  # the residual reads the state one step earlier too
    assert da["residual_l2"] == db["residual_l2"] and da["mass"] == db["mass"]


@pytest.mark.parametrize("storage", ["f64", "f32", "f16", "bf16", "f16s", "bf16s"])
@pytest.mark.parametrize("bounds", sorted(BOUNDARIES))
@pytest.mark.parametrize("size", [(1, 1), (1, 40), (130, 1), (64, 8), (65, 9), (33, 2), (258, 33)],
                         ids=lambda s: f"{s[0]}x{s[1]}")
def test_many_steps_on_the_chip_equal_single_steps(lbm, size, bounds, storage):
    one, many = pair(lbm, *size, storage, bounds)
    for n in (2, 3, 12):  # odd and even counts, counters carried from launch to launch
        for _ in range(n):
            one.step(1)
        many.step(n)
        same(one, many)


@pytest.mark.parametrize("storage,size", [
    ("f32", (640, 160)), ("f32", (1216, 255)), ("f32", (1217, 257)), ("f16s", (777, 301)), ("f16s", (1216, 256)),
    ("bf16", (4096, 64)), ("f16", (70, 1000)), ("f64", (320, 90)), ("f64", (512, 128)), ("f64", (700, 200)),
])
def test_the_largest_tiles_and_the_first_lattices_beyond_them(lbm, storage, size):
    one, many = pair(lbm, *size, storage, "jet")
    for _ in range(9):
        one.step(1)
    many.step(9)
    same(one, many)


@pytest.mark.parametrize("storage", ["f16s", "bf16s"])
@pytest.mark.parametrize("bounds", ["jet", "substrate", "pipe"])
def test_smooth_flows_of_the_moment_split_types_equal_single_steps(lbm, bounds, storage):
    """Where the deviations are small, one FP32 rounding of a ghost cell's linear part shows: a
    hot smooth flow, quiet at the axis, over many nodes and steps."""
    nx, nr = 2000, 48
    x, r = torch.arange(nx).double()[None] / nx, (torch.arange(nr).double()[:, None] + 0.5) / nr
    for seed in range(6):
        one, many = pair(lbm, nx, nr, storage, bounds, seed)
        gen = torch.Generator().manual_seed(seed)
        a = torch.rand(4, generator=gen).double()
        ux = 0.03 + 0.02 * torch.sin(5 * x + 6 * a[0]) * torch.cos(3 * r)
        ur = 0.01 * r * torch.cos(7 * x + 6 * a[1]) * (1 - r)
        T = 1 + (5 + 5 * a[2]) * (1 - 0.6 * x) * torch.exp(-3 * r * r)
        w9 = [4 / 9] + [1 / 9] * 4 + [1 / 36] * 4
        e9 = [(0, 0), (1, 0), (0, 1), (-1, 0), (0, -1), (1, 1), (-1, 1), (-1, -1), (1, -1)]
        f = torch.stack([w * (1 + 3 * (ux * c + ur * d) + 4.5 * (ux * c + ur * d) ** 2 - 1.5 * (ux ** 2 + ur ** 2))
                         for w, (c, d) in zip(w9, e9)])
        g = torch.stack([0.25 * T * (1 + 2 * (ux * c + ur * d)) for c, d in e9[1:5]])
        g = g * (1 + 4e-4 * (torch.rand(g.shape, generator=gen).double() - 0.5))
        one.set_state(f.cuda(), g.cuda(), 0)
        many.set_state(f.cuda(), g.cuda(), 0)
        for _ in range(120):
            one.step(1)
        many.step(120)
        same(one, many)


def test_lattices_on_two_streams(lbm):
    lats = [pair(lbm, 500, 120, "f32", "jet", seed=7 + k) for k in range(4)]
    streams = [torch.cuda.Stream() for _ in lats]
    for _ in range(5):
        for (_, many), s in zip(lats, streams):
            many.step(20, stream=s)
    torch.cuda.synchronize()
    for one, many in lats:
        for _ in range(100):
            one.step(1)
        same(one, many)


def test_the_resident_waits_are_bounded(lbm):
    one, many = pair(lbm, 200, 96, "f32", "jet")
    many.step(5)
    assert many.selftest_wait_timeout() == 1  # LBM_STATUS_TIMEOUT from either kernel's waits
    many.step(5)
    for _ in range(10):
        one.step(1)
    same(one, many)
