"""Which lattices run on the chip, in which tiles, and that their steps ran there: the comparisons of the two paths
compare two paths."""
import ctypes as C
import subprocess

import pytest

from paper_1002_3028_gb300 import build as B
from paper_1002_3028_gb300 import inputs as I

torch = pytest.importorskip("torch")

BOUNDARIES = {
    "jet": dict(),
    "pipe": dict(bc_top="wall"),
    "substrate": dict(bc_out="wall"),
    "closed_axis": dict(bc_top="wall", bc_out="wall"),
    "annulus_open": dict(bc_bottom="wall", r0=3.0),
    "annulus_pipe": dict(bc_bottom="wall", r0=3.0, bc_top="wall"),
    "annulus_substrate": dict(bc_bottom="wall", r0=3.0, bc_out="wall"),
    "annulus_closed": dict(bc_bottom="wall", r0=3.0, bc_top="wall", bc_out="wall"),
}


@pytest.fixture(scope="module")
def lbm():
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_1002_3028_gb300 import lbm as L

    L.lib()
    return L


def pair(lbm, nx, nr, storage, bounds="jet", seed=3, ntab=64, **cfg):
    c = I.LatticeConfig(nx=nx, nr=nr, T_top=1.2, T_bottom=1.5, T_out=0.8, noise_amp=1e-3, seed=seed,
                        **{**BOUNDARIES[bounds], **cfg})
    u_in, T_in = I.jet_profiles(nr, max(1.0, nr / 3.0), 0.06, 1.0, 4.0)
    nu, al = I.power_law_tables(ntab, 0.8, 4.0, nu_max=0.2) if ntab > 1 else I.constant_tables(0.1, 0.15)
    w = I.Workload("tiles", c, u_in, T_in, nu, al, 0.8, 4.0)
    f, g = I.random_state(nx, nr, [4 / 9] + [1 / 9] * 4 + [1 / 36] * 4, [0.3] * 4, 0.04, seed)
    lats = [lbm.Lattice.from_workload(w, storage, device="cuda:0") for _ in range(2)]
    for lat in lats:
        lat.set_state(f, g, 5)
    return lats


def same(a, b):
    assert a.check() == 0 and b.check() == 0
    assert a.step_count == b.step_count
    assert torch.equal(a.save()[0], b.save()[0]) and torch.equal(a.fields(), b.fields())
    da, db = a.diagnostics(), b.diagnostics()
    assert da["residual_l2"] == db["residual_l2"] and da["mass"] == db["mass"]


def many_equal_single(one, many, counts):
    for n in counts:
        before = many.resident()["steps"]
        for _ in range(n):
            one.step(1)
        many.step(n)
        assert many.resident()["steps"] == before + n
        same(one, many)
    assert one.resident()["steps"] == 0


# a size of each tile shape (columns, rows, rows a warp) on the 152 SMs of a GB300
SHAPES = [("f32", (150, 70), (32, 8, 1)), ("f16s", (512, 128), (64, 8, 1)), ("f32", (640, 160), (64, 8, 1)),
          ("f32", (900, 140), (64, 16, 1)), ("bf16", (777, 301), (64, 16, 2)), ("f16s", (1000, 250), (64, 16, 2)),
          ("f64", (200, 60), (32, 8, 1)), ("f64", (500, 130), (32, 16, 1))]


@pytest.mark.gpu
@pytest.mark.parametrize("bounds", sorted(BOUNDARIES))
@pytest.mark.parametrize("storage,size,tile", SHAPES, ids=lambda v: str(v).replace(" ", ""))
def test_every_tile_shape_under_every_boundary_set(lbm, storage, size, tile, bounds):
    one, many = pair(lbm, *size, storage, bounds)
    r = many.resident()
    assert (r["tile_cols"], r["tile_rows"], r["rows_per_warp"]) == tile
    many_equal_single(one, many, (7, 6))
    held = many.resident()
    assert held["inbox_held"] == held["inbox_bytes"] == r["inbox_bytes"] > 0 and r["inbox_held"] == 0


@pytest.mark.gpu
@pytest.mark.parametrize("storage,size", [("f32", (150, 70)), ("f16s", (512, 128)), ("f32", (900, 140)),
                                          ("f16", (777, 301)), ("f64", (200, 60))])
@pytest.mark.parametrize("ntab,axisym", [(1, True), (256, True), (257, True), (1000, False), (64, False)])
def test_tables_and_the_planar_model(lbm, storage, size, ntab, axisym):
    one, many = pair(lbm, *size, storage, ntab=ntab, axisym=axisym)
    many_equal_single(one, many, (8, 7))


@pytest.mark.gpu
@pytest.mark.parametrize("storage,nx,nr,cfg", [
    ("f32", 1400, 400, {}), ("f16s", 2048, 256, {}), ("f64", 700, 200, {}),
    ("f32", 200, 96, dict(bc_in="periodic", bc_out="periodic"))])
def test_lattices_beyond_the_chip_take_the_step_kernel(lbm, storage, nx, nr, cfg):
    one, many = pair(lbm, nx, nr, storage, **cfg)
    many.step(8)
    r = many.resident()
    assert r["tile_cols"] == 0 and r["steps"] == 0 and r["inbox_held"] == 0
    with pytest.raises(lbm.LbmError):
        many.selftest_resident_timeout()
    aa = lbm.Lattice(I.LatticeConfig(nx=100, nr=40), "f32", device="cuda:0", pattern="aa")
    assert aa.resident()["tile_cols"] == 0


@pytest.mark.gpu
@pytest.mark.parametrize("storage", ["f32", "f64", "f16s"])
def test_launch_shapes_and_single_steps_between_launches_on_the_chip(lbm, storage):
    one, many = pair(lbm, 200, 96, storage)
    plan = many.resident()

    def go(n, on):
        before = many.resident()["steps"]
        many.step(n)
        for _ in range(n):
            one.step(1)
        assert many.resident()["steps"] - before == (n if on else 0)

    m = plan["min_steps"]
    go(m, True)
    go(1, False)
    go(m + 1, True)
    if m > 2:
        go(m - 1, False)
    many.set_launch(3)
    assert many.resident()["tile_cols"] == 0
    go(9, False)
    many.set_launch(0)
    assert {k: many.resident()[k] for k in ("tile_cols", "tiles_across", "tiles_up")} == \
        {k: plan[k] for k in ("tile_cols", "tiles_across", "tiles_up")}
    go(8, True)
    many.set_item_group(1)
    go(7, False)
    many.set_item_group(0)
    go(7, True)
    many.set_launch(0, 2)
    go(8, False)
    many.set_launch(0, 1)
    if storage != "f64":
        many.set_strip_width(32)
        go(9, False)
        many.set_strip_width(0)
    go(m, True)
    same(one, many)


@pytest.mark.gpu
def test_a_batch_member_is_not_on_the_chip(lbm):
    one, many = pair(lbm, 200, 96, "f32")
    batch = lbm.Batch("f32")
    batch.add(many)
    assert many.resident()["tile_cols"] == 0
    batch.step(9)
    batch.remove(many)
    for _ in range(9):
        one.step(1)
    many_equal_single(one, many, (5,)) if many.resident()["tile_cols"] else pytest.fail("on the chip again")


@pytest.mark.gpu
@pytest.mark.parametrize("storage,size", [("f32", (150, 70)), ("f16s", (512, 128)), ("f32", (900, 140)),
                                          ("bf16", (777, 301)), ("f64", (200, 60))])
def test_the_waits_of_the_tiles_give_up(lbm, storage, size):
    one, many = pair(lbm, *size, storage)
    assert many.selftest_resident_timeout() == 1  # LBM_STATUS_TIMEOUT, before any inbox was filled
    many_equal_single(one, many, (6,))
    assert many.selftest_resident_timeout() == 1
    assert many.selftest_wait_timeout() == 1
    many_equal_single(one, many, (7,))


def test_resident_struct_matches_header_layout(tmp_path):
    from paper_1002_3028_gb300 import lbm as L

    names = [f[0] for f in L.Resident._fields_]
    src = tmp_path / "layout.c"
    src.write_text('#include <stdio.h>\n#include <stddef.h>\n#include "lbm.h"\nint main(void){'
                   + "".join(f'printf("%zu ", offsetof(lbm_resident, {n}));' for n in names)
                   + 'printf("%zu", sizeof(lbm_resident)); return 0;}\n')
    exe = tmp_path / "layout"
    subprocess.run(["gcc", "-std=c99", "-I", B.INCLUDE, str(src), "-o", str(exe)], check=True)
    got = [int(v) for v in subprocess.run([str(exe)], capture_output=True, text=True, check=True).stdout.split()]
    assert got == [getattr(L.Resident, n).offset for n in names] + [C.sizeof(L.Resident)]
