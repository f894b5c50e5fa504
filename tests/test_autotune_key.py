"""A cached tuning is applied only to the lattices and the kernels that it was timed with."""
import hashlib
import json
from types import SimpleNamespace

import pytest

from paper_1002_3028_gb300 import autotune


class FakeLattice:
    storage, pattern, nx, nr = "f32", "ab", 1024, 256

    def __init__(self, bc_in="inlet"):
        self.cfg = SimpleNamespace(bc_in=bc_in)
        self.shape = None

    def set_strip_width(self, cols):
        self.cols = cols

    def set_launch(self, band, warps):
        self.shape = (self.cols, band, warps)

    def step(self, n):
        pass


@pytest.fixture
def tuner(tmp_path, monkeypatch):
    monkeypatch.setattr(autotune, "CACHE", str(tmp_path / "autotune.json"))
    monkeypatch.setattr(autotune, "_gpu_name", lambda: "fake GPU")
    return autotune


CANDIDATES = [(64, 0, 1), (32, 1, 1)]


def timings(monkeypatch, tuner, lat, best):
    monkeypatch.setattr(tuner, "_time", lambda run, steps, warmup: 0.01 if lat.shape == best else 0.02)


def test_an_entry_of_the_old_format_is_not_applied(tuner, monkeypatch):
    digest = hashlib.sha1(repr([(1024, 256)]).encode()).hexdigest()[:12]
    with open(tuner.CACHE, "w") as fh:  # without the code: tuned for a kernel that kept no lattice on the chip
        json.dump({f"fake GPU|f32|ab|1|{digest}": {"strip": 32, "band": 1, "warps": 1}}, fh)
    lat = FakeLattice()
    timings(monkeypatch, tuner, lat, (64, 0, 1))
    assert tuner.tune(lat, candidates=CANDIDATES, steps=2, warmup=1) == (64, 0, 1) == lat.shape


def test_an_entry_of_other_kernels_is_not_applied(tuner, monkeypatch):
    lat = FakeLattice()
    timings(monkeypatch, tuner, lat, (32, 1, 1))
    assert tuner.tune(lat, candidates=CANDIDATES, steps=2, warmup=1) == (32, 1, 1)
    monkeypatch.setattr(tuner, "_code", lambda: "other")
    timings(monkeypatch, tuner, lat, (64, 0, 1))
    assert tuner.tune(lat, candidates=CANDIDATES, steps=2, warmup=1) == (64, 0, 1)
    assert len(json.load(open(tuner.CACHE))) == 2


def test_periodic_ends_have_their_own_entry(tuner, monkeypatch):
    lat, wrap = FakeLattice(), FakeLattice("periodic")
    timings(monkeypatch, tuner, lat, (64, 0, 1))
    assert tuner.tune(lat, candidates=CANDIDATES, steps=2, warmup=1) == (64, 0, 1)
    timings(monkeypatch, tuner, wrap, (32, 1, 1))
    assert tuner.tune(wrap, candidates=CANDIDATES, steps=2, warmup=1) == (32, 1, 1)
    monkeypatch.setattr(tuner, "_time", lambda *a: pytest.fail("timed a cached shape"))
    assert tuner.tune(FakeLattice(), candidates=CANDIDATES) == (64, 0, 1)
    assert tuner.tune(FakeLattice("periodic"), candidates=CANDIDATES) == (32, 1, 1)
    assert tuner.lattice_key("f32", [(1024, 256)]) != tuner.lattice_key("f32", [(1024, 256, True)])
