"""Lattices on several streams and threads: few run on the chip, many leave it to the step kernel, with the same bits."""
import threading

import pytest

from paper_1002_3028_gb300 import inputs as I

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def lbm():
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_1002_3028_gb300 import lbm as L

    L.lib()
    return L


def make(lbm, storage, size, k):
    return [lbm.Lattice.from_workload(I.jet_workload(nx=size[0], nr=size[1]), storage, device="cuda:0") for _ in range(k)]


def reference(lbm, storage, size, n):
    lat = make(lbm, storage, size, 1)[0]
    lat.set_item_group(1)  # the step kernel
    lat.step(n)
    assert lat.resident()["steps"] == 0
    return lat.save()[0]


# (how many lattices, whether each call runs on the chip)
@pytest.mark.parametrize("storage,size,k,all_resident", [
    ("f32", (200, 96), 3, True), ("f32", (200, 96), 7, False), ("f16", (400, 100), 6, False),
    ("f32", (150, 70), 6, True),      # two fit together
    ("f32", (400, 120), 6, True),     # above 42 000 nodes
    ("f16s", (200, 96), 6, True),     # moment-split storage
    ("f64", (200, 96), 1, True), ("f64", (200, 96), 3, False)], ids=lambda v: str(v).replace(" ", ""))
def test_many_streams(lbm, storage, size, k, all_resident):
    want = reference(lbm, storage, size, 9015)
    lats = make(lbm, storage, size, k)
    streams = [torch.cuda.Stream() for _ in lats]
    torch.cuda.synchronize()
    for n in (8000, 7, 1000, 8):  # the first calls keep the GPU busy (24 ms each) while the others are queued
        for lat, s in zip(lats, streams):
            lat.step(n, stream=s)
    torch.cuda.synchronize()
    steps = [lat.resident()["steps"] for lat in lats]
    for lat in lats:
        assert lat.check() == 0 and torch.equal(lat.save()[0], want)
    if all_resident:
        assert steps == [9015] * k
    else:
        assert 8000 <= sum(steps) <= (1 if storage == "f64" else 3) * 9015


def test_one_after_the_other_stays_on_the_chip(lbm):
    """Lattices whose work is done, and the calls of one stream, count for nothing."""
    lats = make(lbm, "f32", (200, 96), 6)
    for lat in lats[:5]:
        lat.step(500)
    lats[5].step(500, stream=torch.cuda.Stream())  # beside one other stream
    torch.cuda.synchronize()
    assert [lat.resident()["steps"] for lat in lats] == [500] * 6
    for lat in lats:
        lat.step(50, stream=torch.cuda.Stream())
        torch.cuda.synchronize()
    assert [lat.resident()["steps"] for lat in lats] == [550] * 6


def test_threads_that_create_step_and_close(lbm):
    want, errors = reference(lbm, "f32", (200, 96), 400), []

    def work():
        try:
            stream = torch.cuda.Stream()
            with torch.cuda.stream(stream):
                for _ in range(15):
                    lat = make(lbm, "f32", (200, 96), 1)[0]
                    for n in (300, 2, 98):
                        lat.step(n)
                    got = lat.save()[0]
                    stream.synchronize()
                    if not torch.equal(got, want):
                        errors.append("bits")
                    lat.step(200)
                    lat.close()
            stream.synchronize()
        except Exception as e:
            errors.append(repr(e))

    threads = [threading.Thread(target=work) for _ in range(6)]
    for t in threads:
        t.start()
    for t in threads:
        t.join()
    assert not errors, errors[:3]
