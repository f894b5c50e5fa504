"""The inboxes of a lattice kept on the chip: released without holding up other streams, and without a leak."""
import time

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


def test_closing_a_lattice_does_not_hold_up_the_default_stream(lbm):
    lat = lbm.Lattice.from_workload(I.jet_workload(nx=200, nr=96), "f32", device="cuda:0")
    side, done = torch.cuda.Stream(), torch.cuda.Event()
    lat.step(10, stream=side)
    torch.cuda.synchronize()
    lat.step(200000, stream=side)  # some 0.6 s
    lat.close()
    done.record(torch.cuda.default_stream())
    t = time.monotonic()
    while not done.query() and time.monotonic() - t < 10:
        time.sleep(1e-3)
    assert not side.query()
    side.synchronize()


def test_inboxes_are_given_back(lbm):
    def cycle(n):
        for _ in range(n):
            lat = lbm.Lattice.from_workload(I.jet_workload(nx=1000, nr=250), "f32", device="cuda:0")
            lat.step(4)
            lat.close()
        torch.cuda.synchronize()
        return torch.cuda.mem_get_info()[0]

    free = cycle(5)
    assert cycle(60) > free - 64 * 2 ** 20  # an inbox each would be 500 MB


@pytest.mark.parametrize("default_stream", [False, True])
def test_a_first_step_leaves_another_streams_capture_alone(lbm, default_stream):
    lat = lbm.Lattice.from_workload(I.jet_workload(nx=200, nr=96), "f32", device="cuda:0")
    side = torch.cuda.default_stream() if default_stream else torch.cuda.Stream()
    x = torch.zeros(8, device="cuda:0")
    torch.cuda.synchronize()
    graph = torch.cuda.CUDAGraph()
    with torch.cuda.graph(graph, capture_error_mode="global"):
        x += 1
        lat.step(5, stream=side)
        lat._L.lbm_destroy(lat._h)
        lat._h = None
    graph.replay()
    torch.cuda.synchronize()
    assert bool((x == 1).all())
