"""lbm_step refuses a stream that is being captured, takes no step, and goes on afterwards."""
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


@pytest.mark.parametrize("nx,nr", [(200, 96), (2048, 256)])
@pytest.mark.parametrize("before", [0, 5])
def test_a_captured_step_is_refused(lbm, nx, nr, before):
    a, b = (lbm.Lattice.from_workload(I.jet_workload(nx=nx, nr=nr), "f32", device="cuda:0") for _ in range(2))
    side = torch.cuda.Stream()
    a.step(before, stream=side)
    torch.cuda.synchronize()
    graph = torch.cuda.CUDAGraph()
    with torch.cuda.stream(side):
        graph.capture_begin()
        with pytest.raises(lbm.LbmError) as e:
            a.step(5)
        assert e.value.code == -3
        with pytest.raises(RuntimeError):
            graph.capture_end()
    torch.cuda.synchronize()
    assert a.step_count == before
    a.step(4, stream=side)
    a.step(3, stream=side)
    torch.cuda.synchronize()
    b.step(before + 7)
    assert a.check() == 0 and torch.equal(a.save()[0], b.save()[0])
