"""A checkpoint may lie at any address, inside a packed buffer of bytes for instance."""
import ctypes as C

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


@pytest.mark.parametrize("offset", [1, 2, 3, 4, 7, 8, 12])
@pytest.mark.parametrize("storage,pattern", [("f64", "ab"), ("f32", "ab"), ("f16", "ab"), ("f16s", "ab"), ("f32", "aa")])
def test_save_and_restore_at_any_address(lbm, storage, pattern, offset):
    w = I.jet_workload(nx=133, nr=11)
    a, b = (lbm.Lattice.from_workload(w, storage, device="cuda:0", pattern=pattern) for _ in range(2))
    a.step(3)
    want = a.save()[0].flatten().view(torch.uint8)
    n = want.numel()
    box = torch.full((n + 32,), 0xA5, dtype=torch.uint8, device="cuda:0")
    at, stream = C.c_void_p(box.data_ptr() + offset), C.c_void_p(int(torch.cuda.current_stream().cuda_stream))
    assert lbm.lib().lbm_save(a.handle, at, stream) == 0
    assert torch.equal(box[offset:offset + n], want)
    assert bool((box[:offset] == 0xA5).all()) and bool((box[offset + n:] == 0xA5).all())
    assert lbm.lib().lbm_restore(b.handle, at, C.c_int64(3), stream) == 0
    assert torch.equal(a.fields(), b.fields())
