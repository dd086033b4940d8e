"""Device buffers that end before the state does are refused, by every call that
takes one, and the handle works on."""
import ctypes

import pytest

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu

N = (64, 32, 20)
BYTES = 5 * 64 * 32 * 20 * 8


@pytest.fixture(scope="module")
def S():
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_1709_09713_gb300 import build

    build.build()
    from paper_1709_09713_gb300 import sbli

    sbli.lib()
    return sbli


@pytest.fixture(scope="module")
def allocate(S):
    """Memory of its own allocation (torch's pools put many tensors in one)."""
    cuda = ctypes.CDLL("libcuda.so.1")
    torch.zeros(1, device="cuda")
    made = []

    def alloc(n):
        p = ctypes.c_void_p()
        assert cuda.cuMemAlloc_v2(ctypes.byref(p), ctypes.c_size_t(n)) == 0
        made.append(p)
        return p.value

    yield alloc
    torch.cuda.synchronize()
    for p in made:
        cuda.cuMemFree_v2(p)


def _refused(call):
    with pytest.raises(Exception, match="cudaMemcpyAsync|copy result"):
        call()


@pytest.mark.parametrize("precision", [0, 1, 2, 3])
def test_short_buffers_are_refused(S, allocate, precision):
    full, short = allocate(BYTES), allocate(BYTES - 8192)
    g = S.Grid(N, precision)
    b = S.Batch([N, (16, 16, 16)], precision)
    g.init_tgv(0.9)
    b.init_tgv([0.9, 0.9])
    want = g.get_state().clone()
    S.sbli_get_state(g.handle, full, False)
    for p in (short, full + 8):  # an allocation too small; one entered too late
        _refused(lambda: S.sbli_set_state(g.handle, p, False))
        _refused(lambda: S.sbli_get_state(g.handle, p, False))
        _refused(lambda: S.sbli_batch_set_state(b.handle, 0, p, False))
        _refused(lambda: S.sbli_batch_get_state(b.handle, 0, p, False))
    S.sbli_set_state(g.handle, full, False)
    S.sbli_batch_set_state(b.handle, 0, full, False)
    assert torch.allclose(g.get_state(), want, rtol=1e-6, atol=1e-9)
    assert torch.equal(b.get_state(0), g.get_state())
    g.close()
    b.close()
    srv = S.Server(64 << 20)
    r = S.request(N, precision, 1, 1e-4)
    r.result, r.result_is_host = ctypes.c_void_p(short), 0
    srv.submit(r)

    def serve():
        for _ in range(50):
            srv.tick()

    _refused(serve)
    srv.close()
