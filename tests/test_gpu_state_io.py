"""State import and export in one pass, and the marched kinetic energy and
enstrophy, at the sizes where their tiles and strides can go wrong."""
import numpy as np
import pytest

from paper_1709_09713_gb300 import workloads

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu

E0 = 1.0 / (1.4 * 0.4 * 0.01)


@pytest.fixture(scope="module")
def S():
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_1709_09713_gb300 import build

    build.build()
    from paper_1709_09713_gb300 import sbli

    sbli.lib()
    return sbli


def _state(n, seed):
    return workloads.smooth_state(n, seed, offsets=(1.0, 0.0, 0.0, 0.0, E0 + 0.5))


# an odd number of points (fields at odd multiples of 8 bytes), fewer than one block, one block and one point more
@pytest.mark.parametrize("precision", [0, 1, 2, 3])
@pytest.mark.parametrize("n", [(5, 5, 5), (32, 32, 1 + 4), (41, 5, 5), (33, 17, 9)])
def test_device_host_and_offset_buffers_agree(S, n, precision):
    q = _state(n, 7)
    P = n[0] * n[1] * n[2]
    want = None
    for kind in ("host", "device", "offset"):
        g = S.Grid(n, precision)
        if kind == "host":
            g.set_state(torch.from_numpy(q))
            out = torch.empty(g.shape, dtype=torch.float64)
            g.step_n(1, 1e-4)
            g.get_state(out)
        else:
            off = 1 if kind == "offset" else 0
            src = torch.empty(5 * P + 1, dtype=torch.float64, device="cuda")[off:off + 5 * P].view(g.shape)
            src.copy_(torch.from_numpy(q))
            g.set_state(src)
            src.fill_(float("nan"))  # on the same stream: the import has read it
            out = torch.empty(5 * P + 1, dtype=torch.float64, device="cuda")[off:off + 5 * P].view(g.shape)
            g.step_n(1, 1e-4)
            g.get_state(out)
            out = out.cpu()
        want = out if want is None else want
        assert torch.equal(out, want), kind
        g.close()


# edges of the 32 x 8 tiles, runs of one plane, more planes than SMs
@pytest.mark.parametrize("n", [(5, 5, 5), (32, 16, 8), (33, 17, 6), (31, 15, 160), (64, 24, 51), (70, 40, 12)])
def test_kinetic_energy_and_enstrophy(S, orc, n):
    q = _state(n, 11)
    ke, ens = orc.ke_enstrophy(orc.params(n), q)
    d = torch.from_numpy(q).cuda()
    out = torch.empty(2, dtype=torch.float64, device="cuda")
    S.sbli_kinetic_energy_noalloc(d.data_ptr(), *n, 1.0, out.data_ptr(), torch.cuda.current_stream().cuda_stream)
    g = S.Grid(n, 0)
    g.set_state(d)
    for a, b in (out.cpu().tolist(), g.kinetic_energy()):
        assert a == pytest.approx(ke, rel=1e-13) and b == pytest.approx(ens, rel=1e-12)
    g.close()


@pytest.mark.parametrize("n", [(5, 5, 5), (300, 3 + 2, 33), (16, 40, 32)])
def test_initial_field(S, orc, n):
    g = S.Grid(n, 0)
    g.init_tgv(0.93)
    q = g.get_state().cpu().numpy()
    w = orc.init_tgv(orc.params(n), 0.93)
    assert np.max(np.abs(q - w)) <= 1e-14 * np.max(np.abs(w))
    g.close()
