"""The scheme has no preferred point: a state shifted along an axis has the
shifted residual, bit for bit, in every algorithm class and precision."""
import pytest

from paper_1709_09713_gb300 import workloads

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu

N = (37, 19, 23)
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


@pytest.mark.parametrize("variant,precision", [("SBLI_FUSED", 0), ("SBLI_FUSED", 1), ("SBLI_FUSED", 2), ("SBLI_FUSED", 3),
                                               ("SBLI_STORE_ALL", 0), ("SBLI_STORE_ALL", 1), ("SBLI_RS", 0),
                                               ("SBLI_SS", 0), ("SBLI_RA", 0), ("SBLI_SN", 0), ("SBLI_SN2", 0)])
def test_shifted_state_has_shifted_residual(S, variant, precision):
    q = torch.from_numpy(workloads.smooth_state(N, 41, offsets=(1.0, 0.0, 0.0, 0.0, E0 + 0.5))).cuda()
    g = S.Grid(N, precision, getattr(S, variant))
    g.set_state(q)
    want = g.rhs().clone()
    for axis in (1, 2, 3):  # x2, x1, x0
        for by in (1, 5, 10):
            g.set_state(torch.roll(q, by, axis).contiguous())
            assert torch.equal(g.rhs(), torch.roll(want, by, axis)), (axis, by)
    g.close()
