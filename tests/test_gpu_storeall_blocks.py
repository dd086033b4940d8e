"""The store-all derivative launches (blocks of 32 x 8 columns, nine planes of one
array or three of a set of arrays) where a block's columns and planes end."""
import numpy as np
import pytest

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def S():
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_1709_09713_gb300 import build

    build.build()
    from paper_1709_09713_gb300 import sbli

    sbli.lib()
    return sbli


@pytest.mark.parametrize("n", [(5, 5, 5), (32, 8, 9), (33, 9, 10), (31, 7, 8), (64, 5, 19)])
@pytest.mark.parametrize("variant", ["SBLI_STORE_ALL", "SBLI_RS", "SBLI_SS"])
def test_residual_equals_fused(S, n, variant):
    """Store-all and stored-gradient residuals of a rough state against the fused
    kernel's.  The largest term is H0 div u with H0 = 1 / ((gamma - 1) M^2) = 250 and,
    for velocities within 1.2, first derivatives within 18 x 1.2 / (12 h) each; some 64
    roundings of terms of that size on either side."""
    rng = np.random.default_rng(sum(n))
    q = rng.uniform(-0.1, 0.1, (5, n[2], n[1], n[0]))
    out = []
    for v in (S.SBLI_FUSED, getattr(S, variant)):
        g = S.Grid(n, S.SBLI_FP64, v)
        g.init_tgv()
        g.set_state(g.get_state() + torch.as_tensor(q, device="cuda").reshape(g.get_state().shape))
        out.append(g.rhs().clone().double().cpu().numpy())
        g.close()
    h = 2 * np.pi / max(n)
    assert np.abs(out[0] - out[1]).max() <= 2 * 64 * 2.0**-53 * 250 * 3 * 18 * 1.2 / (12 * h)
