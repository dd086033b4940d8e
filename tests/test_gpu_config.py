"""Launch configurations: what a grid or batch reports can be set again and is
what runs."""
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


# 128^3 lies above the planes a CTA slot from which fused grids take the TMEM queue
@pytest.mark.parametrize("n", [24, 128])
@pytest.mark.parametrize("variant,precision", [("SBLI_FUSED", 0), ("SBLI_FUSED", 1), ("SBLI_FUSED", 2), ("SBLI_FUSED", 3),
                                               ("SBLI_STORE_ALL", 0), ("SBLI_STORE_ALL", 1), ("SBLI_RS", 0),
                                               ("SBLI_SS", 0), ("SBLI_RA", 0), ("SBLI_SN", 0), ("SBLI_SN2", 0)])
def test_reported_config_can_be_set(S, variant, precision, n):
    g = S.Grid(n, precision, getattr(S, variant))
    cfg = g.config()
    g.set_config(*cfg)
    assert g.config() == cfg
    g.close()
