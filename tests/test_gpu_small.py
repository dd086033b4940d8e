"""Binary32 work decompositions picked for small grids, and default
configurations: bitwise the state of one CTA per tile, the same diagnostics."""
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


# one plane a CTA, two, three, the smallest configurable four, and more; odd row counts (row pairs with one valid row)
@pytest.mark.parametrize("precision", [1, 2])
@pytest.mark.parametrize("n", [(5, 5, 5), (31, 7, 20), (40, 9, 12), (32, 32, 32), (33, 40, 40), (64, 33, 41), (96, 70, 50)])
def test_default_agrees_with_whole_tiles(S, n, precision):
    seen = []
    for cfg in (None, (8, 4, 0, 1), (8, 4, 1, 1), (8, max(4, n[2]), 0, 1)):
        g = S.Grid(n, precision)
        if cfg:
            g.set_config(*cfg)
            assert g.config() == (cfg[0], max(4, min(cfg[1], n[2])), cfg[2], cfg[3])
        g.init_tgv(0.9)
        hist = g.step_n_history(2, 1e-3).cpu().numpy()
        g.step_n(1, 1e-3)
        seen.append((torch.stack([g.get_state(), g.rhs()]), hist))
        g.close()
    for q, h in seen[:-1]:
        assert torch.equal(q, seen[-1][0])
        assert np.allclose(h, seen[-1][1], rtol=1e-13, atol=0)


@pytest.mark.parametrize("precision", [1, 2])
@pytest.mark.parametrize("sizes", [[(5, 5, 5)], [(64, 64, 64), (33, 20, 40)], [(40, 40, 40)] * 9])
def test_small_batches_agree_with_single_grids(S, sizes, precision):
    b = S.Batch(sizes, precision)
    b.init_tgv([1.0] * len(sizes))
    assert b.schedule()[1] == [min(32, n[2]) for n in sizes]
    hist = b.step_n_history(2, 1e-3).cpu().numpy()
    for m, n in enumerate(sizes):
        g = S.Grid(n, precision)
        g.init_tgv(1.0)
        alone = g.step_n_history(2, 1e-3).cpu().numpy()
        assert torch.equal(b.get_state(m), g.get_state()), n
        assert np.allclose(hist[:, m], alone, rtol=1e-12, atol=0), n
        g.close()
    b.close()
