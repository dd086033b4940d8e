"""Work splits of the binary64-register kernels: an even split of all planes
over the SMs and chunks of planes per CTA give bitwise the same state and the
same diagnostics, where the runs cross tiles, end inside them, or hold one plane."""
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


# fewer planes than CTA slots; one more and one less than a full wave (304 planes of 16 x 8 tiles); runs over several
# tiles; the last tile one column, or one column short; a chunk that beats the split
SIZES = [(5, 5, 5), (33, 9, 7), (32, 8, 151), (32, 8, 153), (16, 8, 304), (17, 8, 23), (31, 8, 23), (40, 17, 61),
         (48, 48, 24), (150, 75, 61)]


@pytest.mark.parametrize("precision", [0, 3])
@pytest.mark.parametrize("n", SIZES)
def test_splits_agree_bitwise(S, n, precision):
    seen = []
    # the rule takes the chunks for some of these and the even split for others; the last one with the TMEM queue
    for zc, zq in ((4, 0), (21, 0), (n[2], 0), (21, 1)):
        g = S.Grid(n, precision)
        g.set_config(8, max(4, zc), zq, 1)
        g.init_tgv(0.9)
        hist = g.step_n_history(2, 1e-3).cpu().numpy()
        g.step_n(1, 1e-3)
        seen.append((g.get_state().clone(), g.rhs().clone(), hist))
        g.close()
    for q, r, h in seen[1:]:
        assert torch.equal(q, seen[0][0]) and torch.equal(r, seen[0][1])
        assert np.allclose(h, seen[0][2], rtol=1e-13, atol=0)  # partial sums of other groups of points


@pytest.mark.parametrize("precision", [0, 3])
def test_batch_members_cross_ctas(S, precision):
    """Members of one plane a CTA and of many: state bitwise and diagnostics as alone."""
    sizes = [(5, 5, 5), (64, 40, 37), (33, 9, 7), (40, 17, 61), (32, 8, 150)]
    b = S.Batch(sizes, precision)
    b.init_tgv([1.0] * len(sizes))
    hist = b.step_n_history(2, 1e-3).cpu().numpy()
    for m, n in enumerate(sizes):
        g = S.Grid(n, precision)
        g.init_tgv(1.0)
        alone = g.step_n_history(2, 1e-3).cpu().numpy()
        assert torch.equal(b.get_state(m), g.get_state()), n
        assert np.allclose(hist[:, m], alone, rtol=1e-12, atol=0), n
        g.close()
    b.close()
