"""The vorticity of the stage kernels' diagnostics is a difference of two
derivatives: where the two are the same sum of the same values it is zero, bit
for bit, however large they are."""
import math

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


BINARY32 = [(8, 8, 0, 1), (8, 8, 1, 1), (16, 8, 0, 1), (16, 8, 1, 1), (8, 8, 0, 2)]


@pytest.mark.parametrize("precision,configs", [(0, [(8, 8, 0, 1), (8, 8, 1, 1)]), (1, BINARY32), (2, BINARY32),
                                               (3, [(8, 8, 0, 1), (8, 8, 1, 1)])])
def test_irrotational_strain_has_no_enstrophy(S, precision, configs):
    """u0 = u1 = f(x0 + x1), u2 = 0: D1_x0 u1 and D1_x1 u0 are equal.  The
    derivatives along x2 are exactly zero too: the values have 20 bits and the
    weights there are powers of two (1/(12 h) = 2, which sets L)."""
    n = (23, 23, 32)
    L = n[2] / (24.0 * 2.0 * math.pi)
    f = np.random.default_rng(5).integers(-2**19, 2**19, n[0]) / 2.0**19
    v = f[(np.arange(n[0])[None, :] + np.arange(n[1])[:, None]) % n[0]]
    q = np.zeros((5, n[2], n[1], n[0]))
    q[0] = 1.0
    q[1:3] = v
    q[4] = 200.0
    for cfg in configs:
        g = S.Grid(n, precision, L=L)
        g.set_config(*cfg)
        g.set_state(torch.from_numpy(q))
        ke, ens = g.step_n_history(1, 1e-5)[0].tolist()
        assert ens == 0.0, (cfg, ke, ens)
        assert ke == pytest.approx(np.mean(v * v), rel=1e-6)
        g.close()
