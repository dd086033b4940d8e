"""Grids of more x2 planes than 65,535 blocks of planes: the initial field, the
state in and out, diagnostics and a residual."""
import numpy as np
import pytest

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu

N = (5, 6, 2**21 + 70)


@pytest.fixture(scope="module")
def S():
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_1709_09713_gb300 import build

    build.build()
    from paper_1709_09713_gb300 import sbli

    sbli.lib()
    return sbli


def test_initial_field_of_a_long_grid(S):
    rng = np.random.default_rng(3)
    k = np.concatenate([[0, 31, 32, 2**21 - 1, 2**21, N[2] - 1], rng.integers(0, N[2], 500)])
    i, j = rng.integers(0, N[0], k.size), rng.integers(0, N[1], k.size)
    g = S.Grid(N, S.SBLI_FP64)
    g.init_tgv(0.9)
    q = g.sample_state(torch.from_numpy(i + N[0] * (j + N[1] * k.astype(np.int64))).cuda()).cpu().numpy()
    x, y, z = (2.0 * np.pi / n * v for n, v in zip(N, (i, j, k)))
    u0 = 0.9 * np.sin(x) * np.cos(y) * np.cos(z)
    u1 = -0.9 * np.cos(x) * np.sin(y) * np.cos(z)
    dp = 0.81 / 16.0 * (np.cos(2 * x) + np.cos(2 * y)) * (2.0 + np.cos(2 * z))
    rho = 1.0 + 1.4 * 0.01 * dp
    want = np.stack([rho, rho * u0, rho * u1, 0 * rho, (1.0 / (1.4 * 0.01) + dp) / 0.4 + 0.5 * rho * (u0**2 + u1**2)])
    # 2 pi k / n and the products of it: a few units in the last place of 2 pi, of each field's size
    assert (np.abs(q - want) <= 1e-14 * np.abs(want).max(1, keepdims=True)).all()
    ke, _ = g.kinetic_energy()
    # the average of the exact field: sin^2 and cos^2 average 1/2 on 5 and 6 points, rho to first order in the Mach number squared
    assert ke == pytest.approx(0.81 / 8.0, rel=5e-3)
    assert torch.isfinite(g.rhs()).all()
    g.close()
