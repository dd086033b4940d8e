"""Rounding of the classes that store derivatives: their residuals are as close to
the exact one (extended precision on the host) as that of the class that stores none,
whose derivatives are plain binary64 expressions."""
import numpy as np
import pytest

from paper_1709_09713_gb300 import workloads

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu

LD = np.longdouble
E0 = 1.0 / (1.4 * 0.4 * 0.01)


@pytest.fixture(scope="module")
def S():
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    if np.finfo(LD).eps > 1e-18:
        pytest.skip("no extended precision")
    from paper_1709_09713_gb300 import build

    build.build()
    from paper_1709_09713_gb300 import sbli

    sbli.lib()
    return sbli


def exact_residual(q, n):
    """Eqs. 1-7 in deviations from rho = 1, T = 1 (Re 1600, M 0.1, Pr 0.71)."""
    g, m, pr, re = LD(1.4), LD(0.1), LD(0.71), LD(1600)
    h = [LD("6.283185307179586476925286766559005768") / v for v in n]
    at = lambda f, a, s: np.roll(f, -s, 2 - a)  # noqa: E731
    d1 = lambda f, a: (8 * (at(f, a, 1) - at(f, a, -1)) - (at(f, a, 2) - at(f, a, -2))) / (12 * h[a])  # noqa: E731
    d2 = lambda f, a: (16 * (at(f, a, 1) + at(f, a, -1)) - (at(f, a, 2) + at(f, a, -2)) - 30 * f) / (12 * h[a] ** 2)  # noqa: E731
    rho = 1 + q[0]
    u = [q[1 + i] / rho for i in range(3)]
    p = (g - 1) * (q[4] - sum(q[1 + i] * u[i] for i in range(3)) / 2)
    t = (g * m * m * p - q[0]) / rho
    du = [[d1(u[i], j) for j in range(3)] for i in range(3)]
    div = du[0][0] + du[1][1] + du[2][2]
    skew = lambda f: -(sum(d1(f * u[j], j) + u[j] * d1(f, j) for j in range(3)) + f * div) / 2  # noqa: E731
    r = [-(sum(d1(q[1 + j], j) + u[j] * d1(q[0], j) for j in range(3)) + rho * div) / 2]
    work = -2 * div * div / 3 + sum(du[i][j] * (du[i][j] + du[j][i]) for i in range(3) for j in range(3))
    for i in range(3):
        visc = sum(d2(u[i], j) + (d2(u[i], i) if i == j else d1(du[j][j], i)) / 3 for j in range(3))
        work = work + u[i] * visc
        r.append(skew(q[1 + i]) - d1(p, i) + visc / re)
    r.append(skew(q[4]) - div / ((g - 1) * m * m) + work / re +
             sum(d2(t, j) / ((g - 1) * m * m * pr * re) - d1(p * u[j], j) for j in range(3)))
    return np.stack(r)


def test_stored_derivatives_are_as_close(S):
    rng = np.random.default_rng(77)
    variants = ("SBLI_RA", "SBLI_RS", "SBLI_SS", "SBLI_STORE_ALL")
    square = {v: np.zeros(5) for v in variants}
    for seed in range(16):
        n = tuple(int(v) for v in rng.integers(14, 40, 3))
        q = workloads.smooth_state(n, seed, offsets=(1.0, 0.0, 0.0, 0.0, E0 + 0.5))
        dev = q.copy()
        dev[0] -= 1.0
        dev[4] -= E0
        want = exact_residual(dev.astype(LD), n)
        scale = [float(np.sqrt(np.mean(w * w))) for w in want]
        for v in variants:
            g = S.Grid(n, S.SBLI_FP64, getattr(S, v))
            g.set_state(torch.from_numpy(q).cuda())
            r = g.rhs().cpu().numpy()
            g.close()
            square[v] += [float(np.mean((r[f] - want[f]) ** 2)) / scale[f] ** 2 for f in range(5)]
    for v in variants[1:]:
        # 16 grids of some 20,000 points average the ratio of two sums of rounding errors to about a thousandth
        assert (np.sqrt(square[v] / square["SBLI_RA"]) <= 1.002).all(), (v, np.sqrt(square[v] / square["SBLI_RA"]))
