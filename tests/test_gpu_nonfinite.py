"""States that have blown up at one point (infinities, NaNs, values too large
for the integer stencil sums, so that the lanes of a warp take different
branches): the TMEM queue gives the bits of the shared-memory ring, and points
out of the stencils' reach keep the bits of the run without the bad value."""
import numpy as np
import pytest

from paper_1709_09713_gb300 import workloads

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu

N = (40, 33, 48)
E0 = 1.0 / (1.4 * 0.4 * 0.01)
BAD = (3, 17, 5)  # x2, x1, x0: inside a warp's row, two columns from a tile's halo


@pytest.fixture(scope="module")
def S():
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_1709_09713_gb300 import build

    build.build()
    from paper_1709_09713_gb300 import sbli

    sbli.lib()
    return sbli


def _run(S, q, precision, cfg):
    g = S.Grid(N, precision)
    g.set_config(*cfg)
    g.set_state(q)
    r = g.rhs().clone()
    g.step_n_history(1, 1e-4)  # the stage kernels with and without diagnostics
    out = torch.stack([r, g.get_state()]).cpu().numpy()
    g.close()
    return out


def _same(a, b):
    return np.array_equal(np.isnan(a), np.isnan(b)) and np.array_equal(np.nan_to_num(a), np.nan_to_num(b))


def _away(reach):
    """Points further than `reach` from the bad one along some axis."""
    far = [np.minimum((np.arange(n) - b) % n, (b - np.arange(n)) % n) > reach for n, b in zip(N[::-1], BAD)]
    return far[0][:, None, None] | far[1][None, :, None] | far[2][None, None, :]


@pytest.mark.parametrize("precision,configs", [(0, ((8, 12, 0, 1), (8, 12, 1, 1))), (3, ((8, 12, 0, 1), (8, 12, 1, 1))),
                                               (1, ((8, 12, 0, 1), (8, 12, 1, 1), (16, 12, 1, 1))),
                                               (2, ((8, 12, 0, 1), (8, 12, 1, 1), (16, 12, 1, 1)))])
def test_bad_point_stays_local_and_queues_agree(S, precision, configs):
    clean = torch.from_numpy(workloads.smooth_state(N, 23, offsets=(1.0, 0.0, 0.0, 0.0, E0 + 0.5)))
    want = _run(S, clean, precision, configs[0])
    rhs_away, step_away = _away(4), _away(12)  # D1 of D1, three stages
    for field in (0, 1, 4):
        for value in (float("inf"), float("-inf"), float("nan"), 1.5e308):
            q = clean.clone()
            q[(field,) + BAD] = value
            runs = [_run(S, q, precision, cfg) for cfg in configs]
            for out in runs:
                assert _same(out, runs[0]), (field, value)
                assert not np.isfinite(out[1][field][BAD]), (field, value)
                assert np.array_equal(out[0][:, rhs_away], want[0][:, rhs_away]), (field, value)
                assert np.array_equal(out[1][:, step_away], want[1][:, step_away]), (field, value)


def _finite_residual(q, n):
    """Where Eqs. 1-3 on binary64 values give a number: m / rho is a division (0 of an infinite density)."""
    gm1, gm2 = 0.4, 1.4 * 0.01
    at = lambda f, a, s: np.roll(f, -s, 2 - a)  # noqa: E731
    d1 = lambda f, a: 8.0 * (at(f, a, 1) - at(f, a, -1)) - (at(f, a, 2) - at(f, a, -2))  # noqa: E731
    d2 = lambda f, a: 16.0 * (at(f, a, 1) + at(f, a, -1)) - (at(f, a, 2) + at(f, a, -2)) - 30.0 * f  # noqa: E731
    with np.errstate(all="ignore"):
        rho_p, E = q[0] - 1.0, q[4] - E0
        rho = 1.0 + rho_p
        u = [q[1 + i] / rho for i in range(3)]
        p = gm1 * (E - 0.5 * rho * (u[0] * u[0] + u[1] * u[1] + u[2] * u[2]))
        t = (gm2 * p - rho_p) / rho
        du = [[d1(u[i], j) for j in range(3)] for i in range(3)]
        div = du[0][0] + du[1][1] + du[2][2]
        skew = lambda f: f * div + sum(d1(f * u[j], j) + u[j] * d1(f, j) for j in range(3))  # noqa: E731
        visc = [sum(d2(u[i], j) + (0.0 if i == j else d1(du[j][j], i)) for j in range(3)) for i in range(3)]
        r = [rho * div + sum(d1(q[1 + j], j) + u[j] * d1(rho_p, j) for j in range(3))]
        r += [skew(q[1 + i]) + d1(p, i) + visc[i] for i in range(3)]
        r.append(skew(E) + sum(d1(p * u[j], j) + d2(t, j) + u[j] * visc[j] for j in range(3)) +
                 sum(du[i][j] * (du[i][j] + du[j][i]) for i in range(3) for j in range(3)))
    return np.isfinite(np.stack(r))


@pytest.mark.parametrize("variant", ["SBLI_STORE_ALL", "SBLI_RS", "SBLI_SS", "SBLI_RA", "SBLI_SN", "SBLI_SN2"])
def test_classes_divide_as_binary64_does(S, variant):
    """An infinite density or momentum takes the residual from the points where it
    takes it by the rules of division, and from no others."""
    clean = workloads.smooth_state(N, 23, offsets=(1.0, 0.0, 0.0, 0.0, E0 + 0.5))
    for field, value in ((0, np.inf), (1, -np.inf), (0, np.nan), (4, np.inf)):
        q = clean.copy()
        q[(field,) + BAD] = value
        g = S.Grid(N, S.SBLI_FP64, getattr(S, variant))
        g.set_state(torch.from_numpy(q))
        got = np.isfinite(g.rhs().cpu().numpy())
        g.close()
        assert np.array_equal(got, _finite_residual(q, N)), (field, value, got.sum(), _finite_residual(q, N).sum())
