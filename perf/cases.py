"""The workloads whose speed this repository is judged by, each one pass
through the public entry points as a user's program makes them.

Every case starts from conserved variables that the program holds on the GPU
(a Taylor-Green vortex of its own amplitude with a smooth random perturbation
of all five fields, so that no symmetry makes a term vanish) and returns the
fields that the call computes, one tensor per field: the energy field is a
hundred times larger than the momenta and would hide them in a common norm.

The sizes are those of the repository's tests and benchmark (32^3, 256^3,
512^3, ensembles of 32^3 ... 128^3, requests log-uniform in 32 ... 256) and
ragged ones between them: edges that are no multiple of a tile, short and long
x2 extents.
"""
import math

import numpy as np
import torch

from paper_1709_09713_gb300 import sbli as S

RE, MACH, PR, GAMMA = 1600.0, 0.1, 0.71, 1.4
PRECISION = {"fp64": S.SBLI_FP64, "fp32": S.SBLI_FP32, "fp32df": S.SBLI_FP32_DF, "df64": S.SBLI_DF64}
VARIANT = {"fused": S.SBLI_FUSED, "BL": S.SBLI_STORE_ALL, "RS": S.SBLI_RS, "SS": S.SBLI_SS, "RA": S.SBLI_RA,
           "SN": S.SBLI_SN, "SN2": S.SBLI_SN2}
ENSEMBLE_EDGES = (32, 48, 64, 96, 128)


def _grid(n, precision, steps, tune=False, variant="fused", kind="solve", dt=1e-3):
    return {"kind": kind, "n0": n[0], "n1": n[1], "n2": n[2], "precision": precision, "variant": variant, "steps": steps,
            "dt": dt, "tune": tune}


def _solve(name, *args, **options):
    return {"name": name, **_grid(*args, **options)}


def listed():
    return [
        # the small validation run: ten steps of 32^3 in binary64, launch by launch too short to fill the GPU
        _solve("solve 32 fp64", (32, 32, 32), "fp64", 10),
        # the paper's own grid in binary64, a few steps of a long run
        _solve("solve 256 fp64", (256, 256, 256), "fp64", 2),
        # the residual alone, for a program with its own time integrator, on an uneven box
        _solve("rhs 150x75x61 fp64", (150, 75, 61), "fp64", 1, kind="rhs"),
        # double-float arithmetic, the fast path to binary64 accuracy: an uneven box and the paper's grid
        _solve("solve 129x97x66 df64", (129, 97, 66), "df64", 6),
        _solve("solve 256 df64", (256, 256, 256), "df64", 3, tune=True),
        # the large binary32 run with the binary64 accumulator, autotuned as such a run is
        _solve("solve 512 fp32", (512, 512, 512), "fp32", 8, tune=True, dt=5e-4),
        # a small binary32 run without autotuning
        _solve("solve 40 fp32", (40, 40, 40), "fp32", 24),
        # kinetic energy and enstrophy of every step, binary32 with the double-float accumulator
        _solve("history 192 fp32df", (192, 192, 192), "fp32df", 10, tune=True, kind="history"),
        # the 64-member ensemble of uneven grids and parameters, one launch per stage
        {"name": "ensemble 64 fp32", "kind": "ensemble", "members": 64, "max_edge": 128, "precision": "fp32", "steps": 6,
         "dt": 1e-3, "tune": True},
        # a burst of requests of both precision classes through the serving loop
        {"name": "serving 8", "kind": "serving", "requests": 8, "max_edge": 96, "fp64_as": "df64", "steps": 40, "dt": 1e-3},
        # restart and monitoring: a state in, its kinetic energy and enstrophy by both entry points, the state out
        _solve("monitor 160x200x120 fp64", (160, 200, 120), "fp64", 0, kind="monitor"),
        # the paper's store-all algorithm, the comparison every user of the paper's classes makes
        _solve("solve 128 fp64 BL", (128, 128, 128), "fp64", 2, variant="BL"),
    ]


def _edge(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def draw(rng):
    kind = rng.choice(["solve"] * 6 + ["rhs", "history", "ensemble", "serving", "monitor", "class"])
    if kind == "ensemble":
        return {"kind": kind, "members": _edge(rng, 2, 48), "max_edge": rng.choice(ENSEMBLE_EDGES[2:]),
                "precision": rng.choice(list(PRECISION)), "steps": rng.randint(1, 6), "dt": 1e-3,
                "tune": rng.random() < 0.5}
    if kind == "serving":
        return {"kind": kind, "requests": rng.randint(2, 10), "max_edge": _edge(rng, 40, 112),
                "fp64_as": rng.choice(["fp64", "df64"]), "steps": rng.randint(10, 40), "dt": 1e-3}
    # a box of up to 256^3 points whose edges differ by up to a factor of two or so
    e = math.exp(rng.uniform(math.log(16.0), math.log(230.0)))
    n = tuple(max(5, min(320, int(round(e * math.exp(rng.uniform(-0.4, 0.4)))))) for _ in range(3))
    points = n[0] * n[1] * n[2]
    precision = rng.choice(list(PRECISION))
    if kind == "class":
        return _grid(n, "fp64", 1, variant=rng.choice(["BL", "RS", "SS", "RA", "SN", "SN2"]))
    if kind == "monitor":
        return _grid(n, precision, 0, kind="monitor")
    if kind == "rhs":
        return _grid(n, precision, 1, kind="rhs")
    most = 2 if points > 6e6 else 12 if points > 5e5 else 24
    return _grid(n, precision, rng.randint(1, most), kind=kind, tune=points > 4e6 and rng.random() < 0.5)


# ------------------------------------------------------------------ inputs

def _axes(n, device):
    return [torch.arange(n[a], dtype=torch.float64, device=device) * (2.0 * math.pi / n[a]) for a in range(3)]


def _initial_state(n, seed, mach=MACH, scale=1e-2):
    """A perturbed Taylor-Green field (5, n2, n1, n0), binary64, on the GPU."""
    rng = np.random.default_rng(seed)
    device = torch.device("cuda")
    x, y, z = _axes(n, device)
    x, y, z = x[None, None, :], y[None, :, None], z[:, None, None]
    amp = float(rng.uniform(0.9, 1.1))
    gm2 = GAMMA * mach * mach
    q = torch.empty((5, n[2], n[1], n[0]), dtype=torch.float64, device=device)
    u0 = amp * torch.sin(x) * torch.cos(y) * torch.cos(z)
    u1 = -amp * torch.cos(x) * torch.sin(y) * torch.cos(z)
    dp = amp * amp / 16.0 * (torch.cos(2 * x) + torch.cos(2 * y)) * (2.0 + torch.cos(2 * z))
    q[0] = 1.0 + gm2 * dp
    q[1] = q[0] * u0
    q[2] = q[0] * u1
    q[3] = 0.0
    q[4] = 1.0 / (GAMMA * (GAMMA - 1.0) * mach * mach) + dp / (GAMMA - 1.0) + 0.5 * q[0] * (u0 * u0 + u1 * u1)
    del u0, u1, dp

    def series(t):
        out = torch.zeros_like(t)
        for k in range(1, 5):
            out += float(rng.uniform(-1.0, 1.0)) / k * torch.cos(k * t + float(rng.uniform(0.0, 2.0 * math.pi)))
        return out

    for f in range(5):
        for _ in range(2):
            a, b, c = series(x), series(y), series(z)
            q[f] += (0.5 * scale) * (c * b) * a
    return q


def _members(case, seed):
    """The edges are the case's, the parameters and states the seed's."""
    shape, rng = np.random.default_rng(1709), np.random.default_rng(seed)
    edges = [e for e in ENSEMBLE_EDGES if e <= case["max_edge"]]
    sizes = [(int(n),) * 3 for n in shape.choice(edges, size=case["members"])]
    re = [float(v) for v in rng.uniform(100.0, 1600.0, len(sizes))]
    mach = [float(v) for v in rng.uniform(0.1, 0.4, len(sizes))]
    return sizes, re, mach


def _requests(case, seed):
    """(edge, precision, steps) are the case's; amplitude and Reynolds number the seed's."""
    shape, rng = np.random.default_rng(20), np.random.default_rng(seed)
    out = []
    for _ in range(case["requests"]):
        n = math.exp(shape.uniform(math.log(32.0), math.log(case["max_edge"])))
        n = int(min(case["max_edge"], max(32, 8 * round(n / 8.0))))
        steps = int(shape.integers(max(1, case["steps"] // 4), case["steps"] + 1))
        precision = "fp32" if shape.integers(0, 2) else case["fp64_as"]
        out.append((n, precision, steps, float(rng.uniform(400.0, 1600.0)), float(rng.uniform(0.9, 1.1))))
    return out


def _n(case):
    return case["n0"], case["n1"], case["n2"]


def prepare(case, seed):
    kind = case["kind"]
    if kind == "ensemble":
        sizes, re, mach = _members(case, seed)
        b = S.Batch(sizes, PRECISION[case["precision"]], Re=re, Mach=mach)
        q = [_initial_state(n, seed + 1000 * m, mach[m]) for m, n in enumerate(sizes)]
        for m, v in enumerate(q):
            b.set_state(m, v)
        if case["tune"]:
            b.autotune(2)
        return {"case": case, "batch": b, "q": q, "out": [torch.empty_like(v) for v in q]}
    if kind == "serving":
        reqs = _requests(case, seed)
        out = [torch.empty((5, n, n, n), dtype=torch.float64, device="cuda") for n, *_ in reqs]
        made = [S.request(n, PRECISION[p], steps, case["dt"], Re=re, amplitude=amp, result=out[i])
                for i, (n, p, steps, re, amp) in enumerate(reqs)]
        arena = sum(S.sbli_server_request_bytes(r) + 4096 for r in made)
        return {"case": case, "server": S.Server(arena, max_slots=len(made)), "requests": made, "out": out}
    n = _n(case)
    g = S.Grid(n, PRECISION[case["precision"]], VARIANT[case["variant"]], Re=RE, Mach=MACH, Pr=PR, gamma=GAMMA)
    q = _initial_state(n, seed)
    g.set_state(q)
    if case["tune"]:
        g.autotune(3)
    state = {"case": case, "grid": g, "q": q, "out": torch.empty_like(q)}
    if kind == "monitor":
        state["ke"] = torch.empty(4, dtype=torch.float64, device="cuda")
    return state


def _fields(q):
    return [q[f] for f in range(5)]


def run(state):
    case = state["case"]
    kind = case["kind"]
    if kind == "ensemble":
        b = state["batch"]
        for m, v in enumerate(state["q"]):
            b.set_state(m, v)
        b.step_n(case["steps"], case["dt"])
        return [b.get_state(m, o) for m, o in enumerate(state["out"])]
    if kind == "serving":
        srv = state["server"]
        ids = {srv.submit(r): i for i, r in enumerate(state["requests"])}
        done = {}
        while len(done) < len(ids):
            srv.tick()
            for r in srv.poll():
                done[ids[r.id]] = (r.ke, r.enstrophy)
        return {"state": state["out"], "ke": np.array([done[i] for i in range(len(ids))])}
    g, q, out = state["grid"], state["q"], state["out"]
    g.set_state(q)
    if kind == "rhs":
        return _fields(g.rhs(out))
    if kind == "history":
        hist = g.step_n_history(case["steps"], case["dt"])
        return {"history": hist, "state": _fields(g.get_state(out))}
    if kind == "monitor":
        ke = state["ke"]
        stream = g.stream.cuda_stream
        S.sbli_kinetic_energy_async(g.handle, ke.data_ptr())
        S.sbli_kinetic_energy_noalloc(q.data_ptr(), *_n(case), 1.0, ke.data_ptr() + 16, stream)
        return {"ke": ke, "state": _fields(g.get_state(out))}
    g.step_n(case["steps"], case["dt"])
    return _fields(g.get_state(out))


# ------------------------------------------------------------------ what a pass costs at the least

# bytes per point and stage of the two-register scheme (stage field and accumulator once in, once out; the last stage
# writes no field): fifty values a step in binary64; binary32 fields with eight-byte accumulators
STAGE_BYTES = {"fp64": 400.0 / 3.0, "df64": 400.0 / 3.0, "fp32": 320.0 / 3.0, "fp32df": 320.0 / 3.0}
# operations per point and stage: 60 derivatives of 4 to 7 operations, the 15 products they are taken of, the primitives,
# the assembly of Eqs. 1-3 and the update
STAGE_FLOPS = 500.0


def work(case):
    kind = case["kind"]

    def solve(points, precision, steps):
        # the state in and out of the library's own form, and the stages
        return points * (160.0 + 3 * steps * STAGE_BYTES[precision]), points * 3 * steps * STAGE_FLOPS

    if kind == "ensemble":
        parts = [solve(n[0] * n[1] * n[2], case["precision"], case["steps"]) for n in _members(case, 0)[0]]
    elif kind == "serving":
        parts = [solve(n ** 3, p, steps) for n, p, steps, *_ in _requests(case, 0)]
    else:
        points = case["n0"] * case["n1"] * case["n2"]
        if kind == "rhs":
            parts = [(points * 160.0, points * STAGE_FLOPS)]
        elif kind == "monitor":
            parts = [(points * 160.0, points * 60.0)]
        else:
            parts = [solve(points, case["precision"], case["steps"])]
    return {"bytes": sum(b for b, _ in parts), "flops": sum(f for _, f in parts)}


# ------------------------------------------------------------------ the same in plain torch, 64 bits

RK_A, RK_B = (2.0 / 3.0, 5.0 / 12.0, 3.0 / 5.0), (1.0 / 4.0, 3.0 / 20.0, 3.0 / 5.0)


class _Method:
    """Eqs. 1-7 on whole arrays, in deviations from rho = 1, p = 1/(gamma M^2)."""

    def __init__(self, n, re, mach):
        self.h = [2.0 * math.pi / v for v in n]
        self.re, self.mach = re, mach
        self.gm2 = GAMMA * mach * mach
        self.e_ref = 1.0 / (GAMMA * (GAMMA - 1.0) * mach * mach)
        self.h_ref = 1.0 / ((GAMMA - 1.0) * mach * mach)
        self.kappa = 1.0 / ((GAMMA - 1.0) * mach * mach * PR * re)

    def d1(self, f, a):
        r = lambda s: torch.roll(f, -s, 2 - a)  # noqa: E731
        return (8.0 * (r(1) - r(-1)) - (r(2) - r(-2))) * (1.0 / (12.0 * self.h[a]))

    def d2(self, f, a):
        r = lambda s: torch.roll(f, -s, 2 - a)  # noqa: E731
        return (16.0 * (r(1) + r(-1)) - (r(2) + r(-2)) - 30.0 * f) * (1.0 / (12.0 * self.h[a] ** 2))

    def primitives(self, q):
        rho = 1.0 + q[0]
        u = [q[1 + i] / rho for i in range(3)]
        p = (GAMMA - 1.0) * (q[4] - 0.5 * (q[1] * u[0] + q[2] * u[1] + q[3] * u[2]))
        return rho, u, p, (self.gm2 * p - q[0]) / rho

    def residual(self, q):
        rho, u, p, t = self.primitives(q)
        r = torch.empty_like(q)
        du = [[self.d1(u[i], j) for j in range(3)] for i in range(3)]
        div = du[0][0] + du[1][1] + du[2][2]
        c = rho * div
        for j in range(3):
            c += self.d1(q[1 + j], j) + u[j] * self.d1(q[0], j)
        r[0] = -0.5 * c
        work = torch.zeros_like(div)
        for i in range(3):
            m = q[1 + i]
            c = m * div
            for j in range(3):
                c += self.d1(m * u[j], j) + u[j] * self.d1(m, j)
            visc = torch.zeros_like(div)
            for j in range(3):
                visc += self.d2(u[i], j) + (self.d2(u[i], i) if i == j else self.d1(du[j][j], i)) / 3.0
            work += u[i] * visc
            r[1 + i] = -0.5 * c - self.d1(p, i) + visc / self.re
        for i in range(3):
            for j in range(3):
                work += du[i][j] * (du[i][j] + du[j][i])
        work -= (2.0 / 3.0) * div * div
        c = q[4] * div
        for j in range(3):
            c += self.d1(q[4] * u[j], j) + u[j] * self.d1(q[4], j)
        c = -0.5 * c - self.h_ref * div + work / self.re
        del du
        for j in range(3):
            c += self.kappa * self.d2(t, j) - self.d1(p * u[j], j)
        r[4] = c
        return r

    def averages(self, q):
        rho, u, _, _ = self.primitives(q)
        ke = (0.5 * rho * (u[0] ** 2 + u[1] ** 2 + u[2] ** 2)).mean()
        w = [self.d1(u[2], 1) - self.d1(u[1], 2), self.d1(u[0], 2) - self.d1(u[2], 0), self.d1(u[1], 0) - self.d1(u[0], 1)]
        return torch.stack([ke, (0.5 * rho * (w[0] ** 2 + w[1] ** 2 + w[2] ** 2)).mean()])

    def deviations(self, q):
        q = q.clone()
        q[0] -= 1.0
        q[4] -= self.e_ref
        return q

    def plain(self, q):
        q = q.clone()
        q[0] += 1.0
        q[4] += self.e_ref
        return q

    def advance(self, q, steps, dt, history=None):
        for _ in range(steps):
            if history is not None:
                history.append(self.averages(q))
            acc = q.clone()
            for a, b in zip(RK_A, RK_B):
                r = self.residual(q)
                q = acc + (a * dt) * r
                acc += (b * dt) * r
            q = acc
        return q


def _taylor_green(n, mach, amp):
    """The library's own initial field for a request (deviations)."""
    x, y, z = _axes(n, torch.device("cuda"))
    x, y, z = x[None, None, :], y[None, :, None], z[:, None, None]
    u0 = amp * torch.sin(x) * torch.cos(y) * torch.cos(z)
    u1 = -amp * torch.cos(x) * torch.sin(y) * torch.cos(z)
    dp = amp * amp / 16.0 * (torch.cos(2 * x) + torch.cos(2 * y)) * (2.0 + torch.cos(2 * z))
    rho = 1.0 + GAMMA * mach * mach * dp
    return torch.stack([rho - 1.0, rho * u0, rho * u1, torch.zeros_like(dp),
                        dp / (GAMMA - 1.0) + 0.5 * rho * (u0 * u0 + u1 * u1)])


def exact(case, seed):
    kind = case["kind"]
    if kind == "ensemble":
        sizes, re, mach = _members(case, seed)
        out = []
        for m, n in enumerate(sizes):
            e = _Method(n, re[m], mach[m])
            q = e.deviations(_initial_state(n, seed + 1000 * m, mach[m]))
            out.append(e.plain(e.advance(q, case["steps"], case["dt"])))
        return out
    if kind == "serving":
        states, ke = [], []
        for n, _, steps, re, amp in _requests(case, seed):
            e = _Method((n,) * 3, re, MACH)
            q = e.advance(_taylor_green((n,) * 3, MACH, amp), steps, case["dt"])
            states.append(e.plain(q))
            ke.append(e.averages(q))
        return {"state": states, "ke": torch.stack(ke).cpu().numpy()}
    n = _n(case)
    e = _Method(n, RE, MACH)
    q = e.deviations(_initial_state(n, seed))
    if kind == "rhs":
        return _fields(e.residual(q))
    if kind == "monitor":
        v = e.averages(q)
        return {"ke": torch.cat([v, v]), "state": _fields(e.plain(q))}
    history = [] if kind == "history" else None
    state = _fields(e.plain(e.advance(q, case["steps"], case["dt"], history)))
    return {"history": torch.stack(history), "state": state} if kind == "history" else state


# About four times what another order of the sums was seen to make of the worst field (the x2 momentum, a hundredth of the
# others, on the finest grids): 6.6e-15 binary64, 5.4e-13 double-float, 1e-5 binary32 for a state after its steps; the
# residual alone is 1/(h dt) less exact.
STATE_TOLERANCE = {"fp64": 5e-14, "df64": 3e-12, "fp32": 5e-5, "fp32df": 5e-5}
RHS_TOLERANCE = {"fp64": 1e-11, "df64": 4e-10, "fp32": 1e-2, "fp32df": 1e-2}


def tolerance(case):
    # a burst of requests holds binary32 ones
    precision = "fp32" if case["kind"] == "serving" else case["precision"]
    return {"rel": (RHS_TOLERANCE if case["kind"] == "rhs" else STATE_TOLERANCE)[precision]}
