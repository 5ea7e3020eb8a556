"""Workloads by which the framework's speed is measured.

Each case is one pass through a public entry point as a user's program calls
it: stepping one tank or a batch of tanks (``Sim.step``), the tangent, the
adjoint and the linearization of the step (``Sim.jvp``, ``Sim.vjp``,
``Sim.eval_jvp``), and fitting and running the two surrogates (``lpv.Model``,
``slpv.VelocityModel``).  Tank configurations come from ``workloads``; sizes
from the tests, ``bench.py`` and ``pipeline``.

``listed`` names the cases, ``draw`` gives more of the same ranges,
``prepare`` makes a case's inputs and handles from a seed, ``run`` is one
pass, ``work`` what a pass cannot do without, and ``exact`` the same outputs
in 64 bits by plain torch.
"""
from __future__ import annotations

import math

import numpy as np
import torch

from paper_2604_12505_gb300 import workloads as W

# ---------------------------------------------------------------------------
# the cases
# ---------------------------------------------------------------------------
_FLIGHT = dict(kind="flight", family="BASE", R=0.5, fill=0.5, tanks=1, outer=10, pd=True)


def listed() -> list[dict]:
    return [
        # one sampling period of the small tank, as a control loop around the
        # simulator calls it: the smallest call
        dict(_FLIGHT, name="period_small", dx=0.02, steps=10),
        # the paper's spacecraft (Tables 1-2) flown under the PD attitude law
        dict(_FLIGHT, name="flight_paper", family="PAPER_RINGS", R=0.2, fill=0.6, dx=0.006, outer=50, steps=100),
        # the benchmark tank, 97,748 particles
        dict(_FLIGHT, name="flight_large", dx=0.002, steps=100, pd=False),
        # data set generation: tanks of uneven size stepped together
        dict(_FLIGHT, name="batch", tanks=64, dx=0.004, dx_hi=0.01, fill=0.2, fill_hi=0.8, steps=20, pd=False),
        # the linearization study: copies of the paper's spacecraft, one column of df/dx each
        dict(kind="linearize", name="linearize", family="PAPER_RINGS", R=0.2, fill=0.6, dx=0.006, tanks=256),
        # the differentiation tank, 15,532 particles, windows of 50 steps: forward and reverse mode
        dict(kind="tangent", name="tangent", family="BASE", R=0.5, fill=0.5, dx=0.005, outer=10, steps=50),
        dict(kind="adjoint", name="adjoint", family="BASE", R=0.5, fill=0.5, dx=0.005, outer=10, steps=50, every=10),
        # one iteration of the load surrogate's fit at the study's size
        dict(kind="lpv_gradient", name="lpv_gradient", n_traj=820, T=1000, na=3, n_y=4, n_p=2),
        # its free run on the held-out trajectories
        dict(kind="lpv_predict", name="lpv_predict", n_traj=204, T=1000, na=3, n_y=4, n_p=2),
        # its closed loop in bulk (Monte-Carlo runs of the attitude controller)
        dict(kind="lpv_loop", name="lpv_loop", runs=65536, T=500, na=3, n_y=4, n_p=2),
        # the velocity-level surrogate: one iteration of its fit on the identification trains
        dict(kind="slpv_gradient", name="slpv_gradient", n_traj=24, T=2200, nx=4),
        # and its closed loop in bulk
        dict(kind="slpv_loop", name="slpv_loop", runs=65536, T=600, nx=4),
    ]


def _log_uniform(rng, lo, hi) -> float:
    return math.exp(rng.uniform(math.log(lo), math.log(hi)))


def _log_int(rng, lo, hi) -> int:
    return min(hi, max(lo, int(round(_log_uniform(rng, lo, hi)))))


def draw(rng) -> dict:
    kind = rng.choice(["flight", "flight", "flight", "batch", "linearize", "tangent", "adjoint", "lpv_gradient",
                       "lpv_predict", "lpv_loop", "slpv_gradient", "slpv_loop"])
    if kind in ("flight", "tangent", "adjoint", "linearize"):
        family = rng.choice(["BASE", "BASE", "PAPER_RINGS", "PAPER_CLAMP"])
        R = 0.5 if family == "BASE" else 0.2
        fill = rng.uniform(0.2, 0.8)
        outer = rng.choice([5, 10, 20])
        if kind == "flight":
            # up to the large tank's particles: fill pi R^2 / dx^2 <= 97,748
            dx = _log_uniform(rng, 0.0052 * R * math.sqrt(fill / 0.8), 0.04 * R)
            return dict(kind=kind, family=family, R=R, fill=fill, dx=dx, tanks=1, outer=outer,
                        steps=outer * _log_int(rng, 1, 100 // outer), pd=rng.random() < 0.5)
        if kind == "linearize":
            return dict(kind=kind, family=family, R=R, fill=fill, dx=_log_uniform(rng, 0.035 * R, 0.06 * R),
                        tanks=_log_int(rng, 8, 200))
        dx = _log_uniform(rng, 0.0128 * R * math.sqrt(fill / 0.8), 0.04 * R)
        c = dict(kind=kind, family=family, R=R, fill=fill, dx=dx, outer=outer, steps=outer * rng.randint(1, 40 // outer))
        return dict(c, every=rng.choice([5, 8, 10])) if kind == "adjoint" else c
    if kind == "batch":
        lo = rng.uniform(0.004, 0.006)
        return dict(kind="flight", family="BASE", R=0.5, fill=0.2, fill_hi=rng.uniform(0.4, 0.8), dx=lo,
                    dx_hi=lo * rng.uniform(1.2, 2.0), tanks=_log_int(rng, 3, 48), outer=10, steps=10 * rng.randint(1, 2),
                    pd=rng.random() < 0.5)
    if kind in ("lpv_gradient", "lpv_predict", "lpv_loop"):
        n_y, n_p = rng.choice([3, 4]), rng.choice([0, 1, 2])
        c = dict(kind=kind, na=rng.choice([1, 2, 3]), n_y=n_y, n_p=n_p)
        if kind == "lpv_loop":
            return dict(c, runs=_log_int(rng, 1, 65536), T=_log_int(rng, 50, 500))
        return dict(c, n_traj=_log_int(rng, 1, 820), T=_log_int(rng, 40, 1000))
    if kind == "slpv_gradient":
        return dict(kind=kind, n_traj=_log_int(rng, 1, 70), T=_log_int(rng, 40, 2000), nx=rng.choice([2, 4, 4, 6, 8]))
    return dict(kind=kind, runs=_log_int(rng, 1, 50000), T=_log_int(rng, 50, 600), nx=rng.choice([2, 4, 4, 6]))


# ---------------------------------------------------------------------------
# inputs
# ---------------------------------------------------------------------------
def _gen(seed):
    return torch.Generator(device="cuda").manual_seed(int(seed) % (1 << 62))


def _normal(g, *shape, std=1.0, dtype=torch.float64):
    return torch.randn(shape, generator=g, device="cuda", dtype=dtype) * std


def _uniform(g, *shape, lo=0.0, hi=1.0):
    return torch.rand(shape, generator=g, device="cuda", dtype=torch.float64) * (hi - lo) + lo


def _holds(g, rows, T, mean_hold, amp):
    """[rows, T] piecewise-constant values U[-amp, amp] held for about mean_hold samples."""
    jump = torch.rand((rows, T), generator=g, device="cuda") < 1.0 / mean_hold
    seg = jump.to(torch.int64).cumsum(1)
    return _uniform(g, rows, T + 1, lo=-amp, hi=amp).gather(1, seg)


def _tank_params(case) -> list[dict]:
    """One parameter dict per tank (a case's tanks, whatever the seed of its inputs)."""
    fam = case["family"]
    base = dict(W.BASE if fam == "BASE" else W.PAPER_RINGS if fam == "PAPER_RINGS" else W.PAPER)
    if fam == "PAPER_CLAMP":  # Table 2's single ghost layer holds the fluid when the wall only pushes
        base["ghost_pressure_clamp"] = 1
    base.update(R=case["R"], fill=case["fill"], dx=case["dx"])
    if "outer" in case:
        base["outer_every"] = case["outer"]
    if fam != "BASE":
        base["dt"] = min(base["dt"], 0.15 * base["dx"])  # the paper's 1 ms at its 6 mm, smaller below it
    if "dx_hi" not in case:
        return [base] * case.get("tanks", 1)
    r = np.random.default_rng(1000 + case["tanks"]).uniform(size=(case["tanks"], 2)).tolist()
    return [dict(base, fill=case["fill"] + a * (case["fill_hi"] - case["fill"]),
                 dx=case["dx"] + b * (case["dx_hi"] - case["dx"])) for a, b in r]


def _lattice(p) -> np.ndarray:
    """[n, 2] fluid lattice of a tank: ((i + 1/2) dx, (j + 1/2) dx) inside
    radius R - dx/2 and below the chord of the filled segment, row by row."""
    R, want = p["R"], p["fill"] * math.pi * p["R"] ** 2

    def area(c):
        return R * R * (math.pi - math.acos(c / R)) + c * math.sqrt(R * R - c * c) if abs(c) < R else \
            (0.0 if c < 0 else math.pi * R * R)

    lo, hi = -R, R
    for _ in range(200):
        mid = 0.5 * (lo + hi)
        lo, hi = (mid, hi) if area(mid) < want else (lo, mid)
    c, rin, L = 0.5 * (lo + hi), R - 0.5 * p["dx"], math.ceil(R / p["dx"]) + 2
    a = (np.arange(-L, L + 1) + 0.5) * p["dx"]
    y, x = np.meshgrid(a, a, indexing="ij")
    keep = (x * x + y * y <= rin * rin) & (y <= c)
    return np.stack([x[keep], y[keep]], axis=1)


def _ghosts(p) -> np.ndarray:
    """[n_g, 2] ghost rings of a tank in the body frame."""
    s, out = (p["ghost_spacing"] if p["ghost_spacing"] > 0 else 1.0) * p["dx"], []
    for k in range(p["n_rings"]):
        r = p["R"] + (k + 0.5) * s
        n = int(round(2.0 * math.pi * r / s))
        phi = 2.0 * math.pi * np.arange(n) / n
        out.append(np.stack([r * np.cos(phi), r * np.sin(phi)], axis=1))
    return np.concatenate(out)


def _sph_inputs(case, seed):
    """Parameters and inputs of a simulator case: a spawned fluid (the lattice
    with a jitter of a tenth of its spacing, moving with the tank plus a small
    random motion), the body in flight, piecewise-constant inputs."""
    g = _gen(seed)
    params = _tank_params(case)
    kind, B = case["kind"], len(params)
    body = _uniform(g, B, 6, lo=-1.0, hi=1.0) * torch.tensor([2e-3, 2e-3, 0.3, 0.01, 0.01, 0.1], device="cuda",
                                                             dtype=torch.float64)
    if kind == "linearize":  # copies of one state
        body = body[:1].repeat(B, 1)
    parts, memo = [], {}
    for b, p in enumerate(params):
        if kind == "linearize" and b:
            parts.append(parts[0])
            continue
        key = (p["fill"], p["dx"])
        if key not in memo:
            memo[key] = torch.tensor(_lattice(p), device="cuda")
        x = memo[key] + _uniform(g, *memo[key].shape, lo=-0.1, hi=0.1) * p["dx"]
        c, s = torch.cos(body[b, 2]), torch.sin(body[b, 2])
        xw = torch.stack([c * x[:, 0] - s * x[:, 1], s * x[:, 0] + c * x[:, 1]], 1)
        arm = xw
        v = body[b, 3:5] + body[b, 5] * torch.stack([-arm[:, 1], arm[:, 0]], 1) + _normal(g, *x.shape, std=0.02)
        parts.append(torch.cat([xw + body[b, :2], v], 1))
    d = dict(params=params, xv=torch.cat(parts).float(), body=body, n=[q.shape[0] for q in parts])
    N = d["xv"].shape[0]
    if kind == "linearize":  # copy i carries the unit tangent of one column of df/dx
        n = d["n"][0]
        cols = torch.randperm(4 * n + 6, generator=g, device="cuda")[:B]
        full = torch.zeros((B, 4 * n + 6), device="cuda", dtype=torch.float64)
        full[torch.arange(min(B, 4 * n + 6), device="cuda"), cols] = 1.0
        d["dxv"] = full[:, :4 * n].reshape(B * n, 4).float()
        d["dbody"] = full[:, 4 * n:].contiguous()
        d["u"] = _uniform(g, 1, 3, lo=-5.0, hi=5.0).repeat(B, 1)
        return d
    K = case["steps"]
    amp = torch.tensor([20.0, 20.0, 2.0], device="cuda", dtype=torch.float64)
    d["u"] = _holds(g, 3 * B, K, max(2.0, K / 3.0), 1.0).reshape(B, 3, K).transpose(1, 2).contiguous() * amp
    d["ns"] = -(-K // case["outer"])
    if kind == "flight" and case["pd"]:
        d["ref"] = _holds(g, B, d["ns"], 4.0, 0.3)
    if kind == "tangent":
        d["dxv"] = (_normal(g, N, 4) * torch.tensor([1e-3, 1e-3, 1e-2, 1e-2], device="cuda", dtype=torch.float64)).float()
        d["dbody"] = _normal(g, 1, 6) * torch.tensor([1e-3] * 3 + [1e-2] * 3, device="cuda", dtype=torch.float64)
        d["du"] = _normal(g, 1, K, 3) * amp
    if kind == "adjoint":
        d["ybar"], d["xvbar"], d["bodybar"] = _normal(g, 1, d["ns"], 11), _normal(g, N, 4).float(), _normal(g, 1, 6)
    return d


def _lowpass(u, a):
    """y_k = a y_{k-1} + (1 - a) u_k along dim 1, by doubling."""
    y, w, s = u * (1.0 - a), a, 1
    while s < y.shape[1] and w > 1e-12:
        y = torch.cat([y[:, :s], y[:, s:] + w * y[:, :-s]], 1)
        w, s = w * w, 2 * s
    return y


def _stable(g, n, rho):
    """A random n x n matrix of spectral radius rho (damped rotations in a random basis)."""
    q, _ = torch.linalg.qr(_normal(g, n, n))
    m = torch.zeros((n, n), device="cuda", dtype=torch.float64)
    i = 0
    while i < n:
        r = rho * float(_uniform(g, 1, lo=0.7, hi=1.0))
        t = float(_uniform(g, 1, lo=0.0, hi=0.5))
        if i + 1 < n:
            m[i:i + 2, i:i + 2] = r * torch.tensor([[math.cos(t), -math.sin(t)], [math.sin(t), math.cos(t)]])
        else:
            m[i, i] = r
        i += 2
    return q @ m @ q.T


_BODY = dict(m=500.0, J=50.0, Ts=0.002, n_sub=10, ctrl_omega=0.2 * math.pi, ctrl_xi=0.7)


def _lpv_inputs(case, seed):
    g = _gen(seed)
    n_y, n_p, n_x = case["n_y"], case["n_p"], case["na"] * case["n_y"]
    blocks = []
    for i in range(1 + n_p):
        M = torch.zeros((n_x + n_y, n_x + 3), device="cuda", dtype=torch.float64)
        s = 1.0 if i == 0 else 0.05
        M[:n_x, :n_x] = _stable(g, n_x, 0.98) if i == 0 else _normal(g, n_x, n_x, std=0.002)
        M[:n_x, n_x:] = _normal(g, n_x, 3, std=0.1 * s)
        M[n_x:, :n_x] = _normal(g, n_y, n_x, std=0.3 * s)
        blocks.append(M)
    d = dict(W=torch.stack(blocks).float())
    s_u, s_y = [11.5, 11.5, 1.2], [9.0, 9.0, 1.0, 0.02][:n_y]
    pm, ps, plo, phi = [0.5, 0.0], [0.17, 0.05], [0.2, -0.2], [0.8, 0.2]
    d["scales"] = np.array(s_u + s_y + pm[:n_p] + ps[:n_p] + plo[:n_p] + phi[:n_p], dtype=np.float32)
    T = case["T"]
    if case["kind"] == "lpv_loop":
        n = case["runs"]
        d["F"] = torch.stack([_holds(g, n, T, 100.0, 20.0) for _ in range(2)], 2)
        d["tau"], d["ref"] = _holds(g, n, T, 100.0, 2.0), _holds(g, n, T, 1000.0, 0.3)
        d["fill"] = _uniform(g, n, lo=0.2, hi=0.8)
        return d
    n = case["n_traj"]
    u = torch.stack([_holds(g, n, T, 100.0, a) for a in (20.0, 20.0, 2.0)], 2)
    d["u"] = u.float()
    fill = _uniform(g, n, 1, lo=0.2, hi=0.8).expand(n, T)
    rate = _lowpass(u[:, :, 2], 0.99) * 0.05
    d["p"] = torch.stack([fill, rate], 2)[:, :, :n_p].float().contiguous()
    if case["kind"] == "lpv_gradient":
        y = torch.stack([_lowpass(u[:, :, i % 3], 0.9 + 0.02 * i) for i in range(n_y)], 2)
        rms = y.square().mean((0, 1)).sqrt() + 1e-9
        d["y"] = ((y / rms + _normal(g, n, T, n_y, std=0.1)) * torch.tensor(s_y, device="cuda")).float()
    return d


_SLPV = dict(Ts=0.05, J=133.84, omega=0.2 * math.pi, xi=0.7, sigma2=1e-4)


def _slpv_inputs(case, seed):
    """A velocity-level model: slowly decaying velocities driven by the input,
    a scheduled part of a few per cent, and the network's usual start."""
    g = _gen(seed)
    nx = case["nx"]
    nz = nx + 3
    M0, M1 = (torch.zeros((nz, nz), device="cuda", dtype=torch.float64) for _ in range(2))
    M0[:nx, :nx] = torch.diag(_uniform(g, nx, lo=0.9, hi=0.99)) + _normal(g, nx, nx, std=0.01)
    M0[:nx, nx:] = _normal(g, nx, 3, std=0.01)
    M0[nx:, :nx] = _normal(g, 3, nx, std=0.1)
    for i in range(min(nx, 3)):  # each velocity answers its own input
        M0[i, nx + i] += 0.05
        M0[nx + i, i] += 1.0
    M1[:nx, nx:] = _normal(g, nx, 3, std=0.01)
    M1[nx:, :nx] = _normal(g, 3, nx, std=0.02)
    net = []
    for fan_in, fan_out in ((nz, 4), (4, 4), (4, 1)):
        lim = math.sqrt(6.0 / (fan_in + fan_out))
        net += [_uniform(g, fan_out * fan_in, lo=-lim, hi=lim), _normal(g, fan_out, std=0.1)]
    d = dict(theta=torch.cat([M0.reshape(-1), M1.reshape(-1)] + net).float())
    d["scales"] = np.array([11.5, 11.5, 1.2, 0.02, 0.02, 0.01], dtype=np.float32)
    T = case["T"]
    if case["kind"] == "slpv_loop":
        n = case["runs"]
        d["F"] = torch.stack([_holds(g, n, T, 6.0, 20.0) for _ in range(2)], 2)
        d["tau"], d["ref"] = _holds(g, n, T, 6.0, 2.0), _holds(g, n, T, 40.0, 0.3)
        return d
    n = case["n_traj"]
    u = torch.stack([_holds(g, n, T, 6.0, a) for a in (20.0, 20.0, 2.0)], 2)
    y = _lowpass(u, 0.97)
    y = y / (y.square().mean((0, 1)).sqrt() + 1e-9) + _normal(g, n, T, 3, std=0.05)
    d["u"], d["y"] = u.float(), (y * torch.tensor(d["scales"][3:], device="cuda")).float()
    return d


def _inputs(case, seed):
    kind = case["kind"]
    return _lpv_inputs(case, seed) if kind.startswith("lpv") else \
        _slpv_inputs(case, seed) if kind.startswith("slpv") else _sph_inputs(case, seed)


def prepare(case, seed):
    d = _inputs(case, seed)
    kind = case["kind"]
    if kind.startswith("lpv"):
        from paper_2604_12505_gb300 import lpv
        m = lpv.Model(dict(n_x=case["na"] * case["n_y"], n_u=3, n_y=case["n_y"], n_p=case["n_p"], na=case["na"]))
        m.set_params(d["W"].cpu().numpy(), d["scales"])
        d["model"] = m
    elif kind.startswith("slpv"):
        from paper_2604_12505_gb300 import slpv
        m = slpv.VelocityModel(case["nx"], sigma2=_SLPV["sigma2"])
        m.set_params(d["theta"].cpu().numpy(), d["scales"])
        d["model"] = m
    else:
        from paper_2604_12505_gb300.sph import Sim
        d["sim"] = Sim(d["params"])
        d["sim"].set_state(d["xv"], d["body"])
    return dict(d, case=case)


def run(s):
    case = s["case"]
    kind = case["kind"]
    if kind == "flight":  # from the same rest state, as manoeuvre after manoeuvre is flown
        sim = s["sim"]
        sim.set_state(s["xv"], s["body"])
        ctrl = dict(omega=0.2 * math.pi, xi=0.7) if case["pd"] else None
        y = sim.step(case["steps"], u=s["u"], ctrl=ctrl, theta_ref=s.get("ref"))
        xv, body = sim.state()
        return dict(y=y, xv=xv, body=body)
    if kind == "linearize":
        dacc, dbody = s["sim"].eval_jvp(s["dxv"], s["dbody"], u=s["u"])
        return dict(dacc=dacc, dbody=dbody)
    if kind == "tangent":
        s["sim"].set_state(s["xv"], s["body"])
        y, dy, dxv, dbody = s["sim"].jvp(case["steps"], u=s["u"], du=s["du"], dxv0=s["dxv"], dbody0=s["dbody"])
        return dict(y=y, dy=dy, dxv=dxv, dbody=dbody)
    if kind == "adjoint":
        s["sim"].set_state(s["xv"], s["body"])
        xb, bb, ub = s["sim"].vjp(case["steps"], u=s["u"], ybar=s["ybar"], xvbar=s["xvbar"], bodybar=s["bodybar"],
                                  checkpoint_every=case["every"])
        return dict(xvbar=xb, bodybar=bb, ubar=ub)
    m = s["model"]
    if kind == "lpv_gradient":
        loss, grad = m.loss_grad(s["u"], s["y"], s["p"])
        return dict(loss=loss, grad=grad)
    if kind == "lpv_predict":
        return m.predict(s["u"], s["p"])
    if kind == "lpv_loop":
        return m.simulate(s["F"], s["tau"], s["ref"], s["fill"], _BODY)
    if kind == "slpv_gradient":
        loss, grad = m.loss_grad(s["u"], s["y"])
        return dict(loss=loss, grad=grad)
    return m.simulate(s["F"], s["tau"], s["ref"], _SLPV["Ts"], _SLPV["J"], _SLPV["omega"], _SLPV["xi"])


def work(case):
    kind = case["kind"]
    if kind in ("flight", "linearize", "tangent", "adjoint"):
        fill = 0.5 * (case["fill"] + case.get("fill_hi", case["fill"]))
        dx = math.sqrt(case["dx"] * case.get("dx_hi", case["dx"]))
        N, K = fill * math.pi * (case["R"] / dx) ** 2 * case.get("tanks", 1), case.get("steps", 1)
        nb = math.pi * (2.6 if case["family"] == "BASE" else 2 * 9.42 / 6.0) ** 2  # neighbours within 2h
        # per particle and step: the density (22) and force (35) terms of each
        # neighbour and 27 of the particle; the derivatives about as much again
        # per pass (tangent) or twice as much (adjoint)
        flops = N * K * (57 * nb + 27) * {"flight": 1, "linearize": 2, "tangent": 2, "adjoint": 3}[kind]
        state = N * {"flight": 32, "linearize": 16 + 16 + 8, "tangent": 64, "adjoint": 48}[kind]
        return dict(bytes=state + 24.0 * K * case.get("tanks", 1), flops=flops)
    if kind.startswith("lpv"):
        nx, ny, kt = case["na"] * case["n_y"], case["n_y"], 1 + case["n_p"]
        rows = case.get("n_traj", case.get("runs")) * case["T"]
        mul = 2 * kt * ((nx + ny) * (nx + 3) - 3 * ny)
        if kind == "lpv_loop":
            return dict(bytes=rows * 80.0, flops=rows * (mul + 60.0))
        if kind == "lpv_predict":
            return dict(bytes=rows * 4.0 * (3 + ny + case["n_p"]), flops=rows * float(mul))
        return dict(bytes=rows * 4.0 * (3 + ny + case["n_p"]), flops=rows * 3.0 * mul)
    nx = case["nx"]
    rows = case.get("n_traj", case.get("runs")) * case["T"]
    net = 2 * (4 * (nx + 3) + 16 + 4) + 8 * 10
    mul = 4 * ((nx + 3) ** 2 - 9)
    if kind == "slpv_loop":
        return dict(bytes=rows * 56.0, flops=rows * (mul + 2.0 * net))
    return dict(bytes=rows * 24.0, flops=rows * 3.0 * (mul + net))


# ---------------------------------------------------------------------------
# the same in 64 bits by plain torch
# ---------------------------------------------------------------------------
def _pairs(xi, xj, reach):
    """Indices (i, j) of all pairs closer than reach, found on a grid of that side."""
    lo = torch.minimum(xi.min(0).values, xj.min(0).values) - reach
    ci, cj = (torch.floor((x - lo) / reach).to(torch.int64) for x in (xi, xj))
    w = int(torch.maximum(ci.max(), cj.max())) + 3
    key, order = torch.sort(cj[:, 1] * w + cj[:, 0])
    out = []
    for dy in (-1, 0, 1):
        c = (ci[:, 1] + dy) * w + ci[:, 0]
        a, b = torch.searchsorted(key, c - 1), torch.searchsorted(key, c + 1, right=True)
        n = b - a
        i = torch.repeat_interleave(torch.arange(len(xi), device=xi.device), n)
        j = order[torch.arange(len(i), device=xi.device) - torch.repeat_interleave(n.cumsum(0) - n, n) + a[i]]
        keep = (xi[i] - xj[j]).square().sum(1) < reach * reach
        out.append(torch.stack([i[keep], j[keep]]))
    return torch.cat(out, 1)


def _sum_at(n, i, v):
    return torch.zeros((n,) + tuple(v.shape[1:]), device=v.device, dtype=v.dtype).index_add(0, i, v)


def _dynamics(p, gB, x, v, body):
    """Accelerations of the fluid and the fluid's force and torque on the body (Algorithm 1)."""
    h, n = p["h_over_dx"] * p["dx"], len(x)
    m, sigma = p["rho0"] * p["dx"] ** 2, 5.0 / (14.0 * math.pi)
    c, s, om = torch.cos(body[2]), torch.sin(body[2]), body[5]
    arm = torch.stack([c * gB[:, 0] - s * gB[:, 1], s * gB[:, 0] + c * gB[:, 1]], 1)
    gx, gv = body[:2] + arm, body[3:5] + om * torch.stack([-arm[:, 1], arm[:, 0]], 1)
    i, j = _pairs(x.detach(), x.detach(), 2 * h)
    off = i != j
    i, j = i[off], j[off]
    a, g = _pairs(x.detach(), gx.detach(), 2 * h)
    d, e = x[i] - x[j], x[a] - gx[g]
    r, re = d.square().sum(1).sqrt(), e.square().sum(1).sqrt()

    def kernel(r):
        q = r / h
        return sigma / h ** 2 * ((2 - q) ** 3 - 4 * torch.clamp(1 - q, min=0) ** 3)

    rho = m * (_sum_at(n, i, kernel(r)) + 4 * sigma / h ** 2 + p["gamma1"] * _sum_at(n, a, kernel(re)))
    pr = p["k"] * (rho - p["rho0"]) / rho ** 2
    q = r / h
    G = sigma / h ** 3 * (-3 * (2 - q) ** 2 + 12 * torch.clamp(1 - q, min=0) ** 2) / r
    vr = ((v[i] - v[j]) * d).sum(1)
    visc = 2 * p["alpha"] * h * vr / ((rho[i] + rho[j]) * (r ** 2 + p["eps"] * h * h))
    acc = _sum_at(n, i, (m * (visc - pr[i] - pr[j]) * G)[:, None] * d)
    near = re.detach() < h
    a, g, e, re = a[near], g[near], e[near], re[near]
    Gs = -30.0 / (math.pi * h ** 5) * (h - re) ** 2 / re
    qg = torch.clamp(pr, min=0) if p["ghost_pressure_clamp"] else pr
    vg = ((v[a] - gv[g]) * e).sum(1)
    f = (p["ghost_pressure_sign"] * 2 * m * m * qg[a] * Gs
         + m * m * 2 * p["beta"] * torch.clamp(vg, max=0) / (2 * rho[a] * (re ** 2 + p["eps"] * h * h)) * Gs)
    fe = f[:, None] * e
    grav = torch.tensor([p["grav_x"], p["grav_y"]], device=x.device, dtype=x.dtype)
    acc = acc + _sum_at(n, a, fe) / m + grav
    return acc, -fe.sum(0), -(arm[g, 0] * fe[:, 1] - arm[g, 1] * fe[:, 0]).sum()


def _rollout(p, gB, x, v, body, u, outer, ref=None):
    """Steps x, v, body through u [K, 3]: samples and the final state."""
    y, tau_c, dt = [], 0.0, p["dt"]
    M = torch.tensor([p["m_body"], p["m_body"], p["J_body"]], device=x.device, dtype=x.dtype)
    for k in range(len(u)):
        acc, F, T = _dynamics(p, gB, x, v, body)
        FT = torch.cat([F, T[None]])
        if k % outer == 0:
            y.append(torch.cat([body, FT, x.mean(0)]))
            if ref is not None:
                w = 0.2 * math.pi
                tau_c = p["J_body"] * w * w * (ref[k // outer] - body[2]) - 2 * 0.7 * p["J_body"] * w * body[5]
        uk = u[k] + torch.tensor([0.0, 0.0, 1.0], device=x.device, dtype=x.dtype) * tau_c
        v = v + dt * acc
        x = x + dt * v
        bv = body[3:] + dt * (FT + uk) / M
        body = torch.cat([body[:3] + dt * bv, bv])
    return torch.stack(y), torch.cat([x, v], 1), body


def _exact_sph(case, d):
    kind, o = case["kind"], 0
    xv = d["xv"].double()
    if kind == "flight":
        out = []
        for b, p in enumerate(d["params"]):
            s, o = xv[o:o + d["n"][b]], o + d["n"][b]
            gB = torch.tensor(_ghosts(p), device="cuda")
            ref = d["ref"][b] if "ref" in d else None
            out.append(_rollout(p, gB, s[:, :2], s[:, 2:], d["body"][b], d["u"][b], case["outer"], ref))
        return dict(y=torch.stack([q[0] for q in out]), xv=torch.cat([q[1] for q in out]),
                    body=torch.stack([q[2] for q in out]))
    p, n = d["params"][0], d["n"][0]
    gB = torch.tensor(_ghosts(p), device="cuda")
    x, v, body, u = xv[:n, :2], xv[:n, 2:], d["body"][0], d["u"][0]
    import torch.autograd.forward_ad as fwd
    if kind == "linearize":
        M = torch.tensor([p["m_body"], p["m_body"], p["J_body"]], device="cuda", dtype=torch.float64)
        dacc, dbody = [], []
        for t, db in zip(d["dxv"].double().reshape(-1, n, 4), d["dbody"]):
            with fwd.dual_level():
                acc, F, T = _dynamics(p, gB, fwd.make_dual(x, t[:, :2].contiguous()),
                                      fwd.make_dual(v, t[:, 2:].contiguous()), fwd.make_dual(body, db.contiguous()))
                ta, tF, tT = (fwd.unpack_dual(q).tangent for q in (acc, F, T))
                zero = torch.zeros(3, device="cuda", dtype=torch.float64)
                FT = zero if tF is None else torch.cat([tF, tT.reshape(1)])
                dacc.append(torch.zeros_like(x) if ta is None else ta.clone())
                dbody.append(torch.cat([FT, FT / M]))
        return dict(dacc=torch.cat(dacc), dbody=torch.stack(dbody))
    if kind == "tangent":
        t = d["dxv"].double()
        with fwd.dual_level():
            out = _rollout(p, gB, fwd.make_dual(x, t[:, :2].contiguous()), fwd.make_dual(v, t[:, 2:].contiguous()),
                           fwd.make_dual(body, d["dbody"][0]), fwd.make_dual(u, d["du"][0]), case["outer"])
            (y, dy), (_, dxv), (_, dbody) = (fwd.unpack_dual(q) for q in out)
            return dict(y=y[None].clone(), dy=dy[None].clone(), dxv=dxv.clone(), dbody=dbody[None].clone())
    leaves = [q.clone().requires_grad_(True) for q in (x, v, body, u)]
    y, xvK, bodyK = _rollout(p, gB, *leaves, case["outer"])
    gx, gv, gb, gu = torch.autograd.grad([y, xvK, bodyK], leaves,
                                         [d["ybar"][0], d["xvbar"].double(), d["bodybar"][0]])
    return dict(xvbar=torch.cat([gx, gv], 1), bodybar=gb[None], ubar=gu[None])


def _exact_lpv(case, d):
    nx, n_p, n_y = case["na"] * case["n_y"], case["n_p"], case["n_y"]
    Wm = d["W"].double()
    Wm[:, nx:, nx:] = 0.0
    sc = torch.tensor(d["scales"], device="cuda").double()
    su, sy, (pm, ps, lo, hi) = sc[:3], sc[3:3 + n_y], sc[3 + n_y:].reshape(4, n_p)
    grad = case["kind"] == "lpv_gradient"
    if grad:
        Wm.requires_grad_(True)
    Wf = Wm.permute(1, 0, 2).reshape(nx + n_y, -1).T  # features [z, p_1 z, ...]

    def step(x, u, p):
        z = torch.cat([x, u / su], 1)
        w = torch.cat([z] + [z * ((p[:, i:i + 1] - pm[i]) / ps[i]) for i in range(n_p)], 1)
        o = w @ Wf
        return o[:, :nx], o[:, nx:]

    if case["kind"] == "lpv_loop":
        n, b = case["runs"], _BODY
        x = torch.zeros((n, nx), device="cuda", dtype=torch.float64)
        r, th = torch.zeros((n, 2), device="cuda", dtype=torch.float64), torch.zeros(n, device="cuda", dtype=torch.float64)
        v, w = torch.zeros_like(r), torch.zeros_like(th)
        out = torch.empty((n, case["T"], 6), device="cuda", dtype=torch.float64)
        dt, wn = b["Ts"] / b["n_sub"], b["ctrl_omega"]
        for k in range(case["T"]):
            out[:, k] = torch.cat([r, th[:, None], v, w[:, None]], 1)
            tau = d["tau"][:, k] + b["J"] * wn * wn * (d["ref"][:, k] - th) - 2 * b["ctrl_xi"] * b["J"] * wn * w
            u = torch.cat([d["F"][:, k], tau[:, None]], 1)
            p = torch.stack([d["fill"], w], 1)[:, :n_p]
            x, y = step(x, u, torch.minimum(torch.maximum(p, lo), hi))
            load = u + y[:, :3] * sy[:3]
            for _ in range(b["n_sub"]):
                v, w = v + dt * load[:, :2] / b["m"], w + dt * load[:, 2] / b["J"]
                r, th = r + dt * v, th + dt * w
        return out
    u, p = d["u"].double(), d["p"].double()
    x, ys = torch.zeros((case["n_traj"], nx), device="cuda", dtype=torch.float64), []
    for k in range(case["T"]):
        x, y = step(x, u[:, k], p[:, k])
        ys.append(y)
    y = torch.stack(ys, 1)
    if not grad:
        return y * sy
    loss = (d["y"].double() / sy - y).square().sum(2).mean() + 0.5e-4 * Wm.square().sum()
    (gw,) = torch.autograd.grad(loss, Wm)
    gw = gw.clone()
    gw[:, nx:, nx:] = 0.0
    return dict(loss=float(loss), grad=gw.cpu().numpy())


def _exact_slpv(case, d):
    nx = case["nx"]
    nz, th = nx + 3, d["theta"].double()
    nm = nz * nz
    mask = torch.ones_like(th)
    for o in (0, nm):
        mask[o:o + nm].view(nz, nz)[nx:, nx:] = 0.0
    th = th * mask
    sc = torch.tensor(d["scales"], device="cuda").double()
    su, sy = sc[:3], sc[3:]
    grad = case["kind"] == "slpv_gradient"
    if grad:
        th.requires_grad_(True)
    M0, M1, W1, b1, W2, b2, w3, b3 = torch.split(th, [nm, nm, 4 * nz, 4, 16, 4, 4, 1])
    M0, M1, W1, W2 = M0.view(nz, nz).T, M1.view(nz, nz).T, W1.view(4, nz).T, W2.view(4, 4).T

    def sched(z):
        return (torch.tanh(torch.tanh(z @ W1 + b1) @ W2 + b2) @ w3 + b3)[:, None]

    if grad:
        u, yd = d["u"].double() / su, d["y"].double() / sy
        x, e2 = torch.zeros((case["n_traj"], nx), device="cuda", dtype=torch.float64), 0.0
        for k in range(case["T"]):
            z = torch.cat([x, u[:, k]], 1)
            o = z @ M0 + sched(z) * (z @ M1)
            x, e2 = o[:, :nx], e2 + (o[:, nx:] - yd[:, k]).square().sum()
        loss = e2 / (case["n_traj"] * case["T"]) + 0.5 * _SLPV["sigma2"] * th.square().sum()
        (gt,) = torch.autograd.grad(loss, th)
        return dict(loss=loss.detach()[None], grad=gt * mask)
    n, kp, kd = case["runs"], _SLPV["J"] * _SLPV["omega"] ** 2, 2 * _SLPV["xi"] * _SLPV["J"] * _SLPV["omega"]
    x, e, un = (torch.zeros((n, q), device="cuda", dtype=torch.float64) for q in (nx, 3, 3))
    out = torch.empty((n, case["T"], 6), device="cuda", dtype=torch.float64)
    for k in range(case["T"]):
        z = torch.cat([x, un], 1)
        wd = (z @ M0 + sched(z) * (z @ M1))[:, nx + 2] * sy[2]
        tc = kp * (d["ref"][:, k] - e[:, 2]) - kd * wd
        un = torch.cat([d["F"][:, k], (d["tau"][:, k] + tc)[:, None]], 1) / su
        z = torch.cat([x, un], 1)
        o = z @ M0 + sched(z) * (z @ M1)
        v = o[:, nx:] * sy
        out[:, k] = torch.cat([e, v], 1)
        x, e = o[:, :nx], e + _SLPV["Ts"] * v
    return out


def exact(case, seed):
    d = _inputs(case, seed)
    kind = case["kind"]
    return _exact_lpv(case, d) if kind.startswith("lpv") else \
        _exact_slpv(case, d) if kind.startswith("slpv") else _exact_sph(case, d)
