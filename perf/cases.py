"""The calls this library is used for, at the sizes its workloads have.

Every case is one pass through a public entry point of
paper_2605_14103_gb300.zbus: a batched feeder solve in each of its forms, the
batched solve of several feeders, the serving loop, the differentiable solve
with its gradient, and the Newton-Raphson solve of a transmission grid.  A
case's network, loads and grid come from its seed alone (a feeder with
laterals is one feeder, its loads come from the seed).
"""
from __future__ import annotations

import math

import numpy as np
import torch

from paper_2605_14103_gb300 import feeders, grids, zbus

TOL = 1e-8            # stop tolerance of the feeder workloads (pu)
MAX_ITER = 50
GRID_TOL = 1e-10      # of the grid workloads


def listed():
    return [
        # one small feeder, a handful of scenarios: an operator's what-if
        # question, answered one call at a time (latency)
        _solve("feeder13_b8_fp64", 13, 8, "fp64", 0.0, 0.8, 1.2),
        # the plain FP64 method (the default form) on a town feeder's daily
        # profiles, and on a large feeder with a planning study's batch
        _solve("feeder128_b4096_fp64", 128, 4096, "fp64", 0.3, 0.5, 1.5),
        _solve("feeder1024_b1000_fp64", 1024, 1000, "fp64", 0.3, 0.8, 1.2),
        # the tensor-core form on the same feeders: Monte-Carlo batches
        _solve("feeder128_b4096_fp16", 128, 4096, "fp16_scaled", 0.3, 0.5, 1.5),
        _solve("feeder1024_b16384_fp16", 1024, 16384, "fp16_scaled", 0.3, 0.8, 1.2),
        # the split-BF16 form on a feeder with single- and two-phase laterals
        _solve("partial1024_b5001_bf16x2", 1024, 5001, "bf16x2", 0.3, 0.8, 1.2, lateral=0.3),
        # the sweep form of radial feeders
        _solve("feeder1024_b16384_tree", 1024, 16384, "tree", 0.3, 0.8, 1.2),
        # feeders of uneven size in one call: a utility's whole service area
        {"name": "batch16_fp16", "kind": "batch", "feeders": 16, "buses_lo": 50,
         "buses_hi": 800, "b_lo": 32, "b_hi": 2048, "precision": "fp16_scaled"},
        # requests over a pool of feeders, all waiting when the loop starts
        {"name": "serve_fp16", "kind": "serve", "feeders": 8, "buses_lo": 100,
         "buses_hi": 1000, "b_lo": 1, "b_hi": 1024, "requests": 20,
         "precision": "fp16_scaled"},
        # a learning step: the solve and the gradient of a loss of its voltages
        {"name": "gradient128_b4096_fp64", "kind": "gradient", "buses": 128, "b": 4096,
         "adjoint": "fp64", "delta": 0.3, "lo": 0.5, "hi": 1.5},
        # transmission grids, contingency and load batches
        {"name": "grid2224_b1000_fp64", "kind": "grid", "buses": 2224, "b": 1000,
         "precision": "fp64"},
        {"name": "grid118_b1000_mixed", "kind": "grid", "buses": 118, "b": 1000,
         "precision": "mixed"},
    ]


def _solve(name, buses, b, precision, delta, lo, hi, lateral=0.0):
    return {"name": name, "kind": "solve", "buses": buses, "b": b, "precision": precision,
            "delta": delta, "lo": lo, "hi": hi, "lateral": lateral}


def _log_int(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def draw(rng):
    kind = rng.choice(["solve", "solve", "solve", "solve", "batch", "serve", "gradient", "grid"])
    if kind == "solve":
        precision = rng.choice(["fp64", "fp64", "fp16_scaled", "bf16x2", "tree"])
        buses = _log_int(rng, 13, 1024)
        n = 3 * (buses - 1)
        cap = 1000 * 3069 ** 2 // (n * n) if precision == "fp64" else 16384 * 3069 // n
        b = _log_int(rng, 1, min(16384, cap))
        c = _solve("", buses, b, precision, rng.choice([0.0, 0.3]), *rng.choice(
            [(0.8, 1.2), (0.5, 1.5)]), lateral=rng.choice([0.0, 0.0, 0.3]))
    elif kind == "batch":
        c = {"kind": kind, "feeders": rng.randint(2, 16), "buses_lo": 50,
             "buses_hi": rng.randint(100, 800), "b_lo": 32, "b_hi": rng.randint(64, 2048),
             "precision": rng.choice(["fp16_scaled", "bf16x2", "tree"])}
    elif kind == "serve":
        c = {"kind": kind, "feeders": rng.randint(2, 8), "buses_lo": 100,
             "buses_hi": rng.randint(120, 1000), "b_lo": 1, "b_hi": rng.randint(16, 1024),
             "requests": rng.randint(5, 20), "precision": rng.choice(["fp16_scaled", "tree"])}
    elif kind == "gradient":
        adjoint = rng.choice(["fp64", "tree"])
        buses = _log_int(rng, 13, 1024)
        n = 3 * (buses - 1)
        cap = 4096 * 381 ** 2 // (n * n)
        c = {"kind": kind, "buses": buses, "b": _log_int(rng, 1, max(1, min(4096, cap))),
             "adjoint": adjoint, "delta": rng.choice([0.0, 0.3]), "lo": 0.8, "hi": 1.2}
    else:
        c = {"kind": kind, "buses": _log_int(rng, 14, 2224), "b": _log_int(rng, 1, 1000),
             "precision": rng.choice(["fp64", "mixed"])}
    c.pop("name", None)
    return c


# -- inputs ------------------------------------------------------------------

def _feeder(buses, seed, delta, hi, lateral=0.0):
    if lateral > 0:   # one feeder, so that its phases do not change with the loads' seed
        return feeders.make_partial_feeder(buses, 303, lateral_frac=lateral, delta_frac=delta,
                                           mult_hi=hi)
    return feeders.make_feeder(buses, seed, delta_frac=delta, mult_hi=hi)


def _loads(f, b, lo, hi, seed):
    """(S_wye, S_delta) on the GPU: one multiplier per scenario and load bus."""
    g = torch.Generator(device="cuda")
    g.manual_seed(seed)
    mult = torch.rand((b, f.N - 1, 1), generator=g, dtype=torch.float64, device="cuda")
    mult = mult * (hi - lo) + lo
    delta = f.is_delta[:, None]
    out = []
    for base in (np.where(delta, 0.0, f.base_S), np.where(delta, f.base_S, 0.0)):
        s = mult * torch.from_numpy(base).cuda()
        if isinstance(f, feeders.PhasedFeeder):
            s = s[:, torch.from_numpy(f.phases[1:]).cuda()]
        out.append(s.reshape(b, f.n).contiguous())
    return out


def _pool(case, seed):
    """The feeders of a batch or a pool, sizes spread over the case's range."""
    sizes = np.linspace(case["buses_lo"], case["buses_hi"], case["feeders"]).astype(int)
    return [feeders.make_feeder(int(s), seed + 2 * k, delta_frac=0.4, mult_hi=1.2)
            for k, s in enumerate(sizes)]


def _counts(case, m):
    """m scenario counts spread over the case's range (their logarithm)."""
    c = np.exp(np.linspace(math.log(case["b_lo"]), math.log(case["b_hi"]), m))
    c = np.rint(c).astype(int)
    return [int(c[(5 * k) % m]) if m % 5 else int(c[(7 * k) % m]) for k in range(m)]


def _inputs(case, seed):
    """[(feeder, S_wye, S_delta)] of a feeder case (one per feeder or request)."""
    if case["kind"] == "solve":
        f = _feeder(case["buses"], seed, case["delta"], case["hi"], case["lateral"])
        return [(0, f, *_loads(f, case["b"], case["lo"], case["hi"], seed + 1))]
    if case["kind"] == "gradient":
        f = _feeder(case["buses"], seed, case["delta"], case["hi"])
        return [(0, f, *_loads(f, case["b"], case["lo"], case["hi"], seed + 1))]
    fs = _pool(case, seed)
    m = case["feeders"] if case["kind"] == "batch" else case["requests"]
    return [(i % len(fs), fs[i % len(fs)],
             *_loads(fs[i % len(fs)], b, 0.8, 1.2, seed + 101 + i))
            for i, b in enumerate(_counts(case, m))]


def _grid(case, seed):
    g = grids.make_grid(case["buses"], seed)
    return g, *grids.make_injections(g, case["b"])


def _upstream(shape, seed):
    g = torch.Generator(device="cuda")
    g.manual_seed(seed + 2)
    return torch.randn(shape, generator=g, dtype=torch.complex128, device="cuda")


def prepare(case, seed):
    kind = case["kind"]
    if kind == "grid":
        g, P, Q = _grid(case, seed)
        return {"case": case, "net": zbus.NrNetwork.from_grid(g),
                "P": torch.from_numpy(P).cuda(), "Q": torch.from_numpy(Q).cuda()}
    items = _inputs(case, seed)
    if kind == "serve":
        nets = [zbus.Network.from_feeder(f) for f in _pool(case, seed)]
        return {"case": case, "nets": nets,
                "requests": [{"feeder": k, "S_wye": sw, "S_delta": sd}
                             for k, _, sw, sd in items]}
    nets = [zbus.Network.from_feeder(f) for _, f, _, _ in items]
    state = {"case": case, "nets": nets, "loads": [(sw, sd) for _, _, sw, sd in items]}
    if kind == "gradient":
        for s in state["loads"][0]:
            s.requires_grad_(True)
        state["G"] = _upstream((case["b"], items[0][1].n), seed)
    return state


def run(state):
    case = state["case"]
    kind = case["kind"]
    if kind == "solve":
        sw, sd = state["loads"][0]
        return state["nets"][0].solve(sw, sd, tol=TOL, max_iter=MAX_ITER,
                                      precision=case["precision"])
    if kind == "batch":
        return zbus.solve_batched(state["nets"], state["loads"], tol=TOL, max_iter=MAX_ITER,
                                  precision=case["precision"])
    if kind == "serve":
        out = zbus.serve(state["nets"], state["requests"], max_slots=1024,
                         precision=case["precision"], tol=TOL, max_iter=MAX_ITER)
        return [(r["V"], r["iters"], r["converged"]) for r in out]
    if kind == "gradient":
        sw, sd = state["loads"][0]
        V, it, cv = zbus.solve_differentiable(state["nets"][0], sw, sd,
                                              adj_precision=case["adjoint"])
        dw, dd = torch.autograd.grad(V, (sw, sd), state["G"])
        return V.detach(), it, cv, dw, dd
    return state["net"].solve(state["P"], state["Q"], tol=GRID_TOL,
                              precision=case["precision"])


# -- what a pass cannot do without -------------------------------------------

SWEEPS = 7            # maps of the feeder workloads from the no-load start
NEWTON_STEPS = 5      # of the grid workloads, with this many Krylov vectors
KRYLOV = 28           # in all their steps together


def work(case):
    """Loads (or injections) in, voltages out, the network's matrix once; the
    dense forms' products with it, 8 n^2 operations a scenario and map, and a
    few hundred a bus for the residual or the currents."""
    kind = case["kind"]
    if kind == "grid":
        N, b = case["buses"], case["b"]
        per = KRYLOV * (8 * 4 * N + 14 * N + 2 * 18 * N + 8 * 5.6 * 2 * N)
        return {"bytes": b * N * 32 + 200 * N, "flops": b * per}
    if kind == "solve":
        shapes = [(case["buses"], case["b"])]
    elif kind == "gradient":
        shapes = [(case["buses"], case["b"])]
    else:
        m = case["feeders"] if kind == "batch" else case["requests"]
        sizes = np.linspace(case["buses_lo"], case["buses_hi"], case["feeders"]).astype(int)
        shapes = [(int(sizes[k % len(sizes)]), b) for k, b in enumerate(_counts(case, m))]
    total = {"bytes": 0, "flops": 0}
    seen = set()
    for buses, b in shapes:
        n = 3 * (buses - 1)
        dense = (case.get("precision") or "fp64") != "tree"
        sweeps = SWEEPS
        if kind == "gradient":
            sweeps = 9 + (11 if case["adjoint"] == "fp64" else 0)
        elem = {"fp64": 16, "bf16x2": 8, "fp16_scaled": 4}.get(case.get("precision"), 16)
        if dense and buses not in seen:
            total["bytes"] += elem * n * n
        seen.add(buses)
        total["bytes"] += b * n * 48 + (b * n * 64 if kind == "gradient" else 0)
        total["flops"] += b * sweeps * ((8 * n * n if dense else 0) + 100 * n)
    return total


# -- the same in 64 bits -----------------------------------------------------

def _reduced(f):
    """(Z, w, slot of the next phase at the same bus or -1) of a feeder."""
    Y = torch.zeros((f.n_total, f.n_total), dtype=torch.complex128)
    Y.index_put_((torch.from_numpy(f.Y_row.astype(np.int64)),
                  torch.from_numpy(f.Y_col.astype(np.int64))),
                 torch.from_numpy(f.Y_val), accumulate=True)
    Y = Y.cuda()
    Z = torch.linalg.inv(Y[3:, 3:])
    w = -(Z @ (Y[3:, :3] @ torch.from_numpy(f.v_slack).cuda()))
    bp = getattr(f, "bus_phase", None)
    bp = np.arange(f.n_total) if bp is None else np.asarray(bp)
    where = {int(g): j for j, g in enumerate(bp[3:])}
    nxt = [where.get(3 * (int(g) // 3) + (int(g) + 1) % 3, -1) for g in bp[3:]]
    return Z, w, torch.tensor(nxt, device="cuda")


def _quotient(s, v):
    return torch.where(s != 0, (s / torch.where(s != 0, v, 1.0)).conj(), 0.0)


def _currents(v, sw, sd, nxt):
    i = -_quotient(sw, v)
    x = torch.nonzero(nxt >= 0).flatten()
    y = nxt[x]
    br = _quotient(sd[:, x], v[:, x] - v[:, y])
    i.index_add_(1, x, br, alpha=-1)
    i.index_add_(1, y, br)
    return i


def _fixed_point(f, sw, sd, tol):
    """Each scenario's iterate at which its largest step is within tol."""
    Z, w, nxt = _reduced(f)
    V = w.expand(sw.shape[0], -1).clone()
    active = torch.arange(sw.shape[0], device="cuda")
    for _ in range(MAX_ITER):
        v = V[active]
        new = _currents(v, sw[active], sd[active], nxt) @ Z.T + w
        V[active] = new
        active = active[(new - v).abs().amax(1) > tol]
        if not active.numel():
            break
    return V, Z, nxt


def _gradient(f, sw, sd, G):
    """Loads' gradient at the converged voltages: lambda = G + A^T mu,
    mu = Z^T conj(lambda), to convergence."""
    V, Z, nxt = _fixed_point(f, sw, sd, 1e-10)
    x = torch.nonzero(nxt >= 0).flatten()
    y = nxt[x]
    u = V[:, x] - V[:, y]
    cw = torch.where(sw != 0, (sw / V ** 2).conj(), 0.0)
    cd = (sd[:, x] / u ** 2).conj()
    mu = torch.zeros_like(V)
    for _ in range(60):
        lam = G + cw * mu
        t = cd * (mu[:, x] - mu[:, y])
        lam.index_add_(1, x, t)
        lam.index_add_(1, y, t, alpha=-1)
        new = lam.conj() @ Z
        step = (new - mu).abs().max() / new.abs().max()
        mu = new
        if step < 1e-15:
            break
    dd = torch.zeros_like(V)
    dd[:, x] = -(mu[:, x] - mu[:, y]) / u.conj()
    return V, -mu / V.conj(), dd


def _newton(g, P, Q):
    """Newton's method in polar form, dense, all scenarios at once."""
    N, B = g.N, P.shape[0]
    Y = torch.zeros((N, N), dtype=torch.complex128)
    Y.index_put_((torch.from_numpy(g.Y_row.astype(np.int64)),
                  torch.from_numpy(g.Y_col.astype(np.int64))),
                 torch.from_numpy(g.Y_val), accumulate=True)
    Y = Y.cuda()
    bt = torch.from_numpy(g.bus_type).cuda()
    th_set = torch.nonzero(bt != grids.SLACK).flatten()
    q_set = torch.nonzero(bt == grids.PQ).flatten()
    m = torch.from_numpy(g.v_set).cuda().expand(B, -1).clone()
    m[:, q_set] = 1.0
    th = torch.zeros_like(m)
    S = torch.complex(torch.from_numpy(P).cuda(), torch.from_numpy(Q).cuda())
    for _ in range(8):
        e = torch.polar(torch.ones_like(m), th)
        v = m * e
        I = v @ Y.T
        d = v * I.conj() - S
        F = torch.cat([d.real[:, th_set], d.imag[:, q_set]], 1)
        if float(F.abs().max()) <= 1e-12:
            break
        W = v[:, :, None] * Y.conj()
        Jt = -1j * W * v.conj()[:, None, :] + torch.diag_embed(1j * v * I.conj())
        Jm = W * e.conj()[:, None, :] + torch.diag_embed(e * I.conj())
        J = torch.cat([torch.cat([Jt.real[:, th_set][:, :, th_set],
                                  Jm.real[:, th_set][:, :, q_set]], 2),
                       torch.cat([Jt.imag[:, q_set][:, :, th_set],
                                  Jm.imag[:, q_set][:, :, q_set]], 2)], 1)
        dx = torch.linalg.solve(J, -F[:, :, None])[:, :, 0]
        th[:, th_set] += dx[:, :th_set.numel()]
        m[:, q_set] += dx[:, th_set.numel():]
    return torch.polar(m, th)


def exact(case, seed):
    """The plain form's iterate of the same stop rule; of the other forms,
    which reach the fixed point by other iterates, the fixed point; counts and
    flags have no such value."""
    if case["kind"] == "grid":
        if case["b"] * case["buses"] ** 2 > 2e7:
            return None
        g, P, Q = _grid(case, seed)
        return _newton(g, P, Q), None, None, None
    items = _inputs(case, seed)
    if case["kind"] == "gradient":
        _, f, sw, sd = items[0]
        V, dw, dd = _gradient(f, sw, sd, _upstream(sw.shape, seed))
        return V, None, None, dw, dd
    tol = TOL if case["precision"] == "fp64" else 1e-13
    out = [(_fixed_point(f, sw, sd, tol)[0], None, None) for _, f, sw, sd in items]
    return out[0] if case["kind"] == "solve" else out
