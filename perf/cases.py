"""Workloads of the direct N-body library, as a program of its user runs them.

Four kinds, each through the package's public calls only:

* ``eval``       one force evaluation: ``NBody.predict`` to the block time, then ``NBody.evaluate`` of
                 the active particles (all of them, or a list) with the results left on the device;
* ``integrate``  block time steps of one system over one largest step (``run_until``, or ``run_diag`` with
                 energy and angular momentum sampled at both ends), then the state;
* ``ensemble``   many independent systems advanced together over one largest step, then their state;
* ``grad``       a differentiable shared-step trajectory, forward and backward: loss and gradients.

Inputs are seeded Plummer spheres in Henon units, the model of the repository's configurations (equal or
Salpeter masses, eps = 1e-4).  The mixed precision's sums carry FP32 pair terms, good to about 1e-7, so a program
that asks for it keeps them as float32; FP64 and EX results stay float64.  Only the crackle of an integrated state
is kept as float32: it is a difference quotient of the sums over the cube of the step, which costs it five to seven
of their digits.
"""
from __future__ import annotations

import math

import numpy as np
import torch
import torch.utils.checkpoint

import nb_inputs as ni
import paper_1901_08532_gb300 as nb
from paper_1901_08532_gb300 import adjoint

EPS = 1e-4
PRECISION = {"fp64": nb.NB_FP64, "mixed": nb.NB_MIXED, "ex": nb.NB_EX}
#: time of one interaction of each precision, the mixed one's as the unit (only to keep drawn cases affordable)
COST = {"mixed": 1.0, "ex": 9.0, "fp64": 57.0}
MOST = 2.0 ** 38
#: flops of one interaction (i, j), FMA = 2, as the benchmark counts them
FLOPS = 78.0


def _eval(name, prec, n, n_act=0, imf="equal"):
    return {"name": name, "kind": "eval", "prec": prec, "n": n, "n_act": n_act, "imf": imf}


def listed():
    return [
        # The force evaluation with every particle active: each shared step, the start-up of every run and every
        # synchronisation of the block steps.  Smallest: a few hundred particles, where launches count.
        _eval("mixed_all_384", "mixed", 384),
        _eval("mixed_all_20011", "mixed", 20011),
        # The largest: the headline workload (Salpeter masses, all active) at half its particle count.
        _eval("mixed_all_524288", "mixed", 524288, imf="salpeter"),
        _eval("ex_all_16384", "ex", 16384),
        _eval("fp64_all_8191", "fp64", 8191),
        # The ordinary block step: a fraction of the particles is active, against all of them.
        _eval("mixed_65537_act_130", "mixed", 65537, 130),
        _eval("mixed_1048576_act_32768", "mixed", 1048576, 32768, "salpeter"),
        _eval("ex_262144_act_8192", "ex", 262144, 8192, "salpeter"),
        # Whole integrations by block steps over one largest step: the accuracy reference on a small cluster, and
        # extended precision with the diagnostics sampled on the device.
        {"name": "integrate_fp64_1024", "kind": "integrate", "prec": "fp64", "n": 1024, "dt": 2.0 ** -5, "diag": False},
        {"name": "integrate_ex_diag_8192", "kind": "integrate", "prec": "ex", "n": 8192, "dt": 2.0 ** -5, "diag": True},
        # A batch of clusters of different sizes in one launch.
        {"name": "ensemble_ex_32", "kind": "ensemble", "prec": "ex", "systems": 32, "n_lo": 256, "n_hi": 2048,
         "dt": 2.0 ** -6},
        # Gradients of a trajectory with respect to the initial state and the masses.
        {"name": "grad_fp64_4096", "kind": "grad", "n": 4096, "steps": 4},
    ]


def _log_int(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def draw(rng):
    kind = rng.choice(["all", "all", "some", "some", "integrate", "ensemble", "grad"])
    if kind == "integrate":
        prec = rng.choice(["fp64", "ex"])
        return {"kind": kind, "prec": prec, "n": _log_int(rng, 256, 2500 if prec == "fp64" else 8192),
                "dt": 2.0 ** -rng.choice([5, 6]), "diag": rng.random() < 0.5}
    if kind == "ensemble":
        return {"kind": kind, "prec": rng.choice(["fp64", "ex"]), "systems": rng.randint(8, 40), "n_lo": 256,
                "n_hi": _log_int(rng, 400, 2048), "dt": 2.0 ** -6}
    if kind == "grad":
        return {"kind": kind, "n": _log_int(rng, 256, 4500), "steps": rng.randint(1, 4)}
    while True:
        prec = rng.choice(["mixed", "mixed", "ex", "fp64"])
        n = _log_int(rng, 256, 1 << 20)
        n_act = 0 if kind == "all" else max(1, _log_int(rng, max(1, n >> 10), n // 2))
        if COST[prec] * n * (n_act or n) <= MOST / 4:
            return {"kind": "eval", "prec": prec, "n": n, "n_act": n_act, "imf": rng.choice(["equal", "salpeter"])}


def _inputs(case, seed):
    """Particles of an ``eval`` case: m, x, v and the smooth Plummer acceleration and jerk as the known
    derivatives, which the predictor expands and the snap takes as input; the block time; the active list."""
    n = case["n"]
    m, x, v = ni.plummer(n, seed=seed, imf=case["imf"])
    b2 = (3.0 * math.pi / 16.0) ** 2
    r2 = (x * x).sum(axis=1, keepdims=True) + b2
    a = -x * r2 ** -1.5
    j = -v * r2 ** -1.5 + 3.0 * (x * v).sum(axis=1, keepdims=True) * x * r2 ** -2.5
    active = ni.active_subset(n, case["n_act"], seed) if case["n_act"] else None
    return m, x, v, a, j, 2.0 ** -8, active


def _systems(case, seed):
    sizes = ni.ensemble_sizes(case["systems"], 4, case["n_lo"], case["n_hi"])  # the case's own, whatever the seed
    parts = [ni.plummer(int(k), seed=1000 * seed + q) for q, k in enumerate(sizes)]
    return sizes, parts


def prepare(case, seed):
    kind = case["kind"]
    if kind == "eval":
        m, x, v, a, j, t, active = _inputs(case, seed)
        ctx = nb.NBody(m, x, v, EPS, precision=PRECISION[case["prec"]], start_forces=False)
        ctx.set_state({"a": a, "j": j})
        act = None if active is None else torch.from_numpy(active).cuda()
        return {"case": case, "ctx": ctx, "t": t, "active": act}
    if kind == "integrate":
        m, x, v = ni.plummer(case["n"], seed=seed)
        ctx = nb.NBody(m, x, v, EPS, precision=PRECISION[case["prec"]], dt_max=case["dt"])
        return {"case": case, "ctx": ctx, "t": 0.0}
    if kind == "ensemble":
        sizes, parts = _systems(case, seed)
        m, x, v = (np.concatenate([p[q] for p in parts]) for q in range(3))
        ens = nb.Ensemble(sizes, m, x, v, EPS, precision=PRECISION[case["prec"]], dt_max=case["dt"])
        return {"case": case, "ens": ens, "t": 0.0}
    m, x, v = (torch.from_numpy(q).cuda() for q in ni.plummer(case["n"], seed=seed))
    return {"case": case, "m": m, "x": x, "v": v}


def _kept(st):
    """The state as the program keeps it."""
    return dict(st, c=st["c"].astype(np.float32))


def run(state):
    case = state["case"]
    kind = case["kind"]
    if kind == "eval":
        ctx = state["ctx"]
        ctx.predict(state["t"])
        sums = ctx.evaluate(state["active"], out="device")
        return tuple(s.float() for s in sums) if case["prec"] == "mixed" else sums
    if kind == "integrate":
        ctx = state["ctx"]
        state["t"] += case["dt"]
        if case["diag"]:
            _, sample = ctx.run_diag(state["t"], case["dt"])
            return {"state": _kept(ctx.state()), "ekin": sample["ekin"], "epot": sample["epot"], "L": sample["L"]}
        ctx.run_until(state["t"])
        return {"state": _kept(ctx.state())}
    if kind == "ensemble":
        state["t"] += case["dt"]
        state["ens"].run(state["t"])
        return {"state": _kept(state["ens"].state())}
    loss, gx, gv, gm = adjoint.loss_and_grads(state["m"], state["x"], state["v"], GRAD_EPS, GRAD_H, case["steps"])
    return {"loss": loss, "gx": gx, "gv": gv, "gm": gm}


GRAD_EPS, GRAD_H = 1e-3, 2.0 ** -10

#: block steps and mean active particles per largest step, roughly, for the work of an integration
_STEPS, _ACTIVE = 90.0, 0.06


def _integration_work(n, dt, diag):
    """Bytes and flops of one integration: each block step reads the state of all particles once (the
    prediction) and evaluates the active ones; the diagnostics sum all pairs at both ends."""
    k = max(1.0, dt * 2.0 ** 5)
    steps, pairs = _STEPS * k, _STEPS * k * _ACTIVE * n * n
    return {"bytes": 8.0 * 21 * n * steps, "flops": FLOPS * pairs + (2 * 10.0 * n * n if diag else 0.0)}


def work(case):
    kind = case["kind"]
    if kind == "eval":
        n, k = case["n"], case["n_act"] or case["n"]
        # state, times and masses read once, nine sums per active particle written once
        return {"bytes": 8.0 * 20 * n + 72.0 * k + (4.0 * k if case["n_act"] else 0.0), "flops": FLOPS * n * k}
    if kind == "integrate":
        return _integration_work(case["n"], case["dt"], case["diag"])
    if kind == "ensemble":
        lo, hi = math.log(case["n_lo"]), math.log(case["n_hi"])
        sizes = [math.exp(lo + (hi - lo) * (q + 0.5) / case["systems"]) for q in range(case["systems"])]
        each = [_integration_work(s, case["dt"], False) for s in sizes]
        return {key: sum(w[key] for w in each) for key in ("bytes", "flops")}
    n, s = case["n"], case["steps"]
    # start-up twice, every step forward twice (checkpointed) and its adjoint once
    return {"bytes": 8.0 * 19 * n * (3 * s + 4), "flops": n * n * (FLOPS * (2 * s + 2) + 2 * FLOPS * (s + 2))}


# ---- the same results from plain torch in 64 bits

def _pair_terms(m, xi, vi, ai, xj, vj, aj, eps):
    """Acceleration, jerk and snap on the i-particles from all j, one [k, n, 3] block at a time."""
    r, v, a = xj[None] - xi[:, None], vj[None] - vi[:, None], aj[None] - ai[:, None]
    r2 = (r * r).sum(-1) + eps * eps
    mu = (m / (r2 * r2.sqrt()))[..., None]
    al = ((r * v).sum(-1) / r2)[..., None]
    be = (((v * v).sum(-1) + (r * a).sum(-1)) / r2)[..., None] + al * al
    acc = mu * r
    jerk = mu * v - 3.0 * al * acc
    snap = mu * a - 6.0 * al * jerk - 3.0 * be * acc
    return acc.sum(1), jerk.sum(1), snap.sum(1)


def _sums(m, x, v, a, act, eps):
    rows = max(1, (1 << 25) // len(m))
    out = [_pair_terms(m, x[q], v[q], a[q], x, v, a, eps) for q in act.split(rows)]
    return tuple(torch.cat(o) for o in zip(*out))


def _taylor(f, d):
    x, v, a, j, s, c = f
    return (x + d * (v + d / 2 * (a + d / 3 * (j + d / 4 * (s + d / 5 * c)))),
            v + d * (a + d / 2 * (j + d / 3 * (s + d / 4 * c))), a + d * (j + d / 2 * (s + d / 3 * c)))


def _corrected(x, v, a, j, s, A, J, S, h):
    v1 = v + h / 2 * (a + A) - h * h / 10 * (J - j) + h ** 3 / 120 * (s + S)
    x1 = x + h / 2 * (v + v1) - h * h / 10 * (A - a) + h ** 3 / 120 * (j + J)
    r1, r2, r3 = A - a - h * (j + h / 2 * s), h * (J - j - h * s), h * h * (S - s)
    return (x1, v1, (60 * r1 - 36 * r2 + 9 * r3) / h ** 3, (360 * r1 - 192 * r2 + 36 * r3) / h ** 4,
            (720 * r1 - 360 * r2 + 60 * r3) / h ** 5)


def _integrated(m, x, v, eps, dt_max, t_end, eta=0.4, eta_s=0.01, dt_min=2.0 ** -20):
    """State after block steps to t_end, by the scheme's formulas."""
    every = torch.arange(len(m), device=m.device)
    norm = lambda q: q.norm(dim=1)  # noqa: E731
    pow2 = lambda q: torch.exp2(torch.floor(torch.log2(q))).clamp(dt_min, dt_max)  # noqa: E731
    a, j, _ = _sums(m, x, v, torch.zeros_like(x), every, eps)
    _, _, s = _sums(m, x, v, a, every, eps)
    c = torch.zeros_like(x)
    dt = pow2(eta_s * torch.minimum(norm(a) / norm(j), (norm(a) / norm(s)).sqrt()))
    t = torch.zeros_like(m)
    f = [x.clone(), v.clone(), a, j, s, c]
    while True:
        tn = float((t + dt).min())
        if tn > t_end:
            break
        q = torch.nonzero(t + dt == tn)[:, 0]
        xp, vp, ap = _taylor(f, (tn - t)[:, None])
        A, J, S = _sums(m, xp, vp, ap, q, eps)
        x1, v1, c1, d1, e1 = _corrected(*(g[q] for g in f[:5]), A, J, S, (tn - t[q])[:, None])
        crit = eta * (((norm(A) * norm(S)).sqrt() + norm(J)) / ((norm(c1) * norm(e1)).sqrt() + norm(d1))) ** (1 / 3)
        old = dt[q]
        new = pow2(crit)
        new = torch.where(new > old, torch.where(torch.remainder(torch.full_like(old, tn), 2 * old) == 0, 2 * old, old), new)
        for g, val in zip(f, (x1, v1, A, J, S, c1)):
            g[q] = val
        t[q], dt[q] = tn, new
    return dict(zip("xvajsc", f), t=t, dt=dt)


def _energies(m, x, v, eps):
    pot = sum(float((m[q, None] * m / ((x[q, None] - x).square().sum(-1) + eps * eps).sqrt()).sum())
              for q in torch.arange(len(m), device=m.device).split(1024))
    pot = -0.5 * (pot - float((m * m).sum()) / eps)
    ang = (m[:, None] * torch.linalg.cross(x, v)).sum(0)
    return 0.5 * float((m * v.square().sum(1)).sum()), pot, ang


def _step_sums(m, x, v, a, eps):
    def block(q):
        return _pair_terms(m, x[q], v[q], a[q], x, v, a, eps)

    out = [torch.utils.checkpoint.checkpoint(block, q, use_reentrant=False)
           for q in torch.arange(len(m), device=m.device).split(512)]
    return tuple(torch.cat(o) for o in zip(*out))


def exact(case, seed):
    kind = case["kind"]
    on = lambda q: torch.from_numpy(np.ascontiguousarray(q)).cuda()  # noqa: E731
    if kind == "eval":
        if case["n"] * (case["n_act"] or case["n"]) > 1 << 33:
            return None  # the sums would take too long
        m, x, v, a, j, t, active = _inputs(case, seed)
        act = torch.arange(case["n"]).cuda() if active is None else on(active).long()
        m, x, v, a, j = (on(q) for q in (m, x, v, a, j))
        zero = torch.zeros_like(x)
        return _sums(m, *_taylor((x, v, a, j, zero, zero), t), act, EPS)
    if kind == "integrate":
        m, x, v = (on(q) for q in ni.plummer(case["n"], seed=seed))
        state = _integrated(m, x, v, EPS, case["dt"], case["dt"])
        if not case["diag"]:
            return {"state": state}
        ends = [_energies(m, x, v, EPS), _energies(m, state["x"], state["v"], EPS)]
        return {"state": state, "ekin": np.array([e[0] for e in ends]), "epot": np.array([e[1] for e in ends]),
                "L": torch.stack([e[2] for e in ends])}
    if kind == "ensemble":
        _, parts = _systems(case, seed)
        each = [_integrated(*(on(q) for q in p), EPS, case["dt"], case["dt"]) for p in parts[:]]
        return {"state": {k: torch.cat([e[k] for e in each]) for k in each[0]}}
    m, x, v = (on(q).requires_grad_(True) for q in ni.plummer(case["n"], seed=seed))
    a, j, _ = _step_sums(m, x, v, torch.zeros_like(x), GRAD_EPS)
    _, _, s = _step_sums(m, x, v, a, GRAD_EPS)
    f = (x, v, a, j, s, torch.zeros_like(x))
    for _ in range(case["steps"]):
        A, J, S = _step_sums(m, *_taylor(f, GRAD_H), GRAD_EPS)
        x1, v1, c1, _, _ = _corrected(*f[:5], A, J, S, GRAD_H)
        f = (x1, v1, A, J, S, c1)
    loss = (m * f[0].square().sum(1)).sum()
    gx, gv, gm = torch.autograd.grad(loss, (x, v, m))
    return {"loss": loss.detach(), "gx": gx, "gv": gv, "gm": gm}
