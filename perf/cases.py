"""The solver's work as its users have it done: what a timing run measures.

Every case goes through the public binding (paper_2407_14675_gb300.dp).  The
sizes are those of the workloads in workloads.py, of the tests and of
bench.py; draw() gives others of the same ranges.  Inputs are seeded and made
in plain torch: a value field shaped like a minimum-time value function (0 at
the target, rising to the penalty M, with a seeded ripple) and a policy near
the steepest descent of that field, which is what an iterate of policy
iteration looks like.  exact() repeats a case in plain torch FP64.
"""
import dataclasses
import math

import numpy as np
import torch

from paper_2407_14675_gb300 import dp
from paper_2407_14675_gb300 import workloads as W

DEV = "cuda" if torch.cuda.is_available() else "cpu"
TAU = 2.0 * math.pi


def listed():
    return [
        # one control decision for a handful of satellites: the smallest call a flight program makes
        dict(name="feedback_8", kind="feedback", n0=31, n1=31, n2=31, n3=31, fp64=False, states=8, steps=0),
        # the closed loop that checks a solved grid: 1,024 trajectories, the control decided anew at every step
        dict(name="closed_loop_1024", kind="feedback", n0=61, n1=61, n2=61, n3=61, fp64=False, states=1024, steps=100),
        # FP64 value iteration on the 17^4 box, 16 angles
        dict(name="vi_fp64_17", kind="vi", n0=17, n1=17, n2=17, n3=17, angles=16, sweeps=50),
        # policy iteration on the 61^4 box in FP32: two outer steps (walk improvement + 20 evaluation sweeps) with
        # the value and the policy coming from and going back to pinned host memory
        dict(name="pi_61", kind="pi", n0=61, n1=61, n2=61, n3=61, band=False, fp64=False, diag=False, outer=2, n_eval=20),
        # the same on the 121^4 energy band, the largest single grid (the benchmark's step)
        dict(name="pi_band_121", kind="pi", n0=121, n1=121, n2=121, n3=121, band=True, fp64=False, diag=False, outer=2,
             n_eval=20),
        # FP64 policy iteration on a ragged box with the diagonal-solved evaluation
        dict(name="pi_fp64_ragged", kind="pi", n0=31, n1=41, n2=25, n3=17, band=False, fp64=True, diag=True, outer=2,
             n_eval=40),
        # a whole solve to 1e-6 from nothing, coarse to fine with the FP64-value finish
        dict(name="solve_cascade_61", kind="solve", levels="16,31,61", n_eval=20),
        # the paper's Example 1 at its size: polar dynamics, FP64, thrust off among the controls
        dict(name="example1_110", kind="polar", n0=110, n1=30, n2=30, n3=30, outer=2, n_eval=40),
        # a frozen policy evaluated by GMRES, as the paper prescribes
        dict(name="gmres_41", kind="gmres", n0=41, n1=41, n2=41, n3=41, fp64=False, restart=20, cycles=2),
        # many transfers of uneven sizes solved together (16 of them, sixteen outer steps from nothing)
        dict(name="batch_16", kind="batch", count=16, sizes="17,21,25,31,41", size_seed=7, outer=16, n_eval=20),
        # the warm-start network trained on a grid's value and policy: one epoch of Adam at the benchmark's batch
        dict(name="net_train_25", kind="train", n0=25, n1=25, n2=25, n3=25, batch=16384),
        # the network evaluated at every node of a grid, to start its solve
        dict(name="net_start_61", kind="start", n0=61, n1=61, n2=61, n3=61),
    ]


def _log(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def _sizes(rng, lo, hi, most):
    while True:
        n = [rng.randint(lo, hi) for _ in range(4)]
        if n[0] * n[1] * n[2] * n[3] <= most:
            return dict(n0=n[0], n1=n[1], n2=n[2], n3=n[3])


def draw(rng):
    kind = rng.choice(["feedback", "vi", "pi", "pi", "solve", "polar", "gmres", "batch", "train", "start"])
    if kind == "feedback":
        steps = rng.choice([0, _log(rng, 10, 100)])
        return dict(kind=kind, fp64=rng.random() < 0.4, states=_log(rng, 1, 1024), steps=steps, **_sizes(rng, 13, 41, 10 ** 6))
    if kind == "vi":
        return dict(kind=kind, angles=rng.choice([8, 16, 24, 32]), sweeps=_log(rng, 10, 60), **_sizes(rng, 7, 25, 10 ** 5))
    if kind == "pi":
        fp64 = rng.random() < 0.3
        most = 4 * 10 ** 5 if fp64 else 2 * 10 ** 7
        top = 41 if fp64 else rng.choice([25, 41, 71])
        return dict(kind=kind, band=rng.random() < 0.4, fp64=fp64, diag=rng.random() < 0.5, outer=rng.randint(1, 3),
                    n_eval=rng.choice([5, 10, 20, 40]), **_sizes(rng, 15, top, most))
    if kind == "solve":
        top = rng.randint(25, 55)
        return dict(kind=kind, levels="%d,%d,%d" % ((top + 3) // 4, (top + 1) // 2, top), n_eval=rng.choice([20, 40]))
    if kind == "polar":
        return dict(kind=kind, outer=rng.randint(1, 2), n_eval=rng.choice([20, 40]), n0=rng.randint(30, 110),
                    n1=rng.randint(12, 30), n2=rng.randint(12, 30), n3=rng.randint(12, 30))
    if kind == "gmres":
        return dict(kind=kind, fp64=rng.random() < 0.3, restart=rng.randint(8, 30), cycles=rng.randint(1, 3),
                    **_sizes(rng, 13, 41, 10 ** 6))
    if kind == "batch":
        return dict(kind=kind, count=rng.randint(2, 24), sizes=rng.choice(["17,21,25", "17,21,25,31", "11,17,23,29"]),
                    size_seed=rng.randint(1, 10 ** 6), outer=rng.randint(4, 16), n_eval=rng.choice([10, 20, 40]))
    if kind == "train":
        return dict(kind=kind, batch=512 * _log(rng, 4, 32), **_sizes(rng, 17, 27, 4 * 10 ** 5))
    return dict(kind=kind, **_sizes(rng, 11, 61, 8 * 10 ** 6))


# ---- problems and inputs -------------------------------------------------------------------------------------------


def _n(case):
    return (case["n0"], case["n1"], case["n2"], case["n3"])


def _problem(case, seed):
    """The case's problem.  The seed moves the thrust a little: other inputs of the same size."""
    f = math.exp(np.random.RandomState(seed % (1 << 32)).uniform(-0.2, 0.2))
    kind = case["kind"]
    if kind == "polar":
        return W.example1(n=_n(case), accel=5e-7 * f)
    if kind == "vi":
        return W.config0().replace(n=_n(case), n_angles=case["angles"], accel=1e-3 * f)
    n = _n(case) if "n0" in case else (int(case["levels"].split(",")[-1]),) * 4
    p = W.config1().replace(n=n, accel=2e-4 * f, precision=W.FP64 if case.get("fp64") else W.FP32)
    if case.get("band"):
        e_lo, e_hi = W.energy_band(1.0, 1.05)
        p = p.replace(reduced=1, energy_lo=e_lo, energy_hi=e_hi)
    return p


def _coords(p, idx):
    """FP64 coordinates (4 tensors) of box indices."""
    x = []
    for d in (3, 2, 1, 0):
        i = idx % p.n[d]
        idx = idx // p.n[d]
        x.append(p.lo[d] + i.to(torch.float64) * ((p.hi[d] - p.lo[d]) / (p.n[d] - 1)))
    return x[::-1]


def _field(p, x, rs):
    """The value field at coordinates x; rs: a dict of seeded ripple numbers."""
    if p.dynamics == W.DYN_POLAR:
        e = _elements(p, x)
        cost = 0.4 * ((e[0] - p.a_bar) / 25.0) ** 2 + ((e[1] - p.e_bar) ** 2 + e[2] ** 2) / 0.004 ** 2
    else:
        cost = ((x[0] - p.target_c[0]) / 0.06) ** 2 + (x[1] / 0.06) ** 2
        cost = cost + ((x[2] - torch.sqrt(p.mu / x[0])) / 0.05) ** 2 + 0.1 * (x[3] - 0.9)
    ripple = torch.zeros_like(x[0])
    for d in range(4):
        ripple = ripple + rs["a"][d] * torch.cos(rs["k"][d] * (x[d] - p.lo[d]) / (p.hi[d] - p.lo[d]) + rs["p"][d])
    return p.M() * torch.clamp((1.0 - torch.exp(-0.7 * torch.sqrt(cost + 1e-4))) * (0.93 + 0.02 * ripple), 0.0, 1.0)


def _elements(p, x):
    """Semi-major axis and eccentricity vector of polar states."""
    r, vr, vt, th = x
    a = p.mu * r / (2.0 * p.mu - r * (vr * vr + vt * vt))
    er, et = r * vt * vt / p.mu - 1.0, -r * vr * vt / p.mu
    return a, er * torch.cos(th) - et * torch.sin(th), er * torch.sin(th) + et * torch.cos(th)


def _ripple(seed):
    r = np.random.RandomState((seed * 7919 + 13) % (1 << 32))
    return {"a": r.uniform(0.3, 1.0, 4), "k": r.uniform(1.5, 6.0, 4), "p": r.uniform(0.0, TAU, 4), "s": int(r.randint(1 << 30))}


def _inputs(p, idx, seed):
    """Value (FP64) and policy codes (int64) at the stored nodes `idx`."""
    rs = _ripple(seed)
    x = _coords(p, idx)
    V = _field(p, x, rs)
    g = []
    for d in (1, 2):
        h = 0.25 * (p.hi[d] - p.lo[d]) / (p.n[d] - 1)
        y = list(x)
        y[d] = x[d] + h
        up = _field(p, y, rs)
        y[d] = x[d] - h
        g.append(up - _field(p, y, rs))
    gen = torch.Generator(device=idx.device).manual_seed(rs["s"])
    noise = 0.06 * torch.randn(idx.shape, generator=gen, device=idx.device, dtype=torch.float32).double()
    if p.dynamics == W.DYN_POLAR:   # off where the field is flat
        alpha = torch.atan2(-g[0], -g[1]) + noise
        code = torch.remainder(torch.round(alpha * (65536 / TAU)), 65536).long()
        return V, torch.where(g[0].abs() + g[1].abs() < 1e-6 * p.M(), torch.full_like(code, dp.DP_CODE_OFF), code)
    alpha = torch.atan2(-g[0], -g[1]) + noise
    return V, torch.remainder(torch.round(alpha * (65536 / TAU)), 65536).long()


def _stored(p, g=None):
    if p.reduced:
        return torch.from_numpy(g.active_index()).to(DEV)
    return torch.arange(p.nodes, device=DEV)


def _pinned(t):
    out = torch.empty(t.shape, dtype=t.dtype, pin_memory=DEV == "cuda")
    out.copy_(t)
    return out


def _codes16(code):
    return torch.where(code > 32767, code - 65536, code).to(torch.int16)


def _batch_problems(case, seed):
    n = np.random.RandomState(case["size_seed"])
    sizes = [int(s) for s in case["sizes"].split(",")]
    r = np.random.RandomState((seed + 1) % (1 << 32))
    out = []
    for _ in range(case["count"]):
        shape = tuple(int(s) for s in n.choice(sizes, 4))
        a, r_t, r0 = math.exp(r.uniform(math.log(1e-4), math.log(2e-3))), r.uniform(1.02, 1.10), r.uniform(0.98, 1.02)
        c, w = W.circular_target(r_t)
        out.append(W.Problem(n=shape, lo=(r0 - 0.05, -0.10, 0.85, 0.90), hi=(r_t + 0.10, 0.10, 1.10, 1.00), accel=a, dt=0.05,
                             n_angles=32, refine=1, precision=W.FP32, target_c=c, target_w=w))
    return out


def _states(p, count, seed):
    """Flight states inside the box, away from its faces."""
    r = np.random.RandomState((seed * 31 + 5) % (1 << 32))
    lo, hi = np.array(p.lo), np.array(p.hi)
    return lo + (hi - lo) * (0.3 + 0.4 * r.uniform(size=(count, 4)))


def prepare(case, seed):
    kind = case["kind"]
    s = dict(case=case)
    if kind == "batch":
        s["batch"] = dp.Batch(_batch_problems(case, seed))
        return s
    p = s["p"] = _problem(case, seed)
    if kind == "solve":
        s["grids"] = [dp.Grid(p.replace(n=(int(m),) * 4)) for m in case["levels"].split(",")]
        n = s["grids"][-1].n
        s["V_out"] = torch.empty(n, dtype=torch.float64, pin_memory=True)
        s["code_out"] = torch.empty(n, dtype=torch.int16, pin_memory=True)
        return s
    g = s["grid"] = dp.Grid(p)
    if kind in ("train", "start"):
        s["params"] = dp.flatten_params(W.mlp_init_params(seed=seed % (1 << 32)))
        s["mlp"] = dp.Mlp(p.lo, p.hi, batch_capacity=case["batch"] if kind == "train" else 1 << 18)
        dp.dp_mlp_set_params(s["mlp"].h, s["params"])
        if kind == "start":
            s["V_out"] = torch.empty(g.n, dtype=torch.float32, pin_memory=True)
            s["code_out"] = torch.empty(g.n, dtype=torch.int16, pin_memory=True)
            return s
    V, code = _inputs(p, _stored(p, g), seed)
    f64 = p.precision == W.FP64
    s["V"] = _pinned(V if f64 else V.float())
    s["code"] = _pinned(_codes16(code))
    if kind in ("feedback", "train"):
        _put(s)
        if kind == "feedback":
            s["x"] = _states(p, case["states"], seed)
        return s
    s["V_out"] = torch.empty_like(s["V"], pin_memory=True)
    if kind in ("pi", "polar"):
        s["code_out"] = torch.empty_like(s["code"], pin_memory=True)
    return s


# ---- one pass ------------------------------------------------------------------------------------------------------


def _put(s):
    g = s["grid"]
    (dp.dp_set_value if s["V"].dtype == torch.float64 else dp.dp_set_value_f32)(g.h, s["V"])
    dp.dp_set_policy(g.h, s["code"])


def _get(s, h):
    (dp.dp_get_value if s["V_out"].dtype == torch.float64 else dp.dp_get_value_f32)(h, len(s["V_out"]), s["V_out"])
    if "code_out" in s:
        dp.dp_get_policy(h, len(s["code_out"]), s["code_out"])
        return {"V": s["V_out"], "code": s["code_out"]}
    return {"V": s["V_out"]}


def run(s):
    case = s["case"]
    kind = case["kind"]
    if kind == "feedback":
        if case["steps"] == 0:
            alpha, q = s["grid"].feedback(s["x"], s["p"].dt)
            return {"alpha": alpha, "q": q}
        dt = s["p"].dt
        t, x = s["grid"].simulate(s["x"], dt, dt, case["steps"] * dt)
        return {"t": t, "x": x}
    if kind == "vi":
        _put(s)
        _, st = s["grid"].value_iterate(tol=0.0, max_sweeps=case["sweeps"], warm=1)
        return dict(_get(s, s["grid"].h), residual=st.residual)
    if kind in ("pi", "polar"):
        _put(s)
        diag = case.get("diag", True)
        _, st = s["grid"].policy_iterate(tol=0.0, max_sweeps=case["outer"], n_eval=case["n_eval"], warm=1, polish=0,
                                         eval_solver=dp.DP_EVAL_DIAG if diag else dp.DP_EVAL_JACOBI)
        return dict(_get(s, s["grid"].h), residual=st.residual)
    if kind == "gmres":
        _put(s)
        _, st = s["grid"].policy_evaluate(tol=0.0, max_sweeps=case["cycles"], gmres_restart=case["restart"])
        return _get(s, s["grid"].h)
    if kind == "solve":
        last = None
        for g in s["grids"]:
            if last is not None:
                dp.dp_warm_start_from_grid(last.h, g.h)
            g.policy_iterate(tol=1e-6, max_sweeps=400, n_eval=case["n_eval"], warm=int(last is not None),
                             eval_solver=dp.DP_EVAL_DIAG)
            last = g
        return _get(s, last.h)
    if kind == "batch":
        b = s["batch"]
        b.policy_iterate(tol=1e-6, max_sweeps=case["outer"], n_eval=case["n_eval"], warm=0, polish=1)
        return {"V": [b.get_value(i) for i in range(b.count)], "code": [b.get_policy(i) for i in range(b.count)]}
    m = s["mlp"].h
    if kind == "train":
        dp.dp_mlp_set_params(m, s["params"])
        st = dp.dp_mlp_train_grid(m, s["grid"].h, epochs=1, batch=case["batch"], lr=4e-3)
        return {"params": dp.dp_mlp_get_params(m), "loss": st.last_epoch_loss}
    dp.dp_warm_start(m, s["grid"].h)
    return _get(s, s["grid"].h)


# ---- what a pass cannot do without ---------------------------------------------------------------------------------

_EVAL_FLOPS = 45          # one control at one node: 7 FMAs of the step, 15 lerps
_NET_FLOPS = 2 * 132864   # one sample through the network


def _nodes(case):
    n = case["n0"] * case["n1"] * case["n2"] * case["n3"]
    return int(0.261 * n) if case.get("band") else n


def work(case):
    kind = case["kind"]
    if kind == "feedback":
        decisions = case["states"] * max(1, case["steps"])
        evals = (64 + 16) * decisions
        return {"bytes": 16 * (8 if case["fp64"] else 4) * decisions, "flops": _EVAL_FLOPS * evals}
    if kind == "vi":
        return {"bytes": 16 * _nodes(case) * case["sweeps"], "flops": _EVAL_FLOPS * case["angles"] * _nodes(case) * case["sweeps"]}
    if kind in ("pi", "polar"):
        n, b = _nodes(case), 8 if case.get("fp64") or kind == "polar" else 4
        sweep = (2 * b + 2) * n
        return {"bytes": case["outer"] * (sweep * (1 + case["n_eval"]) + 2 * n),
                "flops": case["outer"] * n * _EVAL_FLOPS * (20 + case["n_eval"])}
    if kind == "gmres":
        n, b = _nodes(case), 8 if case["fp64"] else 4
        m = case["restart"]
        return {"bytes": case["cycles"] * n * b * (m * (m + 5) + 4), "flops": case["cycles"] * n * (_EVAL_FLOPS * m + 4 * m * m)}
    if kind == "solve":
        n = sum(int(m) ** 4 for m in case["levels"].split(","))
        return {"bytes": 20 * n * (12 + 10 * case["n_eval"]), "flops": 20 * n * _EVAL_FLOPS * (20 + case["n_eval"])}
    if kind == "batch":
        n = sum(p.nodes for p in _batch_problems(case, 0))
        return {"bytes": case["outer"] * n * (12 + 10 * case["n_eval"]), "flops": case["outer"] * n * _EVAL_FLOPS * (30 + case["n_eval"])}
    if kind == "train":
        steps = _nodes(case) // case["batch"]
        return {"bytes": 6 * steps * case["batch"], "flops": 3 * _NET_FLOPS * steps * case["batch"]}
    return {"bytes": 6 * _nodes(case), "flops": _NET_FLOPS * _nodes(case)}


# ---- the same in plain torch FP64 ----------------------------------------------------------------------------------


def _target(p):
    t = torch.ones((1,) * 4, dtype=torch.bool, device=DEV)
    for d in range(4):
        if p.target_w[d] > 0:
            x = p.lo[d] + torch.arange(p.n[d], device=DEV, dtype=torch.float64) * ((p.hi[d] - p.lo[d]) / (p.n[d] - 1))
            shape = [1] * 4
            shape[d] = -1
            t = t & ((x - p.target_c[d]).abs() < p.target_w[d]).reshape(shape)
    return t.expand(p.n).reshape(-1)


def _heun(p, x, alpha, dt):
    s, c = torch.sin(alpha), torch.cos(alpha)

    def f(y):
        am = p.accel / y[3]
        return [y[1], y[2] ** 2 / y[0] - p.mu / y[0] ** 2 + am * s, -y[1] * y[2] / y[0] + am * c,
                torch.full_like(y[0], -p.accel / p.exhaust_c)]

    k1 = f(x)
    k2 = f([a + dt * b for a, b in zip(x, k1)])
    return [a + 0.5 * dt * (b + c2) for a, b, c2 in zip(x, k1, k2)]


def _cell(p, z):
    """Box index of the lower corner, fractions and the outside flag of states z."""
    base, frac, out = torch.zeros_like(z[0], dtype=torch.int64), [], torch.zeros_like(z[0], dtype=torch.bool)
    for d in range(4):
        u = (z[d] - p.lo[d]) / ((p.hi[d] - p.lo[d]) / (p.n[d] - 1))
        out |= ~((u >= -1e-12) & (u <= p.n[d] - 1 + 1e-12))
        c = torch.clamp(torch.floor(u), 0, p.n[d] - 2)
        frac.append(torch.clamp(u - c, 0.0, 1.0))
        base = base * p.n[d] + c.long()
    return base, frac, out


def _corners(p, frac):
    """(index offset, weight) of the 16 corners."""
    stride = [p.n[1] * p.n[2] * p.n[3], p.n[2] * p.n[3], p.n[3], 1]
    for m in range(16):
        off, w = 0, 1.0
        for d in range(4):
            bit = (m >> d) & 1
            off += bit * stride[d]
            w = w * (frac[d] if bit else 1.0 - frac[d])
        yield off, w


def _bellman(p, V, x, alpha, dt=None):
    dt = p.dt if dt is None else dt
    base, frac, out = _cell(p, _heun(p, x, alpha, dt))
    v = sum(w * V[base + off] for off, w in _corners(p, frac))
    return dt + p.beta ** (dt / p.dt) * torch.where(out, torch.full_like(v, p.M()), v)


def exact(case, seed):
    kind = case["kind"]
    if kind in ("pi", "polar", "solve", "batch") or (kind == "feedback" and case["steps"]):
        # the search over angles decides near-ties by rounding, so a policy has no 64-bit value of its own, and the
        # values and trajectories that follow depend on it
        return None
    p = _problem(case, seed)
    idx = torch.arange(p.nodes, device=DEV)
    if kind in ("train", "start"):
        return _exact_network(case, p, seed)
    x = _coords(p, idx)
    V, code = _inputs(p, idx, seed)
    if p.precision == W.FP32:
        V = V.float().double()   # the grid stores FP32: these are the inputs
    tgt = _target(p)
    V = torch.where(tgt, torch.zeros_like(V), V)
    alpha = code * (TAU / 65536)
    if kind == "feedback":
        y = [torch.from_numpy(c.copy()).to(DEV).reshape(-1, 1) for c in _states(p, case["states"], seed).T]
        every = torch.arange(65536, device=DEV, dtype=torch.float64) * (TAU / 65536)
        q = torch.cat([_bellman(p, V, [c[k:k + 8].expand(-1, 65536) for c in y], every.expand(len(y[0][k:k + 8]), -1)).amin(1)
                       for k in range(0, case["states"], 8)])
        return {"alpha": None, "q": q}
    if kind == "vi":
        for _ in range(case["sweeps"]):
            new = torch.where(tgt, torch.zeros_like(V), _vi_sweep(p, V, x))
            res = float((new - V).abs().max())
            V = new
        return {"V": V, "residual": res}
    return {"V": _exact_gmres(case, p, V, x, alpha, tgt)}


def _vi_sweep(p, V, x):
    best = None
    for k in range(p.n_angles):
        a = torch.tensor(((k * 65536 + p.n_angles // 2) // p.n_angles) * (TAU / 65536), device=DEV, dtype=torch.float64)
        q = _bellman(p, V, x, a)
        best = q if best is None else torch.minimum(best, q)
    return best


def _exact_gmres(case, p, V, x, alpha, tgt):
    """One evaluation sweep, then per cycle a restarted GMRES correction and another sweep."""
    base, frac, out = _cell(p, _heun(p, x, alpha, p.dt))
    empty = out | tgt

    def wx(v):
        r = sum(w * v[base + off] for off, w in _corners(p, frac))
        return torch.where(empty, torch.zeros_like(r), r)

    b = torch.where(tgt, torch.zeros_like(V), p.dt + p.beta * torch.where(out, torch.full_like(V, p.M()), torch.zeros_like(V)))
    new = b + p.beta * wx(V)
    for _ in range(case["cycles"]):
        r = new - V
        beta0 = float(r.norm())
        Q, H, y = [r / beta0], torch.zeros(case["restart"] + 1, case["restart"], dtype=torch.float64), None
        for k in range(case["restart"]):
            w = Q[k] - p.beta * wx(Q[k])
            for i in range(k + 1):
                H[i, k] = torch.dot(Q[i], w)
            for i in range(k + 1):
                w = w - H[i, k].item() * Q[i]
            H[k + 1, k] = w.norm()
            e1 = torch.zeros(k + 2, 1, dtype=torch.float64)
            e1[0] = beta0
            y = torch.linalg.lstsq(H[:k + 2, :k + 1], e1).solution
            Q.append(w / H[k + 1, k].item())
            if float((e1 - H[:k + 2, :k + 1] @ y).norm()) <= 1e-3 * beta0:
                break
        V = V + sum(c.item() * q for c, q in zip(y.reshape(-1), Q))
        new = b + p.beta * wx(V)
    return new


def _net(params, x):
    h = x
    z = []
    for k, (w, b) in enumerate(params):
        a = h @ w.T + b
        z.append((h, a))
        h = a if k == 3 else 0.5 * a * (1.0 + torch.erf(a / math.sqrt(2.0)))
    return h, z


def _scaled(p, idx):
    return torch.stack([2.0 * (c - p.lo[d]) / (p.hi[d] - p.lo[d]) - 1.0 for d, c in enumerate(_coords(p, idx))], 1)


def _exact_network(case, p, seed):
    flat = dp.flatten_params(W.mlp_init_params(seed=seed % (1 << 32)))
    params = [[torch.from_numpy(a.copy()).to(DEV) for a in layer] for layer in dp.unflatten_params(flat)]
    if case["kind"] == "start":
        V = torch.cat([_net(params, _scaled(p, i))[0][:, 0] for i in torch.arange(p.nodes, device=DEV).split(1 << 19)])
        return {"V": torch.where(_target(p), torch.zeros_like(V), p.M() * V.clamp(0.0, 1.0)), "code": None}
    nodes, B = p.nodes, case["batch"]
    field, code = _inputs(p, torch.arange(nodes, device=DEV), seed)
    field = torch.where(_target(p), torch.zeros_like(field), field.float().double()) / p.M()
    alpha = code * (TAU / 65536)
    goal = torch.stack([field, torch.cos(alpha), torch.sin(alpha)], 1)
    rng = [14675]

    def splitmix():
        rng[0] = (rng[0] + 0x9E3779B97F4A7C15) & (2 ** 64 - 1)
        z = rng[0]
        z = ((z ^ (z >> 30)) * 0xBF58476D1CE4E5B9) & (2 ** 64 - 1)
        z = ((z ^ (z >> 27)) * 0x94D049BB133111EB) & (2 ** 64 - 1)
        return z ^ (z >> 31)

    mult = (splitmix() % nodes) | 1
    while math.gcd(mult, nodes) != 1:
        mult = (mult + 2) % nodes
    off = splitmix() % nodes
    order = torch.remainder(torch.arange(nodes, device=DEV) * mult + off, nodes)
    m = [[torch.zeros_like(a) for a in layer] for layer in params]
    v = [[torch.zeros_like(a) for a in layer] for layer in params]
    total, steps = 0.0, nodes // B
    for t in range(steps):
        i = order[t * B:(t + 1) * B]
        y, z = _net(params, _scaled(p, i))
        d = y - goal[i]
        total += float((d * d).sum())
        d = 2.0 * d / (3.0 * B)
        for k in (3, 2, 1, 0):
            h, a = z[k]
            if k < 3:
                d = d * (0.5 * (1.0 + torch.erf(a / math.sqrt(2.0))) + a * torch.exp(-0.5 * a * a) / math.sqrt(TAU))
            grads = (d.T @ h, d.sum(0))
            d = d @ params[k][0]
            for j, g in enumerate(grads):
                m[k][j] = 0.9 * m[k][j] + 0.1 * g
                v[k][j] = 0.999 * v[k][j] + 0.001 * g * g
                step = (m[k][j] / (1 - 0.9 ** (t + 1))) / ((v[k][j] / (1 - 0.999 ** (t + 1))).sqrt() + 1e-8)
                params[k][j] = params[k][j] - 4e-3 * step
    return {"params": torch.cat([a.reshape(-1) for layer in params for a in layer]), "loss": total / (3.0 * B * steps)}
