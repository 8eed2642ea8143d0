"""The work that a user of this library has it do, as cases that can be timed.

Every case goes through the Python binding (``paper_1608_05794_gb300.ck``),
on device tensors, as a reacting-flow code calls it once per time step:
right-hand sides and Jacobians of a batch of reactors, the linear algebra of
an implicit step, and whole integrations with ROS4 and RKF45.  Mechanisms,
reactor states and time steps are those of ``synth.configs`` (the 10-, 53-
and 111-species workloads and the mixed batch).

``exact`` restates the formulas in plain torch, in 64 bits.
"""
from __future__ import annotations

import math

import numpy as np
import torch

import paper_1608_05794_gb300.ck as ck
from synth.configs import CONFIGS, MIXED, ignition_states, load_mechanism
from synth.draw import draw_densities, draw_states

DEV = "cuda"
F8 = torch.float64

# Interval of the integrations, s: the workload's own, and for RKF45 on the
# 10-species mechanism the middle of the mixed batch's range.
DT = {("small", "ros4"): 1e-4, ("medium", "ros4"): 1e-5, ("large", "ros4"): 1e-5,
      ("small", "rkf45"): 1e-5, ("medium", "rkf45"): 1e-5, ("large", "rkf45"): 1e-5}
# Attempted steps per reactor over it (averages over 2048 reactors and more at
# rtol 1e-9, atol 1e-12), for work(); and over the mixed batch's intervals.
STEPS = {("small", "ros4"): 800.0, ("medium", "ros4"): 348.0, ("large", "ros4"): 54.0,
         ("small", "rkf45"): 70.0, ("medium", "rkf45"): 90.6, ("large", "rkf45"): 16.9}
MIXED_STEPS = {"small": 119.0, "medium": 94.0, "large": 15.7}


def listed():
    return [
        # one small right-hand side call: the 10-species workload at its own
        # batch size, where the launch counts
        dict(name="rhs_small_512", kind="rhs", workload="small", n=512, cv=False),
        # the 53-species workload at its own batch size: an explicit flow
        # solver's source term, or one stage of its own integrator
        dict(name="rhs_medium_131072", kind="rhs", workload="medium", n=131072, cv=False),
        # the largest mechanism as constant-volume reactors, a ragged batch
        dict(name="rhs_large_cv_20011", kind="rhs", workload="large", n=20011, cv=True),
        # analytic Jacobians for a caller's own implicit method
        dict(name="jacobian_medium_8192", kind="jacobian", workload="medium", n=8192, cv=False),
        # factor and solve I/(h gamma) - J for a caller's own implicit method
        dict(name="newton_medium_4096", kind="newton", workload="medium", n=4096),
        # ROS4 over the smallest workload: less than one reactor a resident
        # team, so the latency of a step counts
        dict(name="ros4_small_512", kind="ros4", workload="small", n=512, cv=False, precision=0, jac=0),
        # ROS4 over a block of cells of the 53-species workload (the
        # library's headline integration)
        dict(name="ros4_medium_4096", kind="ros4", workload="medium", n=4096, cv=False, precision=0, jac=0),
        # ROS4 with the 111-species mechanism, in FP64 and in the precision
        # form (FP32 LU with FP64 refinement), ragged batches
        dict(name="ros4_large_1500", kind="ros4", workload="large", n=1500, cv=False, precision=0, jac=0),
        dict(name="ros4_large_p1_1501", kind="ros4", workload="large", n=1501, cv=False, precision=1, jac=0),
        # RKF45 over non-stiff cells: the 53-species mechanism, and a large
        # batch of the 10-species one
        dict(name="rkf45_medium_16384", kind="rkf45", workload="medium", n=16384, cv=False),
        dict(name="rkf45_small_100003", kind="rkf45", workload="small", n=100003, cv=False),
        # cells of three mechanisms in one call, half of them near ignition,
        # time steps over two decades (the mixed batch, captured as a graph)
        dict(name="mixed_rkf45_8000", kind="mixed", n=8000),
    ]


# Largest batch that draw() takes of each kind of call, by workload: what the
# listed cases cost, or less.
MOST = {
    "rhs": {"small": 500000, "medium": 131072, "large": 40000},
    "jacobian": {"small": 100000, "medium": 8192, "large": 1600},
    "newton": {"small": 60000, "medium": 4096, "large": 900},
    "ros4": {"small": 4000, "medium": 3500, "large": 2500},
    "rkf45": {"small": 120000, "medium": 16384, "large": 20000},
}


def draw(rng):
    kind = rng.choice(("rhs", "jacobian", "newton", "ros4", "ros4", "rkf45", "mixed"))
    if kind == "mixed":
        return dict(kind="mixed", n=int(round(math.exp(rng.uniform(math.log(100), math.log(8000))))))
    w = rng.choice(("small", "medium", "large"))
    n = int(round(math.exp(rng.uniform(0.0, math.log(MOST[kind][w])))))
    if kind == "newton":
        return dict(kind=kind, workload=w, n=n)
    c = dict(kind=kind, workload=w, n=n, cv=rng.random() < 0.25)
    if kind == "ros4":
        c["precision"] = rng.choice((0, 0, 1, 2))
        # forward-difference Jacobians, the paper's own choice, cost n + 1
        # right-hand sides each: in the FP64 form of the 10-species mechanism
        c["jac"] = int(w == "small" and n <= 500 and c["precision"] == 0 and rng.random() < 0.5)
    return c


# ------------------------------------------------------------------ inputs
_tables = {}


def _mech(workload):
    if workload not in _tables:
        _tables[workload] = load_mechanism(CONFIGS[workload]["mech"])
    return _tables[workload]


def _states(workload, n, cv, rng):
    """Reactor states of a workload: y [n, S+1] and the pressure, or for
    constant-volume reactors the density."""
    cfg, m = CONFIGS[workload], _mech(workload)
    y, p = draw_states(rng, m["names"], m["elem"], m["mw"], m["elements"], n, cfg["t_range"], cfg["p_range_atm"])
    return _dev(y), _dev(draw_densities(rng, n) if cv else p)


def _dev(a):
    return torch.as_tensor(np.ascontiguousarray(a), device=DEV)


def _newton_inputs(case, rng):
    """Iteration matrices I/(h gamma) - J at step sizes from 1e-9 to 1e-6 s,
    and right-hand sides f(y)."""
    y, p = _states(case["workload"], case["n"], False, rng)
    m = _Plain(case["workload"])
    h = _dev(10.0 ** rng.uniform(-9.0, -6.0, case["n"]))
    a = -_by_rows(lambda q, s: _jac(m, False, q, s), p, y, 2048)
    a.diagonal(dim1=1, dim2=2).add_((1.0 / (h * 0.57282))[:, None])
    return a, _by_rows(lambda q, s: _rhs(m, False, q, s), p, y, 16384)


def _mixed_inputs(n, rng):
    """The mixed batch: (workload, y, p, dt) of its three mechanisms, half of
    the reactors of each from its stored near-ignition states."""
    counts = [max(1, int(round(n * f))) for _, f in MIXED["split"]]
    out = []
    for (name, _), k in zip(MIXED["split"], counts):
        m = _mech(name)
        y, p = draw_states(rng, m["names"], m["elem"], m["mw"], m["elements"], k, MIXED["t_range"],
                           MIXED["p_range_atm"])
        yi, pi = ignition_states(name)
        at = rng.permutation(k)[:k // 2]
        of = rng.integers(len(yi), size=k // 2)
        y[at], p[at] = yi[of], pi[of]
        dt = 10.0 ** rng.uniform(np.log10(MIXED["dt_range"][0]), np.log10(MIXED["dt_range"][1]), k)
        out.append((name, _dev(y), _dev(p), _dev(dt)))
    return out


def prepare(case, seed):
    rng = np.random.default_rng(seed)
    kind = case["kind"]
    s = dict(kind=kind)
    if kind == "newton":
        s["a"], s["b"] = _newton_inputs(case, rng)
        n, dim = s["b"].shape
        s.update(lu=torch.empty_like(s["a"]), x=torch.empty_like(s["b"]),
                 piv=torch.empty((n, dim), dtype=torch.int32, device=DEV),
                 info=torch.empty(n, dtype=torch.int32, device=DEV))
        return s
    if kind == "mixed":
        s["groups"], s["y0"] = [], []
        for name, y, p, dt in _mixed_inputs(case["n"], rng):
            s["y0"].append(y)
            s["groups"].append(dict(mech=ck.load_mechanism(_mech(name)), p=p, y=torch.empty_like(y), dt=dt,
                                    status=torch.empty(len(y), dtype=torch.int32, device=DEV)))
        return s
    w, n = case["workload"], case["n"]
    s["mech"] = ck.load_mechanism(_mech(w), reactor=int(case["cv"]))
    s["y"], s["p"] = _states(w, n, case["cv"], rng)
    dim = s["y"].shape[1]
    if kind == "rhs":
        s["out"] = torch.empty_like(s["y"])
    elif kind == "jacobian":
        s["out"] = torch.empty((n, dim, dim), dtype=F8, device=DEV)
    else:
        s["y1"] = torch.empty_like(s["y"])
        s["dt"] = torch.full((n,), DT[w, kind], dtype=F8, device=DEV)
        s["status"] = torch.empty(n, dtype=torch.int32, device=DEV)
        s["opts"] = ck.SolverOpts.make(precision=case.get("precision", 0), jac=case.get("jac", 0))
    return s


def run(state):
    s, kind = state, state["kind"]
    if kind == "rhs":
        return ck.rhs(s["mech"], s["p"], s["y"], s["out"])
    if kind == "jacobian":
        return ck.jacobian(s["mech"], s["p"], s["y"], s["out"])
    if kind == "newton":  # the library factors and solves in place
        s["lu"].copy_(s["a"])
        s["x"].copy_(s["b"])
        ck.lu_factor(s["lu"], s["piv"], s["info"])
        ck.lu_solve(s["lu"], s["piv"], s["x"])
        return [s["lu"], s["x"], s["piv"], s["info"]]
    if kind == "mixed":
        for g, y0 in zip(s["groups"], s["y0"]):
            g["y"].copy_(y0)
        ck.integrate_groups(1, s["groups"])
        return [[g["y"], g["status"]] for g in s["groups"]]
    s["y1"].copy_(s["y"])  # the library integrates in place
    fn = ck.integrate_ros4 if kind == "ros4" else ck.integrate_rkf45
    fn(s["mech"], s["p"], s["y1"], s["dt"], s["status"], opts=s["opts"])
    return [s["y1"], s["status"]]


# ------------------------------------------------------------------ work
_counts = {}


def _per(workload, cv):
    """The algorithm's flops of each unit (ck_count_work)."""
    if (workload, cv) not in _counts:
        m = ck.load_mechanism(_mech(workload), reactor=int(cv))
        _counts[workload, cv] = ck.count_work(m)
        m.close()
    return _counts[workload, cv]


def work(case):
    kind, n = case["kind"], case["n"]
    if kind == "mixed":
        b = f = 0.0
        for name, share in MIXED["split"]:
            k = max(1, int(round(n * share)))
            b += k * (16.0 * (CONFIGS[name]["n_species"] + 1) + 20.0)
            f += k * MIXED_STEPS[name] * _per(name, False)["rkf45_step_flops"]
        return {"bytes": b, "flops": f}
    w = case["workload"]
    dim = CONFIGS[w]["n_species"] + 1
    c = _per(w, case.get("cv", False))
    if kind == "rhs":
        return {"bytes": n * 8.0 * (2 * dim + 1), "flops": n * c["rhs_flops"]}
    if kind == "jacobian":
        return {"bytes": n * 8.0 * (dim * dim + dim + 1), "flops": n * c["ros4_jeval_flops"]}
    if kind == "newton":
        return {"bytes": n * (16.0 * dim * dim + 16.0 * dim + 4.0 * dim + 4.0),
                "flops": n * (c["lu_flops"] + c["solve_flops"])}
    steps = STEPS[w, kind]
    if kind == "rkf45":
        per = c["rkf45_step_flops"]
    elif case["jac"]:
        per = c["ros4_fd_jeval_flops"] + c["ros4_attempt_flops"]
    else:
        per = c["ros4_step_flops"]
    return {"bytes": n * (16.0 * dim + 20.0), "flops": n * steps * per}


# ------------------------------------------------------------------ the formulas in torch, FP64
R_GAS, P_STD = 8.314462618, 101325.0


class _Plain:
    """A mechanism's arrays on the GPU."""

    def __init__(self, workload):
        m = _mech(workload)
        S = len(m["mw"])
        t = {k: _dev(np.asarray(m[k])) for k in ("mw", "nasa", "tmid", "arrh", "arrh0", "rtype", "rev")}
        self.W, self.nasa, self.tmid = t["mw"], t["nasa"], t["tmid"]
        self.arrh, self.arrh0, self.rtype = t["arrh"], t["arrh0"], t["rtype"]
        self.reversible = (t["rev"] != 0).to(F8)
        pad = lambda a: _dev(np.where(a < 0, S, a).astype(np.int64))  # noqa: E731  (slot S holds 1)
        self.reac, self.prod = pad(m["reac"]), pad(m["prod"])
        R = len(m["rtype"])
        nr, npr = np.zeros((R, S + 1)), np.zeros((R, S + 1))
        for s in range(3):
            np.add.at(nr, (np.arange(R), np.where(m["reac"][:, s] < 0, S, m["reac"][:, s])), 1.0)
            np.add.at(npr, (np.arange(R), np.where(m["prod"][:, s] < 0, S, m["prod"][:, s])), 1.0)
        nu = npr[:, :S] - nr[:, :S]
        self.nu = _dev(nu)                       # [R, S]
        self.dnu = _dev(nu.sum(axis=1))
        eff = np.ones((R, S))
        for i in range(R):
            for e in range(m["eff_ptr"][i], m["eff_ptr"][i + 1]):
                eff[i, m["eff_sp"][e]] = m["eff_val"][e]
        self.eff = _dev(eff)


def _rhs(m, cv, p, y):
    """f(y) = (dT/dt, dY/dt): mass action with K_c from the NASA-7 fits,
    third bodies and Lindemann fall-off, at constant pressure or volume."""
    T, Y = y[:, :1], y[:, 1:]
    lnT = torch.log(T)
    a = torch.where((T < m.tmid).unsqueeze(-1), m.nasa[:, 0], m.nasa[:, 1])  # [N, S, 7]
    a1, a2, a3, a4, a5, a6, a7 = a.unbind(-1)
    cp = a1 + T * (a2 + T * (a3 + T * (a4 + T * a5)))
    h = a1 + T * (a2 / 2 + T * (a3 / 3 + T * (a4 / 4 + T * a5 / 5))) + a6 / T
    g = a1 * lnT + T * (a2 + T * (a3 / 2 + T * (a4 / 3 + T * a5 / 4))) + a7 - h  # (S/R - H/RT)
    rho = p[:, None] if cv else p[:, None] / (R_GAS * T * (Y / m.W).sum(1, keepdim=True))
    X = rho * Y / m.W
    X1 = torch.cat([X, torch.ones_like(T)], 1)
    fwd = X1[:, m.reac[:, 0]] * X1[:, m.reac[:, 1]] * X1[:, m.reac[:, 2]]
    bwd = X1[:, m.prod[:, 0]] * X1[:, m.prod[:, 1]] * X1[:, m.prod[:, 2]]
    lnk = torch.log(m.arrh[:, 0]) + m.arrh[:, 1] * lnT - m.arrh[:, 2] / (R_GAS * T)
    lnkc = g @ m.nu.T + m.dnu * torch.log(P_STD / (R_GAS * T))
    net = torch.exp(lnk) * fwd - m.reversible * torch.exp(lnk - lnkc) * bwd
    M = X @ m.eff.T
    fall = m.rtype == 2
    lnk0 = torch.where(fall, torch.log(torch.where(fall, m.arrh0[:, 0], 1.0)) + m.arrh0[:, 1] * lnT
                       - m.arrh0[:, 2] / (R_GAS * T), lnk)
    pr = torch.exp(lnk0 - lnk) * M
    q = net * torch.where(m.rtype == 1, M, torch.where(fall, pr / (1 + pr), 1.0))
    w = q @ m.nu
    off = 1.0 if cv else 0.0  # u = h - RT and c_v = c_p - R at constant volume
    dT = -T * ((h - off) * w).sum(1, keepdim=True) / (rho * ((cp - off) * Y / m.W).sum(1, keepdim=True))
    return torch.cat([dT, w * m.W / rho], 1)


def _jac(m, cv, p, y):
    cols = []
    for j in range(y.shape[1]):
        e = torch.zeros_like(y)
        e[:, j] = 1.0
        cols.append(torch.func.jvp(lambda s: _rhs(m, cv, p, s), (y,), (e,))[1])
    return torch.stack(cols, 2)


def _by_rows(f, p, y, rows):
    return torch.cat([f(p[i:i + rows], y[i:i + rows]) for i in range(0, len(y), rows)])


# Fehlberg 4(5): stages, propagated weights, error weights.
RK_A = ((), (1 / 4,), (3 / 32, 9 / 32), (1932 / 2197, -7200 / 2197, 7296 / 2197),
        (439 / 216, -8, 3680 / 513, -845 / 4104), (-8 / 27, 2, -3544 / 2565, 1859 / 4104, -11 / 40))
RK_B = (25 / 216, 0, 1408 / 2565, 2197 / 4104, -1 / 5, 0)
RK_E = (16 / 135 - 25 / 216, 0, 6656 / 12825 - 1408 / 2565, 28561 / 56430 - 2197 / 4104, -9 / 50 + 1 / 5, 2 / 55)
RTOL, ATOL = 1e-9, 1e-12


def _sum(c, k, base=0.0):
    for a, v in zip(c, k):
        base = base + a * v
    return base


def _rkf45_step(m, cv, p, y, h):
    k = []
    for a in RK_A:
        k.append(h * _rhs(m, cv, p, _sum(a, k, y)))
    return _sum(RK_B, k, y), _sum(RK_E, k)


def _norm(v, scale):
    return (v / scale).square().mean(1).sqrt()


def _rkf45(m, cv, p, y, dt):
    """Adaptive steps over dt, every reactor with its own step size."""
    y, n = y.clone(), len(y)
    f0 = _rhs(m, cv, p, y)
    sc = ATOL + RTOL * y.abs()
    d0, d1 = _norm(y, sc), _norm(f0, sc)
    ha = torch.where((d0 < 1e-5) | (d1 < 1e-5), 1e-6, 0.01 * d0 / d1)
    d2 = _norm(_rhs(m, cv, p, y + ha[:, None] * f0) - f0, sc) / ha
    dm = torch.maximum(d1, d2)
    hb = torch.where(dm <= 1e-15, torch.clamp(ha * 1e-3, min=1e-6), (0.01 / dm) ** 0.2)
    h = torch.minimum(100 * ha, hb).clamp(max=dt)
    t = torch.zeros(n, dtype=F8, device=DEV)
    after = torch.zeros(n, dtype=torch.bool, device=DEV)  # the last attempt was rejected
    live = torch.arange(n, device=DEV)
    while len(live):
        yl, left = y[live], dt - t[live]
        last = h[live] >= left
        hh = torch.where(last, left, h[live])
        yn, e = _rkf45_step(m, cv, p[live], yl, hh[:, None])
        err = _norm(e, ATOL + RTOL * torch.maximum(yl.abs(), yn.abs()))
        ok = (err < 1) & yn.isfinite().all(1)
        # a trial state that is not finite is rejected with the smallest factor
        fac = torch.where(yn.isfinite().all(1) & err.isfinite(), torch.clamp(0.9 * err ** -0.2, 0.2, 5.0), 0.2)
        y[live] = torch.where(ok[:, None], yn, yl)
        t[live] = torch.where(ok, torch.where(last, dt, t[live] + hh), t[live])
        h[live] = hh * torch.where(after[live] & ok, fac.clamp(max=1.0), fac)
        after[live] = ~ok
        live = live[t[live] < dt]
    return y


def exact(case, seed):
    rng = np.random.default_rng(seed)
    kind, n = case["kind"], case["n"]
    if kind == "mixed":
        return None
    if kind == "newton":
        a, b = _newton_inputs(case, rng)
        lu, piv = torch.linalg.lu_factor(a)
        return [lu, torch.linalg.lu_solve(lu, piv, b.unsqueeze(-1)).squeeze(-1), None, None]
    w, cv = case["workload"], case["cv"]
    m = _Plain(w)
    y, p = _states(w, n, cv, rng)
    if kind == "rhs":
        return _by_rows(lambda q, s: _rhs(m, cv, q, s), p, y, 16384)
    if kind == "jacobian":
        return _by_rows(lambda q, s: _jac(m, cv, q, s), p, y, 1024)
    if kind == "rkf45":
        return [_rkf45(m, cv, p, y, DT[w, kind]), None]
    return None  # ROS4: thousands of small steps with a Jacobian each
