"""The branches that the sizes and values of a call choose, against the oracle.

* Right-hand sides go to one team or one thread a reactor by batch size, and
  take products of concentrations and Gibbs factors in integer arithmetic
  while every factor is in range; a zero, tiny or negative mass fraction or an
  extreme temperature sends a reactor (team) or a warp (thread) the other way.
* A mechanism with more reactions than a team's scratch holds is walked in
  several chunks.

Tolerances: right-hand sides and Jacobians within 1e-12 of max(|oracle|, gross)
(the same sums with every term in absolute value), states within 1e-6 relative
in T and 1e-8 in Y, as in the parity tests.
"""
import numpy as np
import pytest

from synth.configs import CONFIGS, load_mechanism, reactor_states
from oracle import ORA_ROS4, OracleMech

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def ck():
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    import paper_1608_05794_gb300.ck as ck
    return ck


def _dev(a):
    return torch.as_tensor(np.array(a, dtype=np.float64), device="cuda")


def _close(a, b, gross):
    return np.all(np.abs(a - b) <= 1e-12 * np.maximum(np.abs(b), gross) + 1e-20)


def _states(name, n):
    """Reactor states whose first rows leave the integer products' ranges."""
    y, p = reactor_states(name, n=n, seed_offset=41)
    edits = [(0, 1, 0.0), (1, 2, 1e-120), (2, 3, -1e-15), (3, 1, 1e-91), (4, 2, -0.0), (5, 0, 320.0), (6, 0, 3400.0)]
    for row, col, v in edits:
        if row < n:
            y[row, col] = v
    return y, p


# one team a reactor below 26 (10 species), 512 (53) reactors an SM, always for 111
@pytest.mark.parametrize("name,n", [("small", 1), ("small", 9), ("small", 152 * 26 + 1), ("small", 152 * 256 + 33),
                                    ("medium", 9), ("medium", 152 * 512 + 33), ("large", 9), ("large", 400)])
def test_rhs_by_batch_size_and_range(ck, name, n):
    m = load_mechanism(CONFIGS[name]["mech"])
    gm, om = ck.load_mechanism(m), OracleMech(m)
    y, p = _states(name, n)
    yd, out = _dev(y), torch.empty((n, y.shape[1]), dtype=torch.float64, device="cuda")
    ck.rhs(gm, _dev(p), yd, out)
    rows = np.unique(np.r_[0:min(n, 40), max(0, n - 40):n])
    f = out[torch.as_tensor(rows, device="cuda")].cpu().numpy()
    assert _close(f, om.rhs(p[rows], y[rows]), om.rhs_gross(p[rows], y[rows]))


@pytest.mark.parametrize("name", ["small", "medium", "large"])
def test_jacobian_out_of_product_range(ck, name):
    m = load_mechanism(CONFIGS[name]["mech"])
    gm, om = ck.load_mechanism(m), OracleMech(m)
    y, p = _states(name, 8)
    nn = y.shape[1]
    out = torch.empty((8, nn, nn), dtype=torch.float64, device="cuda")
    ck.jacobian(gm, _dev(p), _dev(y), out)
    jo, gross = om.jacobian(p, y, gross=True)
    assert _close(out.cpu().numpy(), jo, gross)


@pytest.mark.parametrize("name,times", [("small", 40), ("medium", 2), ("medium", 3)])
def test_more_reactions_than_the_scratch(ck, name, times):
    # the mechanism's reactions several times over, at a rate smaller by as much
    m = dict(load_mechanism(CONFIGS[name]["mech"]))
    n_eff = len(m["eff_sp"])
    m["eff_ptr"] = np.concatenate([m["eff_ptr"][:-1] + k * n_eff for k in range(times)] + [[times * n_eff]]).astype(np.int32)
    for k in ("reac", "prod", "rtype", "rev", "arrh", "arrh0", "eff_sp", "eff_val"):
        m[k] = np.concatenate([m[k]] * times)
    m["arrh"] = m["arrh"] / np.array([times, 1.0, 1.0])
    m["arrh0"] = m["arrh0"] / np.array([times, 1.0, 1.0])
    gm, om = ck.load_mechanism(m), OracleMech(m)
    y, p = reactor_states(name, n=6, seed_offset=43)
    nn = y.shape[1]
    f = torch.empty((6, nn), dtype=torch.float64, device="cuda")
    j = torch.empty((6, nn, nn), dtype=torch.float64, device="cuda")
    ck.rhs(gm, _dev(p), _dev(y), f)
    ck.jacobian(gm, _dev(p), _dev(y), j)
    jo, gross = om.jacobian(p, y, gross=True)
    assert _close(f.cpu().numpy(), om.rhs(p, y), om.rhs_gross(p, y))
    assert _close(j.cpu().numpy(), jo, gross)
    dt = CONFIGS[name]["dt"] * 0.01
    ends = []
    for fn in (ck.integrate_ros4, ck.integrate_ros4_noalloc):
        yd, st = _dev(y), torch.empty(6, dtype=torch.int32, device="cuda")
        fn(gm, _dev(p), yd, _dev(np.full(6, dt)), st)
        torch.cuda.synchronize()
        ends.append(yd.cpu().numpy())
        assert (st.cpu().numpy() == 0).all()
    assert np.array_equal(*ends)
    yo = om.integrate(ORA_ROS4, p, y, dt)[0]
    assert np.max(np.abs(ends[0][:, 0] - yo[:, 0]) / yo[:, 0]) <= 1e-6
    assert np.max(np.abs(ends[0][:, 1:] - yo[:, 1:])) <= 1e-8


@pytest.mark.parametrize("cv", [0, 1])
def test_rkf45_threads_hand_reactors_to_teams(ck, cv):
    # reactors of more than 160 attempts move from their threads to teams,
    # which take every sum in the threads' order; the server's launches keep
    # them in threads: the same bits
    m = load_mechanism(CONFIGS["small"]["mech"])
    gm = ck.load_mechanism(m, reactor=cv)
    n = 200
    y, p = reactor_states("small", n=n, seed_offset=47)
    if cv:
        p = np.linspace(0.2, 2.5, n)
    dt = np.linspace(1e-6, 6e-5, n)
    opts = ck.SolverOpts.make(form=1)
    yd, st = _dev(y), torch.empty(n, dtype=torch.int32, device="cuda")
    steps, h = torch.empty((n, 2), dtype=torch.int32, device="cuda"), torch.zeros(n, dtype=torch.float64, device="cuda")
    ck.integrate_rkf45(gm, _dev(p), yd, _dev(dt), st, steps=steps, h_inout=h, opts=opts)
    torch.cuda.synchronize()
    total = steps.sum(1).cpu().numpy()
    assert (total > 160).sum() >= 20 and (total < 160).sum() >= 20
    srv = ck.Server(hbm_budget_bytes=1 << 30, streams=1)
    ys, ss = y.copy(), np.zeros((n, 2), np.int32)
    sts = np.zeros(n, np.int32)
    t = srv.submit(gm, ck.Server.RKF45, np.ascontiguousarray(p), ys, dt, sts, ss, opts)
    srv.wait(t)
    srv.release(t)
    srv.close()
    assert np.array_equal(yd.cpu().numpy(), ys)
    assert np.array_equal(steps.cpu().numpy(), ss) and np.array_equal(st.cpu().numpy(), sts)
    # a step limit inside and beyond the threads' share
    for limit in (100, 160, 161, 300):
        o = ck.SolverOpts.make(form=1, max_steps=limit)
        yl = _dev(y)
        ck.integrate_rkf45(gm, _dev(p), yl, _dev(dt), st, steps=steps, opts=o)
        assert np.array_equal(steps.sum(1).cpu().numpy(), np.minimum(total, limit))


def test_graph_of_a_freed_mechanism_is_not_replayed(ck):
    # a mechanism loaded after another was freed may get its handle's address;
    # a cached graph of the old one, whose tables are gone, must not match
    m = load_mechanism(CONFIGS["medium"]["mech"])
    y, p = reactor_states("medium", n=12, seed_offset=51)
    pd, rho, dt = _dev(p), _dev(np.linspace(0.3, 2.0, 12)), _dev(np.full(12, 1e-7))
    yd, st = _dev(y), torch.empty(12, dtype=torch.int32, device="cuda")
    par = torch.empty_like(pd)  # the same buffers in every call
    ends = []
    for cv in (0, 1, 0, 1):
        gm = ck.load_mechanism(m, reactor=cv)
        par.copy_(rho if cv else pd)
        yd.copy_(_dev(y))
        ck.integrate_groups(1, [dict(mech=gm, p=par, y=yd, dt=dt, status=st)], use_graph=True)
        torch.cuda.synchronize()
        yr = _dev(y)
        ck.integrate_rkf45(gm, par, yr, dt, st)
        assert torch.equal(yd, yr)
        ends.append(yr)
        gm.close()
    assert torch.equal(ends[0], ends[2]) and not torch.equal(ends[0], ends[1])
    ck.graph_cache_clear()
