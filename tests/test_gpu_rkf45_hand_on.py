"""The thread-per-reactor RKF45 hands reactors to teams only where its warps
have run out of others; the server's launches never do, and give the same bits.
"""
import time

import numpy as np
import pytest

from synth.configs import CONFIGS, load_mechanism, reactor_states

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


def _both(ck, n, dt, opts, repeats=1, times=1):
    """States, step counts and the best time of the call and of threads alone;
    times: the mechanism's reactions several times over, at lower rates."""
    m = load_mechanism(CONFIGS["small"]["mech"])
    n_eff = len(m["eff_sp"])
    m["eff_ptr"] = np.concatenate([m["eff_ptr"][:-1] + i * n_eff for i in range(times)] + [[times * n_eff]])
    for k in ("reac", "prod", "rtype", "rev", "arrh", "arrh0", "eff_sp", "eff_val"):
        m[k] = np.concatenate([m[k]] * times)
    for k in ("arrh", "arrh0"):
        m[k] = m[k] / np.array([times, 1.0, 1.0])
    gm = ck.load_mechanism(m)
    y, p = reactor_states("small", n=n, seed_offset=61)
    y0, pd, dtd = _dev(y), _dev(p), _dev(dt)
    st = torch.empty(n, dtype=torch.int32, device="cuda")
    srv = ck.Server(hbm_budget_bytes=4 << 30, streams=1, chunk_reactors=n)
    out = []
    for server in (False, True):
        best = np.inf
        for _ in range(repeats + 1):
            yd, steps = y0.clone(), torch.zeros((n, 2), dtype=torch.int32, device="cuda")
            torch.cuda.synchronize()
            t0 = time.perf_counter()
            if server:
                t = srv.submit(gm, ck.Server.RKF45, pd, yd, dtd, st, steps, opts)
                srv.wait(t)
                srv.release(t)
            else:
                ck.integrate_rkf45(gm, pd, yd, dtd, st, steps=steps, opts=opts)
            torch.cuda.synchronize()
            best = min(best, time.perf_counter() - t0)
        out.append((yd.cpu().numpy(), steps.cpu().numpy(), best))
    srv.close()
    return out


def test_full_warps_keep_reactors_of_many_steps(ck):
    # every reactor takes 400 steps: teams, which take a fifth of the steps of
    # full warps, had most of them after the first 160
    n = 100000
    (y, steps, t), (ys, ss, ts) = _both(ck, n, np.full(n, 4e-7), ck.SolverOpts.make(form=1, fixed_h=1e-9), repeats=2)
    assert (steps.sum(1) >= 400).all()
    assert np.array_equal(y, ys) and np.array_equal(steps, ss)
    assert t < 1.5 * ts


# 20 reactions: teams in the latency form; 80 in the general one
@pytest.mark.parametrize("times", [1, 4])
@pytest.mark.parametrize("n", [1, 8, 9, 33, 129, 5000])
def test_same_bits_wherever_a_reactor_is_finished(ck, n, times):
    (y, steps, _), (ys, ss, _) = _both(ck, n, np.geomspace(1e-7, 1e-5, n), ck.SolverOpts.make(form=1), times=times)
    assert np.array_equal(y, ys) and np.array_equal(steps, ss)
