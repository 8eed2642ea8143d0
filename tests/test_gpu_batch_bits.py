"""A reactor's result does not depend on the batch it is in: the batch chooses
the width and the form of the teams and how many reactions they take at a time,
all of which keep the order of every sum.
"""
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


def _sms():
    return torch.cuda.get_device_properties(0).multi_processor_count if torch.cuda.is_available() else 1


def _inputs(ck, name, n, cv=0):
    """The first eight reactors over and over."""
    gm = ck.load_mechanism(load_mechanism(CONFIGS[name]["mech"]), reactor=cv)
    y, p = reactor_states(name, n=8, seed_offset=83)
    if cv:
        p = np.linspace(0.3, 2.0, 8)
    rows = np.arange(n) % 8
    return gm, torch.as_tensor(y[rows], device="cuda"), torch.as_tensor(p[rows], device="cuda"), rows


# one reactor an SM (all rates at once), four (the latency form), then neither
@pytest.mark.parametrize("name,per_sm,dt", [("small", 4, 3e-6), ("medium", 1, 1e-7), ("large", 1, 3e-7)])
@pytest.mark.parametrize("opts", [{}, dict(precision=1), dict(jac=1), dict(team=16)])
def test_ros4(ck, name, per_sm, dt, opts):
    if opts.get("jac"):
        dt *= 0.2
    outs = []
    for n in (8, per_sm * _sms(), per_sm * _sms() + 1):
        gm, y, p, rows = _inputs(ck, name, n)
        st, steps = torch.empty(n, dtype=torch.int32, device="cuda"), torch.zeros((n, 2), dtype=torch.int32, device="cuda")
        h = torch.zeros(n, dtype=torch.float64, device="cuda")
        ck.integrate_ros4(gm, p, y, torch.full((n,), dt, dtype=torch.float64, device="cuda"), st, steps=steps, h_inout=h,
                          opts=ck.SolverOpts.make(**opts))
        assert int(steps.sum(1).min()) > 0
        for a in (y, steps, h, st):
            assert torch.equal(a, a[:8][torch.as_tensor(rows, device="cuda")])
        outs.append([a[:8].clone() for a in (y, steps, h, st)])
    for other in outs[1:]:
        assert all(torch.equal(a, b) for a, b in zip(outs[0], other))


@pytest.mark.parametrize("name", ["small", "medium", "large"])
@pytest.mark.parametrize("cv", [0, 1])
def test_forward_difference_jacobian(ck, name, cv):
    outs = []
    for n in (8, _sms(), _sms() + 1):
        gm, y, p, rows = _inputs(ck, name, n, cv)
        out = torch.empty((n, y.shape[1], y.shape[1]), dtype=torch.float64, device="cuda")
        ck.jacobian_fd(gm, p, y, torch.full((n,), 1e-8, dtype=torch.float64, device="cuda"), out)
        assert torch.equal(out, out[:8][torch.as_tensor(rows, device="cuda")])
        outs.append(out[:8].clone())
    assert torch.equal(outs[0], outs[1]) and torch.equal(outs[0], outs[2])


# 64 and 128 threads, and the latency form
@pytest.mark.parametrize("name,n", [("small", 700), ("medium", 12 * 152), ("large", 600)])
def test_rkf45_teams(ck, name, n):
    outs = []
    for m, opts in ((8, {}), (n, {}), (n, dict(variant=2)), (3 * n, {})):
        gm, y, p, rows = _inputs(ck, name, m)
        st = torch.empty(m, dtype=torch.int32, device="cuda")
        ck.integrate_rkf45(gm, p, y, torch.full((m,), 3e-7, dtype=torch.float64, device="cuda"), st,
                           opts=ck.SolverOpts.make(form=2, **opts))
        assert torch.equal(y, y[:8][torch.as_tensor(rows, device="cuda")])
        outs.append(y[:8].clone())
    assert all(torch.equal(outs[0], o) for o in outs[1:])


# one, two and more warps a matrix, at the sizes where they change
@pytest.mark.parametrize("dim", [1, 2, 24, 25, 40, 41, 54, 128])
def test_lu_and_solve(ck, dim):
    rng = np.random.default_rng(dim)
    a0 = rng.standard_normal((8, dim, dim)) + 2.0 * np.eye(dim)
    b0 = rng.standard_normal((8, dim))
    outs = []
    for n in (8, 8 * _sms(), 8 * _sms() + 1):
        rows = np.arange(n) % 8
        a, b = (torch.as_tensor(v[rows], device="cuda") for v in (a0, b0))
        piv, info = (torch.empty(s, dtype=torch.int32, device="cuda") for s in ((n, dim), (n,)))
        ck.lu_factor(a, piv, info)
        ck.lu_solve(a, piv, b)
        for v in (a, b, piv, info):
            assert torch.equal(v, v[:8][torch.as_tensor(rows, device="cuda")])
        outs.append([v[:8].clone() for v in (a, b, piv, info)])
    for other in outs[1:]:
        assert all(torch.equal(u, v) for u, v in zip(outs[0], other))
    assert int(outs[0][3].abs().sum()) == 0
    x = np.linalg.solve(a0, b0[:, :, None])[:, :, 0]
    assert np.abs(outs[0][1].cpu().numpy() - x).max() <= 1e-12 * np.linalg.cond(a0).max() * np.abs(x).max()
