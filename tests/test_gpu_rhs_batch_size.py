"""ck_rhs gives a reactor the same bits in a batch of any size: up to 64 species
small batches go to one team a reactor, large ones to one thread a reactor,
which add every sum in the same order, a species that fills several slots of a
reaction at once.
"""
import numpy as np
import pytest

from synth.configs import CONFIGS, load_mechanism, reactor_states

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu


def _copies(m, copies, times):
    """A mechanism of copies of m side by side, its reactions several times over."""
    S, n_eff = len(m["mw"]), len(m["eff_sp"])
    reps = copies * times
    shift = lambda a, i: np.where(a < 0, -1, a + i * S)  # noqa: E731
    out = {k: np.concatenate([m[k]] * copies) for k in ("mw", "nasa", "tmid")}
    out.update({k: np.concatenate([m[k]] * reps) for k in ("rtype", "rev", "arrh", "arrh0", "eff_val")})
    out.update({k: np.concatenate([shift(m[k], i % copies) for i in range(reps)]) for k in ("reac", "prod")})
    out["eff_sp"] = np.concatenate([m["eff_sp"] + (i % copies) * S for i in range(reps)])
    out["eff_ptr"] = np.concatenate([m["eff_ptr"][:-1] + i * n_eff for i in range(reps)] + [[reps * n_eff]])
    return out


def _patterns(m):
    """m's species with reactions in which they fill several slots, on one side and on both."""
    rng = np.random.default_rng(5)
    S, R = len(m["mw"]), 240
    reac, prod = -np.ones((R, 3), np.int32), -np.ones((R, 3), np.int32)
    for i in range(R):
        nr, npr = 1 + i % 3, 1 + i // 3 % 3
        few = rng.choice(S, 3, replace=False)
        reac[i, :nr], prod[i, :npr] = rng.choice(few, nr), rng.choice(few if i % 2 else S, npr)
    out = {k: m[k] for k in ("mw", "nasa", "tmid")}
    arrh = np.stack([10.0 ** rng.uniform(0, 3, R), rng.uniform(-1, 1, R), rng.uniform(0, 5e4, R)], 1)
    out.update(reac=reac, prod=prod, arrh=arrh, arrh0=arrh * [1e2, 1, 1], rtype=(np.arange(R) % 5 // 3 * (1 + np.arange(R) % 2)).astype(np.int32),
               rev=(np.arange(R) % 7 > 2).astype(np.int32), eff_ptr=np.zeros(R + 1, np.int32), eff_sp=np.zeros(0, np.int32), eff_val=np.zeros(0))
    return out


# (workload, copies, times over): 10, 20, 30 (the latency form), 40, 53 and 60
# species (96 threads), 10 and 40 species with more reactions than a chunk, 10
# with more than a team's rates have room for; and slots filled by one species
@pytest.mark.parametrize("name,copies,times", [("small", 1, 1), ("small", 2, 3), ("small", 3, 1), ("small", 4, 1),
                                               ("medium", 1, 1), ("small", 6, 1), ("small", 1, 40), ("small", 4, 12),
                                               ("small", 1, 400), ("small", 0, 0)])
@pytest.mark.parametrize("cv", [0, 1])
def test_bits_do_not_depend_on_the_batch(name, copies, times, cv):
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    import paper_1608_05794_gb300.ck as ck
    sms = torch.cuda.get_device_properties(0).multi_processor_count
    m = load_mechanism(CONFIGS[name]["mech"])
    made = _copies(m, copies, times) if copies else _patterns(m)
    copies = max(copies, 1)
    gm = ck.load_mechanism(made, check_atoms=False, reactor=cv)
    y, p = reactor_states(name, n=40, seed_offset=71)
    # rows out of the ranges of the integer products: zero, tiny, negative
    for row, col, v in [(0, 1, 0.0), (1, 2, 1e-120), (2, 3, -1e-15), (3, 1, -0.0), (4, 0, 320.0), (5, 0, 3400.0)]:
        y[row, col] = v
    y = np.concatenate([y[:, :1]] + [y[:, 1:] / copies] * copies, axis=1)
    if cv:
        p = np.linspace(0.2, 2.5, len(p))
    few, pf = (torch.as_tensor(np.ascontiguousarray(a), device="cuda") for a in (y, p))
    out = torch.empty_like(few)
    ck.rhs(gm, pf, few, out)
    assert torch.isfinite(out[6:]).all()
    most = 40 if times == 400 else 520
    for per_sm in (most // 20, most):  # teams; threads
        reps = per_sm * sms // len(few) + 1
        many, pm = few.repeat(reps, 1), pf.repeat(reps)
        outs = torch.empty_like(many)
        ck.rhs(gm, pm, many, outs)
        same = outs.view(torch.int64).view(reps, *few.shape) == out.view(torch.int64)
        assert bool(same.all()), (per_sm, (~same).nonzero()[:4].tolist())
