"""ck_lu_factor on batches in which pivots fail: a zero, infinite or NaN pivot
in every position, between regular matrices.  Most CTAs factor several
matrices one after another, so a team that left a failed factorization out of
step would spoil the next one.

The matrices are L U with entries that make every multiplier and update exact
in FP64 (U's diagonal powers of two, L's entries +-1/4 and +-1/2, small whole
numbers above), so factors are compared by value.
"""
import numpy as np
import pytest

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu


def _factors(rng, n):
    low = np.tril(rng.choice([0.0, 0.0, 0.25, -0.25, 0.5], size=(n, n)), -1)
    up = np.triu(rng.integers(-2, 3, size=(n, n)).astype(float), 1) * 4.0
    up[np.arange(n), np.arange(n)] = rng.choice([16.0, -32.0], size=n)
    return low, up


def _product(low, up):
    a = low @ up + up
    assert np.array_equal(a, np.round(a * 4) / 4) and np.abs(a).max() < 2.0**40  # exact
    return a


# a warp alone, teams of 4 and of 8 warps, at the edges of their ranges
@pytest.mark.parametrize("n", [2, 11, 24, 25, 54, 64, 65, 112, 128])
def test_failing_pivots_between_regular_matrices(n):
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    import paper_1608_05794_gb300.ck as ck
    rng = np.random.default_rng(n)
    low, up = _factors(rng, n)
    good = _product(low, up)
    kinds, mats = [], []
    for k in range(n):
        zero = up.copy()
        zero[k, k] = 0.0
        kinds.append(k + 1)
        mats.append(_product(np.where(np.arange(n)[None, :] == k, 0.0, low), zero))
        for v in (np.inf, np.nan):
            a = good.copy()
            a[n - 1, k] = v
            kinds.append(k + 1)
            mats.append(a)
    kinds, mats = np.array([0] + kinds), np.array([good] + mats)
    batch = 152 * 12 * 4
    which = np.where(rng.random(batch) < 0.5, 0, rng.integers(1, len(kinds), batch))
    a = torch.as_tensor(mats, device="cuda")[torch.as_tensor(which, device="cuda")].contiguous()
    piv = torch.empty((batch, n), dtype=torch.int32, device="cuda")
    info = torch.empty(batch, dtype=torch.int32, device="cuda")
    ck.lu_factor(a, piv, info)
    assert np.array_equal(info.cpu().numpy(), kinds[which])
    regular = torch.as_tensor(which == 0, device="cuda")
    want = torch.as_tensor(low + up, device="cuda")
    assert bool((a[regular] == want).all())
    assert bool((piv[regular] == torch.arange(n, dtype=torch.int32, device="cuda")).all())
    # up to the failed pivot the factors are those of the regular matrix
    left = torch.as_tensor(kinds[which] - 1, device="cuda")
    j = torch.arange(n, device="cuda")
    done = (left >= 0)[:, None, None] & (torch.minimum(j[:, None], j[None, :])[None] < left[:, None, None])
    last = torch.zeros((n, n), dtype=torch.bool, device="cuda")
    last[n - 1] = True  # (the row that carried the infinity or NaN)
    same = (a == want) | last | ~done
    same |= (j[None, None, :] == left[:, None, None])  # the failed column
    assert bool(same.all())
