"""Diagonal blocks of the mixed path at every cluster size (one, two or four
CTAs per block, by the number of problems): the factor of a problem does not
depend on it, bit for bit, lnL meets the oracle within the path's 1e-2, and
points that are not positive definite fail at the oracle's column, in any
block and row of the cluster, without touching the others."""

import numpy as np
import pytest

import oracle as O
from synth.instrument import random_problem

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def P():
    import paper_2501_12928_gb300 as P
    return P


def _like(P, p, T, nk):
    lk = P.Likelihood("mixed")
    lk.set_T(T, p["kbin"], nk, 2.0)
    lk.set_data(p["d"], p["noise_var"])
    lk.precompute()
    return lk


@pytest.mark.parametrize("n", [5, 128, 145, 300])
def test_factor_is_the_same_at_every_cluster_size(P, n):
    nk = 3 if n > 5 else 2
    p = random_problem(n + 40, n, nk, seed=n + 2)
    lk = _like(P, p, p["T"], nk)
    ph = np.random.default_rng(n).uniform(-2, 2, (160, nk))
    M = O.herm_dense(p["T"], p["noise_var"])
    db = O.dbar_dense(p["T"], p["noise_var"], p["d"])
    ref = O.evaluate(M, db, p["kbin"], ph[0], 2.0)["lnl"]
    base = None
    for B in (1, 36, 37, 38, 76, 77, 160):   # four CTAs per block up to 36 problems, two up to 76, one beyond
        lnl, st = lk.lnl(ph[:B])
        assert np.all(st == 0)
        assert abs(lnl[0] - ref) <= 1e-2
        f = lk.factor(0)
        base = f if base is None else base
        np.testing.assert_array_equal(f, base)


@pytest.mark.parametrize("col", [1, 15, 16, 40, 127, 129, 200])
def test_failing_pivot_at_every_cluster_size(P, col):
    """Columns 0 and col of T are equal (2 at one visibility of unit noise), the
    other columns do not see that visibility, and phi = 400 takes Phi^-1 of their
    k bin to 0: pivot col is 4 - 2 * 2 = 0 exactly."""
    p = random_problem(300, 210, 3, seed=9)
    T, nv, kbin = p["T"].copy(), p["noise_var"].copy(), p["kbin"].copy()
    T[0, :] = 0.0
    T[:, 0] = 0.0
    T[:, col] = 0.0
    T[0, 0] = T[0, col] = 2.0
    nv[0] = 1.0
    kbin[kbin == 0] = 1
    kbin[0] = kbin[col] = 0
    p.update(noise_var=nv, kbin=kbin)
    lk = _like(P, p, T, 3)
    good = np.array([0.3, -0.5, 1.0])
    ref = lk.lnl(good[None])[0][0]
    for B in (2, 50, 100):
        ph = np.repeat(good[None], B, axis=0)
        ph[B // 2, 0] = 400.0
        lnl, st = lk.lnl(ph)
        want = np.zeros(B, int)
        want[B // 2] = col + 1
        np.testing.assert_array_equal(st, want)
        assert lnl[B // 2] == -np.inf
        np.testing.assert_allclose(np.delete(lnl, B // 2), ref, rtol=1e-12)
