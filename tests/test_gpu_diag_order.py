"""Float64 diagonal blocks at every cluster size (eight CTAs per block up to 15
problems, four up to 36, two up to 76, one beyond): the operations on an element
do not depend on it, so lnL and the factor are the same bits; a point that is not
positive definite fails at its column without touching the others."""

import numpy as np
import pytest

import oracle as O
from synth.instrument import random_problem

pytestmark = pytest.mark.gpu


def _like(p, T, nk, precision):
    import paper_2501_12928_gb300 as P

    lk = P.Likelihood(precision)
    lk.set_T(T, p["kbin"], nk, 2.0)
    lk.set_data(p["d"], p["noise_var"])
    lk.precompute()
    return lk


@pytest.mark.parametrize("n", [5, 128, 145, 300])
def test_same_bits_at_every_cluster_size(n):
    nk = 3 if n > 5 else 2
    p = random_problem(n + 40, n, nk, seed=n + 3)
    lk = _like(p, p["T"], nk, "fp64")
    ph = np.random.default_rng(n).uniform(-2, 2, (90, nk))
    M, db = O.herm_dense(p["T"], p["noise_var"]), O.dbar_dense(p["T"], p["noise_var"], p["d"])
    ref = O.evaluate(M, db, p["kbin"], ph[0], 2.0)["lnl"]
    base = None
    for B in (1, 15, 16, 36, 37, 76, 77, 90):
        lnl, st = lk.lnl(ph[:B])
        assert np.all(st == 0)
        assert abs(lnl[0] - ref) <= 1e-9 * abs(ref)
        f = lk.factor(0)
        base = (f, lnl[0]) if base is None else base
        np.testing.assert_array_equal(f, base[0])
        assert lnl[0] == base[1]


@pytest.mark.parametrize("precision", ["fp64", "mean"])
@pytest.mark.parametrize("col", [1, 15, 16, 40, 127, 129, 200])
def test_failing_pivot(precision, col):
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
    lk = _like(p, T, 3, "mixed" if precision == "mean" else precision)
    good, bad = np.array([0.3, -0.5, 1.0]), np.array([400.0, -0.5, 1.0])
    if precision == "mean":
        assert lk.posterior_mean(bad)[1] == col + 1
        assert lk.posterior_mean(good)[1] == 0
        return
    for B in (2, 30, 50, 80):
        ph = np.repeat(good[None], B, axis=0)
        ph[B // 2] = bad
        lnl, st = lk.lnl(ph)
        want = np.zeros(B, int)
        want[B // 2] = col + 1
        np.testing.assert_array_equal(st, want)
        assert lnl[B // 2] == -np.inf and np.ptp(np.delete(lnl, B // 2)) == 0
