"""Triangular solves of small batches (a step's block in every CTA) and of large
ones (in one CTA): the same bits, at sizes of one block to several with a ragged
last one, alone and with problems of other sizes beside them."""

import numpy as np
import pytest

from synth.instrument import random_problem

pytestmark = pytest.mark.gpu


def _like(P, n, nk, precision):
    p = random_problem(n + 40, n, nk, seed=n + 5)
    lk = P.Likelihood(precision)
    lk.set_T(p["T"], p["kbin"], nk, 2.0)
    lk.set_data(p["d"], p["noise_var"])
    lk.precompute()
    return lk


@pytest.mark.parametrize("n", [3, 128, 129, 300, 520])
def test_quadratic_form_is_the_same_in_small_and_large_batches(n):
    """Float64: every step of lnL has one order, so the batch must not show."""
    import paper_2501_12928_gb300 as P

    lk = _like(P, n, 2, "fp64")
    ph = np.random.default_rng(n).uniform(-2, 2, (160, 2))
    small, st = lk.lnl(ph[:1])
    large, st2 = lk.lnl(ph)
    assert st[0] == 0 and np.all(st2 == 0)
    assert small[0] == large[0]


@pytest.mark.parametrize("precision,rtol", [("fp64", 0.0), ("mixed", 1e-10)])
def test_problems_of_several_sizes(precision, rtol):
    """Problems that end (and, backward, begin) at different steps, in a batch on
    either side of the rule.  Mixed: the residual's sums are split by the batch,
    which moves the correction of the quadratic form by its rounding only."""
    import paper_2501_12928_gb300 as P

    likes = [_like(P, n, 2, precision) for n in (3, 300, 129)]
    rng = np.random.default_rng(11)
    phis = [rng.uniform(-2, 2, (b, 2)) for b in (70, 60, 50)]
    large, sl = P.lnl_multi(likes, phis)
    small, ss = P.lnl_multi(likes, [ph[:2] for ph in phis])
    for a, b, sa, sb in zip(large, small, sl, ss):
        assert np.all(sa == 0) and np.all(sb == 0)
        np.testing.assert_allclose(a[:2], b, rtol=rtol, atol=0)
