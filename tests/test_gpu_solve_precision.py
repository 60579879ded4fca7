"""lnL's triangular solves apply the inverse diagonal blocks in float64.

Sigma = (1 + 2^-30) I: the inverse blocks are known to 2^-62 and the right-hand side
is exact, so that x~ carries the two roundings of its two passes, 2^-53 each at
most, and the residual beside it nothing above 2^-77 (d - x is exact, M x is 2^-30 of
it).  Each component of the right-hand side is 2^-49 from the next pair of float32
numbers, relative to itself, which a solve in such pairs would lose."""

import numpy as np
import pytest

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("n, B", [(1, 1), (100, 1), (128, 1), (128, 40), (300, 1), (300, 60)])
def test_solve_keeps_the_right_hand_side(n, B):
    import paper_2501_12928_gb300 as P

    rng = np.random.default_rng(n)
    # 1 + r, 2^-25 <= r < 2^-24 halfway between two float32 numbers
    part = lambda: rng.choice([-1.0, 1.0], n) * (1.0 + rng.integers(1 << 23, (1 << 24) - 1, n) * 2.0 ** -48 + 2.0 ** -49)
    dbar = part() + 1j * part()
    lo = dbar.real - dbar.real.astype(np.float32)
    assert np.all(np.abs(lo - lo.astype(np.float32)) == 2.0 ** -49)
    lk = P.Likelihood("mixed")
    lk.set_T(2.0 ** -15 * np.eye(n, dtype=np.complex128), np.zeros(n, np.int32), 1, 1.0)
    lk.set_data(2.0 ** 15 * dbar, np.ones(n))
    lk.precompute()
    np.testing.assert_array_equal(lk.get_dbar(), dbar)
    lnl, st = lk.lnl(np.zeros((B, 1)))
    assert np.all(st == 0)
    assert lk.stats()["resid_rel_max"] <= 1.05 * 2.0 ** -52
