"""The float64-accurate residual at every group of problems (1, 2, 4, 8 or 16
per work item, a problem alone in two tiles per item) and every tile count per
item: a point's lnL does not depend on how many points it is evaluated with,
beyond the rounding of the float64 sums across tiles, and meets the oracle
within the path's 1e-2."""

import numpy as np
import pytest

import oracle as O
from synth.instrument import random_problem

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def like():
    import paper_2501_12928_gb300 as P
    made = {}

    def make(n, nk=3):
        if n not in made:
            p = random_problem(n + 60, n, nk, seed=n)
            lk = P.Likelihood("mixed")
            lk.set_T(p["T"], p["kbin"], nk, 2.0)
            lk.set_data(p["d"], p["noise_var"])
            lk.precompute()
            made[n] = (lk, p)
        return made[n]
    return make


@pytest.mark.parametrize("n", [60, 130, 700])
def test_lnl_does_not_depend_on_the_group(like, n):
    lk, p = like(n)
    ph = np.random.default_rng(n).uniform(-2, 2, (33, 3))
    alone = np.array([lk.lnl(q[None])[0][0] for q in ph])
    for B in (2, 3, 4, 5, 8, 9, 16, 17, 33):
        lnl, st = lk.lnl(ph[:B])
        assert np.all(st == 0)
        np.testing.assert_allclose(lnl, alone[:B], rtol=1e-12)
    M, db = O.herm_dense(p["T"], p["noise_var"]), O.dbar_dense(p["T"], p["noise_var"], p["d"])
    for i in (0, 32):
        assert abs(alone[i] - O.evaluate(M, db, p["kbin"], ph[i], 2.0)["lnl"]) <= 1e-2


def test_lnl_with_several_tiles_per_item(like):
    lk, _ = like(1100)
    ph = np.random.default_rng(4).uniform(-2, 2, (3, 3))
    alone = np.array([lk.lnl(q[None])[0][0] for q in ph])
    lnl, st = lk.lnl(np.tile(ph, (200, 1)))   # 9 block rows x 3 groups of four tiles x 38 groups of problems
    assert np.all(st == 0)
    np.testing.assert_allclose(lnl.reshape(200, 3), np.tile(alone, (200, 1)), rtol=1e-12)
