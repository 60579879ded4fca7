"""A new data set on an instrument that has been evaluated before: the batch's
buffers and graph are taken up again, and must give what a fresh context gives,
bit for bit; until the next evaluation the old one's results are out of reach."""

import numpy as np
import pytest

from synth.instrument import random_problem

pytestmark = pytest.mark.gpu


def _like(P, p, precision, seed=None):
    lk = P.Likelihood(precision)
    lk.set_T(p["T"], p["kbin"], 3, 2.0)
    _data(lk, p, seed)
    return lk


def _data(lk, p, seed):
    rng = np.random.default_rng(seed)
    d = p["d"] * rng.uniform(0.5, 2.0, p["d"].shape)
    lk.set_data(d, p["noise_var"] * rng.uniform(0.5, 2.0, p["noise_var"].shape))
    lk.precompute()


@pytest.mark.parametrize("precision", ["mixed", "fp64"])
def test_same_as_a_fresh_context(precision):
    import paper_2501_12928_gb300 as P

    p, q = (random_problem(n + 40, n, 3, seed=n) for n in (300, 140))
    ph = np.random.default_rng(0).uniform(-2, 2, (5, 3))
    a, b = _like(P, p, precision, 1), _like(P, q, precision, 2)
    for swap in range(3):
        got = [a.lnl(ph)[0], a.posterior_mean(ph[1])[0], P.lnl_multi([a, b], [ph, ph[:2]])[0]]
        fa, fb = _like(P, p, precision, 1 + 10 * swap), _like(P, q, precision, 2 if swap == 0 else 20)
        want = [fa.lnl(ph)[0], fa.posterior_mean(ph[1])[0], P.lnl_multi([fa, fb], [ph, ph[:2]])[0]]
        np.testing.assert_array_equal(got[0], want[0])
        np.testing.assert_array_equal(got[1], want[1])
        for x, y in zip(got[2], want[2]):
            np.testing.assert_array_equal(x, y)
        _data(a, p, 1 + 10 * (swap + 1))
        if swap == 0:
            _data(b, q, 20)
        with pytest.raises(P.BeorError):
            a.factor(0)
        with pytest.raises(P.BeorError):
            a.terms(5)


def test_device_buffers_and_another_model():
    """Asynchronous calls on new data (the first one of a slot is complete on return),
    and a model of another size on the same context."""
    torch = pytest.importorskip("torch")
    import paper_2501_12928_gb300 as P

    p, q = (random_problem(n + 40, n, 3, seed=n) for n in (300, 140))
    ph = np.random.default_rng(0).uniform(-2, 2, (4, 3))
    lk = _like(P, p, "mixed", 1)
    s = torch.cuda.Stream()
    phd = torch.from_numpy(ph).cuda()
    out, st = torch.zeros(4, dtype=torch.float64, device="cuda"), torch.zeros(4, dtype=torch.int32, device="cuda")
    torch.cuda.synchronize()
    for seed in (1, 2, 3):
        if seed > 1:
            _data(lk, p, seed)
            with pytest.raises(P.BeorError):
                P.lnl_multi_wait([lk], [4], 1, s.cuda_stream)
        want = _like(P, p, "mixed", seed).lnl(ph)[0]
        for _ in range(2):
            P.lnl_multi_async([lk], [phd], [out], [st], 1, s.cuda_stream)
            P.lnl_multi_wait([lk], [4], 1, s.cuda_stream)
            np.testing.assert_array_equal(out.cpu().numpy(), want)
    lk.set_T(q["T"], q["kbin"], 3, 2.0)
    _data(lk, q, 5)
    np.testing.assert_array_equal(lk.lnl(ph)[0], _like(P, q, "mixed", 5).lnl(ph)[0])
