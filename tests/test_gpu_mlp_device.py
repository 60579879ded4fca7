"""Predictions on device arrays that overlap: the same as those of host arrays."""

import numpy as np
import pytest

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("n, n_in, end", [(64, 2, 0), (64, 2, 1), (5003, 9, 0), (5003, 9, 1), (65536, 3, 0),
                                          (65536, 3, 1), (70001, 2, 0)])
def test_output_over_the_inputs(n, n_in, end):
    """The predictions go over the head of x, or (end) over its end and one float
    further.  65,536 points at a time, each read before it is overwritten."""
    torch = pytest.importorskip("torch")
    import paper_2501_12928_gb300 as P

    em = P.Emulator(n_in, 64, 2)
    x = np.random.default_rng(n).uniform(-2, 2, (n, n_in)).astype(np.float32)
    want = em.infer(x)
    buf = torch.empty(n * n_in + 1, dtype=torch.float32, device="cuda")
    start = n * n_in + 1 - n if end else 0
    for _ in range(5):
        buf[:-1] = torch.from_numpy(x.reshape(-1)).cuda()
        em.infer(buf[:-1].view(n, n_in), out=buf[start:start + n])
        np.testing.assert_array_equal(buf[start:start + n].cpu().numpy(), want)
