"""beor_get_M to device memory, aligned to 16 bytes and to 8: the host's matrix."""

import ctypes

import numpy as np
import pytest

from synth.instrument import random_problem

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("n", [1, 31, 300])
@pytest.mark.parametrize("offset", [0, 1])
def test_device_output(n, offset):
    torch = pytest.importorskip("torch")
    import paper_2501_12928_gb300 as P
    from paper_2501_12928_gb300 import beor

    p = random_problem(n + 40, n, 1, seed=n)
    lk = P.Likelihood("mixed")
    lk.set_T(p["T"], p["kbin"], 1, 2.0)
    lk.set_data(p["d"], p["noise_var"])
    lk.precompute()
    out = torch.full((2 * n * n + 2,), 7.0, dtype=torch.float64, device="cuda")
    torch.cuda.synchronize()
    assert beor._lib().beor_get_M(lk._h, ctypes.c_void_p(out.data_ptr() + 8 * offset)) == 0
    got = out.cpu().numpy()
    np.testing.assert_array_equal(got[offset:offset + 2 * n * n].view(np.complex128).reshape(n, n), lk.get_M())
    assert np.all(got[:offset] == 7.0) and np.all(got[offset + 2 * n * n:] == 7.0)
