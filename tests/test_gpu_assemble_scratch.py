"""The structured normal matrix does not depend on what its scratch held: every
element of its tiles is written, those above the diagonal as zeros."""

import ctypes

import numpy as np
import pytest

pytestmark = pytest.mark.gpu

NAME = "_ZN4beor19precompute_factoredEPK7double2S2_iliiPKdS2_iiPS0_S5_S5_S5_S5_P11CUstream_st"


@pytest.mark.parametrize("table", [True, False])
@pytest.mark.parametrize("nf, ntb, ncells, nx", [(2, 9, 1, 5), (3, 20, 5, 7), (2, 40, 24, 11), (4, 17, 3, 90)])
def test_scratch_of_nan(nf, ntb, ncells, nx, table):
    torch = pytest.importorskip("torch")
    from paper_2501_12928_gb300 import beor

    f = getattr(beor._lib(), NAME)
    i, p = ctypes.c_int, ctypes.c_void_p
    f.argtypes = [p, p, i, ctypes.c_int64, i, i, p, p, i, i, p, p, p, p, p, p]
    f.restype = i
    rng = np.random.default_rng(nf + ncells)
    z = lambda *s: rng.standard_normal(s) + 1j * rng.standard_normal(s)
    A, W, w, d = z(nf, ntb, ncells), z(nf, nx), rng.uniform(0.5, 2.0, (nf, ntb)), z(nf, ntb)
    n = ncells * nx
    nt = (n + 127) // 128
    dev = lambda a: torch.from_numpy(np.ascontiguousarray(a)).cuda()
    nan = lambda k: torch.full((2 * k,), float("nan"), dtype=torch.float64, device="cuda")
    a = [dev(A), dev(W), dev(w), dev(d)]
    G, u, P = nan(nf * ncells * ncells), nan(nf * ncells), nan(nf * nx * nx)
    M, dbar = nan(nt * (nt + 1) // 2 * 128 * 128), nan(nt * 128)
    torch.cuda.synchronize()
    assert f(a[0].data_ptr(), a[1].data_ptr(), nf, ntb, ncells, nx, a[2].data_ptr(), a[3].data_ptr(), n, nt,
             G.data_ptr(), u.data_ptr(), P.data_ptr() if table else None, M.data_ptr(), dbar.data_ptr(), None) == 0
    torch.cuda.synchronize()
    T = (A[:, :, :, None] * W[:, None, None, :]).reshape(nf * ntb, n)
    want = np.zeros((nt * 128, nt * 128), np.complex128)
    want[:n, :n] = np.tril(T.conj().T @ (w.reshape(-1, 1) * T))
    got = M.cpu().numpy().view(np.complex128).reshape(-1, 128, 128)
    scale = 8e-16 * nf * ntb * np.abs(A).max() ** 2 * np.abs(W).max() ** 2 * 2.0   # rounding of the longest sums
    for I in range(nt):
        for J in range(I + 1):
            tile = got[I * (I + 1) // 2 + J].T   # stored by columns
            ref = want[128 * I:128 * I + 128, 128 * J:128 * J + 128]
            assert np.all(np.abs(tile - ref) <= scale), (I, J)
            if I == J:
                assert np.all(tile[np.triu_indices(128, 1)] == 0)
