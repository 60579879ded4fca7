"""The float64 precompute of factored instruments at sizes around its 16 x 16
tiles and eight-row steps, the dense dbar over several chunks of visibilities,
and the exported normal matrix (one band, several bands, device output) against
the oracle: 1e-13 of the largest element, as for the whole instruments."""

import ctypes

import numpy as np
import pytest

import oracle as O
from synth.instrument import random_problem

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def P():
    import paper_2501_12928_gb300 as P
    return P


def _close(a, b):
    assert np.abs(a - b).max() <= 1e-13 * np.abs(b).max()


@pytest.mark.parametrize("ncells", [1, 15, 16, 17, 33])
@pytest.mark.parametrize("ntb", [1, 7, 8, 9, 2100])
def test_factored(P, ncells, ntb):
    nf, nx = 3, 4
    g = np.random.default_rng(100 * ncells + ntb)

    def cn(*shape):
        return g.standard_normal(shape) + 1j * g.standard_normal(shape)
    A, W, d = cn(nf, ntb, ncells), cn(nf, nx), cn(nf * ntb)
    var = 0.5 + g.random(nf * ntb)
    kbin = np.zeros(ncells * nx, np.int32)
    lk = P.Likelihood("fp64")
    lk.set_instrument(A, W, kbin, 1, 2.0)
    lk.set_data(d, var)
    lk.precompute()
    _close(lk.get_M(), O.herm_structured(A, W, var))
    _close(lk.get_dbar(), O.dbar_structured(A, W, var, d))


@pytest.mark.parametrize("nvis,n", [(1, 3), (255, 31), (257, 33), (4097, 65), (9000, 20)])
def test_dense(P, nvis, n):
    p = random_problem(nvis, n, 2, seed=nvis)
    for precision in ("fp64", "mixed"):
        lk = P.Likelihood(precision)
        lk.set_T(p["T"], p["kbin"], 2, 2.0)
        lk.set_data(p["d"], p["noise_var"])
        lk.precompute()
        _close(lk.get_dbar(), O.dbar_dense(p["T"], p["noise_var"], p["d"]))
        M, ref = lk.get_M(), O.herm_dense(p["T"], p["noise_var"])
        assert np.abs(M - ref).max() <= (1e-13 if precision == "fp64" else 2.0 ** -38) * np.abs(ref).max()
        np.testing.assert_array_equal(M, M.conj().T)


@pytest.mark.parametrize("n", [31, 32, 33, 129, 4200])
def test_normal_matrix_in_bands_and_on_the_device(P, n):
    """4200 modes exceed one 256 MB band."""
    import torch
    p = random_problem(6, n, 2, seed=n)
    lk = P.Likelihood("fp64")
    lk.set_T(p["T"], p["kbin"], 2, 2.0)
    lk.set_data(p["d"], p["noise_var"])
    lk.precompute()
    M = lk.get_M()
    _close(M, O.herm_dense(p["T"], p["noise_var"]))
    out = torch.empty((n, n), dtype=torch.complex128, device="cuda")
    assert P.beor._lib().beor_get_M(lk._h, ctypes.c_void_p(out.data_ptr())) == 0
    np.testing.assert_array_equal(out.cpu().numpy(), M)


@pytest.mark.parametrize("ncells,nx", [(2, 3), (3, 2), (9, 40), (40, 9), (41, 41)])
def test_factored_weights(P, ncells, nx):
    """The products of weights from a table (nx <= ncells) and formed per element,
    over one tile and over several with a ragged last one."""
    nf, ntb = 5, 11
    g = np.random.default_rng(100 * ncells + nx)

    def cn(*shape):
        return g.standard_normal(shape) + 1j * g.standard_normal(shape)
    A, W, d = cn(nf, ntb, ncells), cn(nf, nx), cn(nf * ntb)
    var = 0.5 + g.random(nf * ntb)
    lk = P.Likelihood("fp64")
    lk.set_instrument(A, W, np.zeros(ncells * nx, np.int32), 1, 2.0)
    lk.set_data(d, var)
    lk.precompute()
    _close(lk.get_M(), O.herm_structured(A, W, var))


def test_dense_dbar_of_many_chunks(P):
    """Enough chunks of visibilities for the wide kernel.  Bound: chains of 1024
    rows, the product with the weight and 320 chunk sums, each step within 2^-53 of
    the sum of magnitudes."""
    nvis, n = 327680, 3
    p = random_problem(nvis, n, 2, seed=5)
    lk = P.Likelihood("fp64")
    lk.set_T(p["T"], p["kbin"], 2, 2.0)
    lk.set_data(p["d"], p["noise_var"])
    lk.precompute()
    wd = p["d"] / p["noise_var"]
    ref = np.array([np.sum((np.conj(p["T"][:, j]) * wd).astype(np.clongdouble)) for j in range(n)])
    mag = np.abs(p["T"]).T @ np.abs(wd)
    assert np.all(np.abs(lk.get_dbar() - ref) <= 2 * (1024 + 320 + 8) * 2.0 ** -53 * mag)
