"""The adjoint -(Bbar X^T + X Bbar^T) / 2 around the switch to the tensor cores and at the
edges of its tiles, against NumPy in FP64.

Per chunk of 16 right-hand sides an entry's slices leave out at most
(2^-50 + 6 16 4 2^-56) M < 2^-46.9 M of each of the two products, M the largest
max_i |b_ik| max_j |x_jk| of the chunk's columns (row scales are at most twice the row's
maximum, the column balance at most doubles one side); FP64 sums on either side add
2 nrhs 2^-53 sum_k.  With sum_k in place of M, 2^-45 per chunk covers all of it.
"""
import numpy as np
import pytest
import torch

from paper_2601_14466_gb300 import jmg

pytestmark = pytest.mark.gpu


def _run(Bb, X):
    dev = "cuda"
    b = jmg.colmajor_copy(torch.from_numpy(Bb).to(dev))
    x = jmg.colmajor_copy(torch.from_numpy(X).to(dev))
    return jmg.sym_grad(b, x).cpu().numpy()


@pytest.mark.parametrize("n", [1, 63, 128, 577, 1024, 1025, 1153])
@pytest.mark.parametrize("nrhs", [1, 5, 6, 11, 12, 16, 17, 33])
@pytest.mark.parametrize("spread", [0, 40])
def test_sym_grad_sizes(n, nrhs, spread):
    rng = np.random.default_rng(n * 100 + nrhs + spread)
    Bb = rng.standard_normal((n, nrhs)) * 2.0 ** rng.integers(-spread, spread + 1, nrhs)
    X = rng.standard_normal((n, nrhs)) * 2.0 ** rng.integers(-spread, spread + 1, nrhs)
    G = _run(Bb, X)
    P = Bb @ X.T
    ref = -0.5 * (P + P.T)
    chunks = (nrhs + 15) // 16
    tol = 2.0**-45 * chunks * np.sum(np.abs(Bb).max(0) * np.abs(X).max(0))
    assert np.array_equal(G, G.T)
    assert np.abs(G - ref).max() <= tol


@pytest.mark.parametrize("bad", [np.nan, np.inf])
def test_sym_grad_not_finite(bad):
    rng = np.random.default_rng(7)
    Bb, X = rng.standard_normal((600, 16)), rng.standard_normal((600, 16))
    Bb[130, 3] = bad
    X[5, 1] = 0.0
    G = _run(Bb, X)
    with np.errstate(invalid="ignore"):
        ref = -0.5 * (np.einsum("ik,jk->ij", Bb, X) + np.einsum("ik,jk->ij", X, Bb))
    assert np.array_equal(np.isnan(G), np.isnan(ref))
    assert np.array_equal(np.isinf(G), np.isinf(ref))
    ok = np.isfinite(ref)
    assert np.abs(G[ok] - ref[ok]).max() <= 2.0**-45 * 16 * 36
