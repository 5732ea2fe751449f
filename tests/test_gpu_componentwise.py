"""Componentwise accuracy of the FP64 routes whose products run in slices.  A row is cut
against its largest entry, so products of rows whose large entries never meet would be
lost; such rows take FP64 FMAs instead.  The bounds are those of the FP64 FMAs, entry by
entry (with rows that stay on the slices, sum |p_k q_k| > 2^-13 K max|p| max|q| against an
error of about 2^-56 sqrt(K) max|p| max|q|: below n u of it for every n here)."""
from __future__ import annotations

import numpy as np
import pytest
import torch

from helpers import DEV, U64, host, to_dev_colmajor
from paper_2601_14466_gb300 import jmg

pytestmark = pytest.mark.gpu


def _wide(shape, seed, decades=20):
    """Signed entries with magnitudes spread evenly over `decades`."""
    g = torch.Generator().manual_seed(seed)
    mag = 10.0 ** (-decades * torch.rand(shape, generator=g, dtype=torch.float64))
    return mag * (torch.randint(0, 2, shape, generator=g) * 2 - 1)


def _matrix(kind, n):
    if kind == "kernel":  # exponential covariance of a 2-D grid, from 1 down to 1e-36
        i = torch.arange(n, dtype=torch.float64)
        x, y = i % 27, torch.div(i, 27, rounding_mode="floor")
        return torch.exp(-2.0 * torch.hypot(x[:, None] - x, y[:, None] - y))
    L = torch.tril(_wide((n, n), n), -1) + 4.0 * torch.eye(n, dtype=torch.float64)
    A = (L.numpy().astype(np.longdouble) @ L.numpy().T.astype(np.longdouble)).astype(np.float64)
    return torch.from_numpy(A)


@pytest.mark.parametrize("kind,n", [("kernel", 700), ("wide", 65), ("wide", 600)])
def test_factor_keeps_small_entries(kind, n):
    A = _matrix(kind, n)
    Ad, _ = to_dev_colmajor(A)
    assert int(jmg.potrf_(Ad).item()) == 0
    L = np.tril(host(Ad)).astype(np.longdouble)
    R = np.abs(A.numpy() - L @ L.T)
    bound = (2 * n + 2) * U64 * (np.abs(L) @ np.abs(L).T)
    assert np.all(np.tril(R <= bound) | (np.triu(np.ones((n, n)), 1) > 0))


def _potrs_fast(L, B):
    n, nrhs = B.shape
    Ld, Bd = jmg.colmajor_copy(L.to(DEV)), jmg.colmajor_copy(B.to(DEV))
    nbytes = int(jmg.load().jmg_workspace_fast(jmg.OP_POTRS, n, nrhs, jmg.JMG_F64, None))
    assert nbytes > jmg.workspace_size(jmg.OP_POTRS, n, nrhs)  # the blocked route
    work = torch.empty(nbytes, dtype=torch.uint8, device=DEV)
    st = jmg.load().jmg_potrs(n, nrhs, Ld.data_ptr(), n, Bd.data_ptr(), n, jmg.JMG_F64,
                              work.data_ptr(), nbytes, torch.cuda.current_stream().cuda_stream)
    assert st == 0
    torch.cuda.synchronize()
    return host(Bd)


def test_solve_keeps_the_tails_of_a_local_operator():
    # L = I with -0.9 below the diagonal, unit right-hand sides: every term of either
    # substitution is positive, so each entry carries the relative error of the 4 n
    # operations on its path, down to 0.9^4100 = 2e-188
    n, nrhs, a = 4100, 63, 0.9
    L = torch.eye(n, dtype=torch.float64)
    L.diagonal(-1).fill_(-a)
    at = [(j * 67) % n for j in range(nrhs)]
    B = torch.zeros(n, nrhs, dtype=torch.float64)
    B[at, range(nrhs)] = 1.0
    X = _potrs_fast(L, B)
    i = np.arange(n, dtype=np.longdouble)
    q = np.longdouble(a)
    for c, j in enumerate(at):  # (L L^T)^-1 e_j: sum over k >= max(i, j) of a^(2 k - i - j)
        m = np.maximum(i, j)
        want = q ** (2 * m - i - j) * (1 - q ** (2 * (n - m))) / (1 - q * q)
        np.testing.assert_allclose(X[:, c], want.astype(np.float64), rtol=8 * n * U64, atol=0)


def test_solve_keeps_small_entries():
    # an M-matrix factor and right-hand sides with entries over 20 decades: positive
    # terms only, so entry by entry against the same substitution in long double
    # (three of the right-hand sides)
    n, nrhs = 4096, 62
    L = -torch.tril(_wide((n, n), 5).abs(), -1) / n + torch.eye(n, dtype=torch.float64)
    B = _wide((n, nrhs), 6).abs()
    X = _potrs_fast(L, B)[:, ::30]
    Ll, Y = L.numpy().astype(np.longdouble), B.numpy()[:, ::30].astype(np.longdouble)
    for k in range(n):
        Y[k + 1:] -= Ll[k + 1:, k:k + 1] * Y[k]
    for k in range(n - 1, -1, -1):
        Y[:k] -= Ll[k:k + 1, :k].T * Y[k]
    np.testing.assert_allclose(X, Y.astype(np.float64), rtol=64 * n * U64, atol=0)


@pytest.mark.parametrize("n,nrhs", [(65, 12), (300, 16), (513, 21)])
def test_adjoint_keeps_small_entries(n, nrhs):
    Y, X = _wide((n, nrhs), 7), _wide((n, nrhs), 8)
    Y[::3], X[::3] = torch.sign(Y[::3]), torch.sign(X[::3])  # flat rows in between
    G = jmg.sym_grad(jmg.colmajor_copy(Y.to(DEV)), jmg.colmajor_copy(X.to(DEV))).cpu().numpy()
    Yl, Xl = Y.numpy().astype(np.longdouble), X.numpy().astype(np.longdouble)
    want = -(Yl @ Xl.T + Xl @ Yl.T) / 2
    bound = (2 * nrhs + 2) * U64 * (np.abs(Yl) @ np.abs(Xl).T + np.abs(Xl) @ np.abs(Yl).T)
    assert np.all(np.abs(G - want) <= bound)


@pytest.mark.parametrize("where", ["L", "B"])
@pytest.mark.parametrize("value", [float("inf"), float("nan")])
def test_solve_with_entries_that_are_not_finite(where, value):
    # as substitution has it: what does not depend on the entry stays finite (the other
    # right-hand sides, or nothing at all once L has it), the rest is not finite
    n, nrhs = 4096, 64
    g = torch.Generator().manual_seed(9)
    L = torch.tril(torch.randn(n, n, generator=g, dtype=torch.float64) / n ** 0.5, -1) \
        + 2.0 * torch.eye(n, dtype=torch.float64)
    B = torch.randn(n, nrhs, generator=g, dtype=torch.float64)
    clean = _potrs_fast(L, B)
    if where == "B":
        B[1000, 5] = value
    else:
        L[1000, 700] = value
    X = _potrs_fast(L, B)
    if where == "B":
        keep = np.arange(nrhs) != 5
        np.testing.assert_array_equal(X[:, keep], clean[:, keep])
        assert not np.isfinite(X[:, 5]).any()
    else:
        assert not np.isfinite(X).all(axis=0).any()
