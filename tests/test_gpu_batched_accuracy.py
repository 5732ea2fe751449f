"""Accuracy of the batched small systems: no further from the exact factor and solution
than the textbook algorithm in blocks of 32 columns in the same precision (with a quarter
for the scatter of 30 systems), and the whole range of pivots."""
from __future__ import annotations

import numpy as np
import pytest
import torch

from helpers import DEV
from paper_2601_14466_gb300 import jmg

pytestmark = pytest.mark.gpu


def _textbook(A, B, dt, block=32):
    """Blocked right-looking Cholesky and substitution over a batch, every operation in dt."""
    A, X = A.astype(dt), B.astype(dt)
    n = A.shape[1]
    L = np.zeros_like(A)
    for p in range(0, n, block):
        e = min(n, p + block)
        for j in range(p, e):
            L[:, j, j] = np.sqrt(A[:, j, j])
            L[:, j + 1:, j] = A[:, j + 1:, j] / L[:, j, j, None]
            A[:, j + 1:, j + 1:e] -= L[:, j + 1:, j, None] * L[:, None, j + 1:e, j]
        A[:, e:, e:] -= L[:, e:, p:e] @ L[:, e:, p:e].transpose(0, 2, 1)
    for j in range(n):
        X[:, j] /= L[:, j, j, None]
        X[:, j + 1:] -= L[:, j + 1:, j, None] * X[:, j, None]
    for j in range(n - 1, -1, -1):
        X[:, j] /= L[:, j, j, None]
        X[:, :j] -= L[:, j, :j, None] * X[:, j, None]
    return L, X


@pytest.mark.parametrize("n", [8, 48, 70, 128])
def test_error_against_the_textbook_algorithm(n):
    rng = np.random.default_rng(n)
    M = rng.standard_normal((30, n, 2 * n))
    A = M @ M.transpose(0, 2, 1) / (2 * n) + 0.1 * np.eye(n)
    A = (A + A.transpose(0, 2, 1)) / 2
    B = rng.standard_normal((30, n, 3))
    X, L, info = jmg.posv_batched(torch.from_numpy(A).to(DEV), torch.from_numpy(B).to(DEV))
    assert not info.any()
    Le, Xe = _textbook(A, B, np.longdouble)
    Lt, Xt = _textbook(A, B, np.float64)
    got = np.tril(L.cpu().numpy().transpose(0, 2, 1)), X.cpu().numpy()

    def err(a, e):
        return float(np.sqrt((((a - e) / np.abs(e).max()) ** 2).mean()))

    assert err(got[0], Le) <= 1.25 * err(Lt, Le)
    assert err(got[1], Xe) <= 1.25 * err(Xt, Xe)


@pytest.mark.parametrize("dtype,n", [(torch.float64, 1), (torch.float64, 70), (torch.float32, 1),
                                     (torch.float32, 48), (torch.float32, 49)])
def test_pivots_over_the_whole_range(dtype, n):
    # A = d I, B = d: X = 1 and L = sqrt(d) for every d of the type, subnormal ones included
    # (FP64 above order 1: normal ones, since 0 / d is taken as 0 (1 / d))
    fi = torch.finfo(dtype)
    below = 18 if dtype == torch.float32 else (40 if n == 1 else 0)
    lo, hi = np.log2(float(fi.tiny)) - below, np.log2(float(fi.max))
    e = np.random.default_rng(4).uniform(lo, hi, 500)
    d = torch.from_numpy(np.concatenate([2.0 ** e, [float(fi.tiny), float(fi.max), 1.0, 0.25, 4.0]])).to(dtype)
    u = float(fi.eps) / 2
    A = (d[:, None, None] * torch.eye(n, dtype=dtype)).to(DEV)
    X, L, info = jmg.posv_batched(A, d[:, None, None].expand(-1, n, 1).contiguous().to(DEV))
    assert not info.any()
    # 1 / d to 0.51 ulp (FP32: from sqrt(d) rounded, twice, and two divisions) and a product
    assert float((X.cpu().double() - 1).abs().max()) <= 5 * u
    r = torch.sqrt(d.double())
    got = L.cpu().double().diagonal(dim1=1, dim2=2)
    assert float(((got - r[:, None]) / r[:, None]).abs().max()) <= 2 * u
