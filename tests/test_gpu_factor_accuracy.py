"""The FP64 factorisation's error against the exact factor: no larger than that of the
blocked algorithm with blocks of 32 columns (with a quarter for the scatter)."""
from __future__ import annotations

import numpy as np
import pytest
import torch

from helpers import DEV
from paper_2601_14466_gb300 import jmg

pytestmark = pytest.mark.gpu


def _blocked(A, dt, block=32):
    A = A.astype(dt)
    n = A.shape[1]
    L = np.zeros_like(A)
    for p in range(0, n, block):
        e = min(n, p + block)
        for j in range(p, e):
            L[:, j, j] = np.sqrt(A[:, j, j])
            L[:, j + 1:, j] = A[:, j + 1:, j] / L[:, j, j, None]
            A[:, j + 1:, j + 1:e] -= L[:, j + 1:, j, None] * L[:, None, j + 1:e, j]
        A[:, e:, e:] -= L[:, e:, p:e] @ L[:, e:, p:e].transpose(0, 2, 1)
    return L


@pytest.mark.parametrize("n,count", [(65, 60), (96, 30), (200, 6)])
def test_error_against_the_blocked_algorithm(n, count):
    rng = np.random.default_rng(n)
    q, _ = np.linalg.qr(rng.standard_normal((count, n, n)))
    lam = np.exp(np.linspace(0.0, np.log(10.0), n))
    A = (q * lam) @ q.transpose(0, 2, 1)
    A = (A + A.transpose(0, 2, 1)) / 2
    L = []
    for b in range(count):
        Ld = jmg.colmajor_copy(torch.from_numpy(A[b]).to(DEV))
        assert int(jmg.potrf_(Ld).item()) == 0
        L.append(np.tril(Ld.cpu().numpy()))
    exact = _blocked(A, np.longdouble)

    def err(a):
        return float(np.sqrt((((a - exact) / np.abs(exact).max()) ** 2).mean()))

    assert err(np.stack(L)) <= 1.25 * err(_blocked(A, np.float64))
