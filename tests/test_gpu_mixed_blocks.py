"""The mixed factorisation where a panel's update factors the next diagonal block itself:
sizes at the edges of the 128-row tiles, both panel widths, and the position of a pivot
that fails in any block.

A = I + u u^T / n, |u_i| <= 1, has x = b - u (u.b / n) / (1 + u.u / n) in closed form,
|A|_inf <= 2 and |A^-1|_inf <= 2; refined to a backward error of 1e-13 a solve is off by at
most |A^-1| 1e-13 (|A| |x| + |b|) <= 8e-13 |x| (inf-norms).
"""
import numpy as np
import pytest
import torch

from paper_2601_14466_gb300 import jmg

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("prec,nb", [("bf16", 64), ("bf16", 128), ("fp16", 128), ("fp8", 128)])
@pytest.mark.parametrize("n", [1, 64, 65, 127, 128, 129, 192, 256, 257, 1024, 1025, 1153])
def test_diagonal_blocks_edges(n, prec, nb):
    rng = np.random.default_rng(n)
    u, b = rng.uniform(-1, 1, n), rng.standard_normal(n)
    A = np.eye(n) + np.outer(u, u) / n
    x = b - u * ((u @ b) / n) / (1 + (u @ u) / n)
    Ad = torch.from_numpy(A).cuda().mT  # (symmetric)
    X, si = jmg.posv(Ad, torch.from_numpy(b[:, None]).cuda(), prec=prec, nb=nb)
    assert np.abs(X.cpu().numpy()[:, 0] - x).max() <= 1e-12 * np.abs(x).max()


@pytest.mark.parametrize("k", [0, 127, 128, 255, 256, 400, 1023, 1024, 1151])
def test_failing_pivot_position(k):
    n = 1152
    A = torch.eye(n, dtype=torch.float64, device="cuda")
    A[k, k] = -1.0
    _, si = jmg.posv(A.mT, torch.ones(n, 1, dtype=torch.float64, device="cuda"), prec="bf16",
                     shift_retry=False, check=False)
    assert si.info == k + 1
