"""The FP32 trailing update with the next diagonal block in its launch, at the edges of
its 128 x 128 tiles, for both panel widths and odd leading dimensions.  Tolerance:
FP32 Cholesky satisfies |A - L L^T|_ij <= gamma_(n+1) (|L| |L^T|)_ij <=
(n + 2) u sqrt(a_ii a_jj), u = 2^-24; a factor of 2 covers the second order."""
from __future__ import annotations

import ctypes

import numpy as np
import pytest
import torch

from helpers import DEV, host
from paper_2601_14466_gb300 import inputs, jmg

pytestmark = pytest.mark.gpu
U32 = 2.0 ** -24


def _factor(A: torch.Tensor, nb: int, lda: int):
    n = A.shape[0]
    buf = torch.full((n, lda), float("nan"), dtype=torch.float32, device=DEV)
    buf[:, :n] = A.t().to(DEV)
    view = buf.t()[:n]
    info = torch.full((1,), 77, dtype=torch.int32, device=DEV)
    o = jmg.default_options(nb=nb)
    st = jmg.load().jmg_potrf(n, view.data_ptr(), lda, jmg.JMG_F32, info.data_ptr(),
                              ctypes.byref(o), None, 0, torch.cuda.current_stream().cuda_stream)
    assert st == 0
    torch.cuda.synchronize()
    assert torch.isnan(buf[:, n:]).all()
    return host(view), int(info.item())


@pytest.mark.parametrize("n,nb,lda", [(128, 128, 128), (129, 128, 131), (193, 64, 193), (255, 64, 256),
                                      (256, 128, 256), (257, 128, 257), (385, 128, 390),
                                      (640, 64, 641)])
def test_fp32_factor_at_tile_edges(n, nb, lda):
    A = inputs.gram_shift(n, 1.0, seed=inputs.seed_for("syrk32", n)).float()
    Lower = torch.tril(A) + torch.triu(torch.full_like(A, float("nan")), 1)
    L, info = _factor(Lower, nb, lda)
    assert info == 0
    assert np.isnan(L[np.triu_indices(n, 1)]).all()
    L, A = np.tril(L).astype(np.float64), A.double().numpy()
    s = np.sqrt(np.diag(A))
    assert np.max(np.abs(A - L @ L.T) / np.outer(s, s)) <= 2 * (n + 2) * U32


@pytest.mark.parametrize("k", [0, 127, 128, 200, 383])
def test_fp32_factor_reports_the_first_bad_pivot(k):
    A = inputs.gram_shift(384, 1.0, seed=5).float()
    A[k, k] = -1.0
    assert _factor(A, 128, 384)[1] == k + 1
