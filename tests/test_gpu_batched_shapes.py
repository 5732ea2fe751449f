"""Batched small systems at the edges of the kernel's shapes: one row and one more
than a lane group, the thread-count and register steps (24, 32, 48, 64, 96, 128),
right-hand sides around the lanes-per-system steps, FP32 on both sides of order 48,
padded leading dimensions, a failing system among good ones.  Tolerances as in the
batched parity tests (64 n u max |x| in FP64, backward error 8 n u in FP32)."""
from __future__ import annotations

import numpy as np
import pytest
import torch

import oracle
from helpers import DEV, U64
from paper_2601_14466_gb300 import inputs, jmg

pytestmark = pytest.mark.gpu
U32 = 2.0 ** -24


@pytest.mark.parametrize("n,nrhs", [(2, 1), (24, 3), (25, 9), (32, 33), (33, 5), (48, 17), (49, 4),
                                    (64, 65), (65, 2), (96, 35), (97, 1), (127, 40), (128, 9)])
@pytest.mark.parametrize("dtype", [torch.float64, torch.float32])
def test_batched_shapes(n, nrhs, dtype):
    batch, bad = 5, 3
    A = torch.stack([inputs.gram_shift(n, 1.0, seed=40 + b) for b in range(batch)])
    B = torch.stack([inputs.uniform(n, nrhs, seed=50 + b) for b in range(batch)])
    A[bad, n // 2, n // 2] = -1.0
    A, B = A.to(dtype), B.to(dtype)
    lda, ldb = n + 3, n + 1
    Ad = torch.full((batch, n, lda), float("nan"), dtype=dtype, device=DEV)
    Ad[:, :, :n] = A.transpose(1, 2).to(DEV)
    Ad[:, :, :n] += torch.tril(torch.full((n, n), float("nan"), dtype=dtype, device=DEV), -1)
    Bd = torch.full((batch, nrhs, ldb), float("nan"), dtype=dtype, device=DEV)
    Bd[:, :, :n] = B.transpose(1, 2).to(DEV)
    info = torch.full((batch,), 77, dtype=torch.int32, device=DEV)
    st = jmg.load().jmg_posv_batched(n, nrhs, batch, Ad.data_ptr(), lda, lda * n, Bd.data_ptr(), ldb,
                                     ldb * nrhs, jmg.JMG_F64 if dtype == torch.float64 else jmg.JMG_F32,
                                     info.data_ptr(), torch.cuda.current_stream().cuda_stream)
    assert st == 0
    torch.cuda.synchronize()
    assert info.cpu().tolist() == [0 if b != bad else n // 2 + 1 for b in range(batch)]
    assert torch.isnan(Ad[:, :, n:]).all() and torch.isnan(Bd[:, :, n:]).all()
    for b in range(batch):
        X = Bd[b, :, :n].t().double().cpu().numpy()
        if b == bad:
            assert np.array_equal(X, B[b].double().numpy())
            continue
        A64, B64 = A[b].double().numpy(), B[b].double().numpy()
        if dtype == torch.float64:
            Xo, _ = oracle.posv(A64, B64)
            assert np.abs(X - Xo).max() <= 64 * max(n, 8) * U64 * max(1.0, np.abs(Xo).max())
            Lo, _ = oracle.potrf(A64)
            L = np.triu(Ad[b, :, :n].cpu().numpy()).T
            assert np.abs(L - np.tril(Lo)).max() <= 64 * n * U64 * np.abs(Lo).max()
        else:
            assert oracle.bwd_err(A64, np.asfortranarray(X), B64)[0] <= 8 * n * U32
