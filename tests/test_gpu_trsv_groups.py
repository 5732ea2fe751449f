"""The one-launch triangular solves at the edges of their shapes: one block and
one row more, as many blocks as a leader multiplies itself and one more, one
leader per right-hand side (up to 16), leaders of four, a ragged last group, odd
leading dimensions.  Against the oracle's substitution; tolerance: substitution
in either order of summation satisfies |L dx| <= n u |L| |x| per direction, and
inputs.lower_factor keeps || L^-1 || |L| of order one (factor 64 as in the other
parity tests)."""
from __future__ import annotations

import numpy as np
import pytest
import torch

import oracle
from helpers import U64, host, to_dev_colmajor
from paper_2601_14466_gb300 import inputs, jmg

pytestmark = pytest.mark.gpu
U32 = 2.0 ** -24


@pytest.mark.parametrize("n,nrhs", [(1, 1), (31, 2), (32, 16), (33, 17), (96, 4), (97, 20),
                                    (160, 1), (161, 16), (255, 3), (257, 33), (289, 5)])
@pytest.mark.parametrize("dtype", [torch.float64, torch.float32])
def test_potrs_at_block_and_group_edges(n, nrhs, dtype):
    L = inputs.lower_factor(n, seed=3).to(dtype)
    B = inputs.uniform(n, nrhs, seed=4).to(dtype)
    Xo = oracle.potrs(np.asfortranarray(L.double().numpy()), B.double().numpy())
    lda = n + (n % 3)
    Lb = torch.full((n, lda), float("nan"), dtype=dtype, device="cuda")
    Lb[:, :n] = torch.tril(L).t().to("cuda")
    Ld = Lb.t()[:n]
    Bd = B.to("cuda").t().contiguous().t()
    jmg.potrs_(Ld, Bd)
    first = Bd.clone()
    u = U64 if dtype == torch.float64 else U32
    assert np.abs(host(Bd).astype(np.float64) - Xo).max() <= 64 * n * u * max(1.0, np.abs(Xo).max())
    Bd.copy_(B)
    jmg.potrs_(Ld, Bd)  # fixed order of summation: the same bits again
    assert torch.equal(first, Bd)
