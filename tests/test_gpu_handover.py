"""Blocks that several leaders hand to the helpers of a one-launch solve: a helper reads
the columns of every leader after one wait on all of their counters, each lane of a warp
on another one.  A helper that read a block too early would use the right-hand side in its
place, so the result must be the same from run to run and solve the system."""
from __future__ import annotations

import pytest
import torch

from helpers import DEV, U64
from paper_2601_14466_gb300 import inputs, jmg

pytestmark = pytest.mark.gpu
RUNS = 12


def _repeat(solve, n, nrhs, dtype, tol):
    L = inputs.lower_factor(n, seed=11)
    B = inputs.uniform(n, nrhs, seed=12).to(dtype)
    Ld = jmg.colmajor_copy(L.to(dtype).to(DEV))
    first = None
    for _ in range(RUNS):
        Bd = jmg.colmajor_copy(B.to(DEV))
        solve(Ld, Bd)
        first = Bd.clone() if first is None else first
        assert torch.equal(first, Bd)
    Y = torch.linalg.solve_triangular(Ld.double(), B.double().to(DEV), upper=False)
    X = torch.linalg.solve_triangular(Ld.double().mT, Y, upper=True)
    assert float((first - X).abs().max()) <= tol * max(1.0, float(X.abs().max()))


@pytest.mark.parametrize("n,nrhs", [(1500, 9), (3000, 16), (3000, 64)])
def test_block_inverse_solves_repeat(n, nrhs):
    # 5, 8 and 16 leaders; the bound of the other tests of these solves
    _repeat(jmg.sv_potrs_, n, nrhs, torch.float32, 2048 * 2.0 ** -24)


@pytest.mark.parametrize("n,nrhs", [(1500, 3), (3000, 16), (1000, 40)])
def test_fp64_solves_repeat(n, nrhs):
    # 3 and 16 leaders of one right-hand side, groups of 4 leaders of four
    _repeat(jmg.potrs_, n, nrhs, torch.float64, 64 * n * U64)
