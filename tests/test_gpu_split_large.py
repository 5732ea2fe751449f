"""The FP64 routes with products in slices at sizes where a CTA takes several tiles of an
update, the raster of the tiles has whole triangular groups, and the panel solve spreads a
row over 8, 4 and 2 lanes instead of 16."""
from __future__ import annotations

import pytest
import torch

from helpers import DEV, U64
from paper_2601_14466_gb300 import jmg

pytestmark = pytest.mark.gpu


def _gram(n, g):
    M = torch.randn(n, n, generator=g, dtype=torch.float64, device=DEV)
    A = M @ M.t() / n
    A = (A + A.t()) / 2
    A.diagonal().add_(0.5)
    return A


@pytest.mark.parametrize("n,lda", [(1700, 1700), (2600, 2603), (5200, 5200), (10500, 10500)])
def test_factor_reproduces_its_input(n, lda):
    g = torch.Generator(device=DEV).manual_seed(n)
    A = _gram(n, g)
    buf = torch.full((n, lda), float("nan"), dtype=torch.float64, device=DEV)
    buf[:, :n] = A + torch.full_like(A, float("nan")).tril_(-1)  # (rows of buf are columns)
    W = buf.t()[:n]
    assert int(jmg.potrf_(W).item()) == 0
    assert torch.isnan(buf[:, n:]).all() and torch.isnan(buf[:, :n].tril(-1)).sum() == n * (n - 1) // 2
    L = torch.tril(W)
    # A V against L (L^T V) for V of signs: (2 n + 2) u s_i s_j per entry of A - L L^T, n u of
    # |L| |L^T| per product here, and |L| |L^T| <= s_i s_j.  (A tile left out or taken twice
    # moves rows by 1e-2 and more.)
    V = torch.randint(0, 2, (n, 16), generator=g, device=DEV).double() * 2 - 1
    R = (A @ V - L @ (L.t() @ V)).abs()
    s = A.diagonal().sqrt()
    assert bool((R <= (5 * n + 2) * U64 * s[:, None] * s.sum()).all())


@pytest.mark.parametrize("n,nrhs", [(12001, 100), (20000, 17)])
def test_solve_satisfies_its_system(n, nrhs):
    g = torch.Generator(device=DEV).manual_seed(n)
    L = torch.randn(n, n, generator=g, dtype=torch.float64, device=DEV).mul_(n ** -0.5).tril_(-1)
    L.diagonal().copy_(2.0 + torch.rand(n, generator=g, dtype=torch.float64, device=DEV))
    B = torch.randn(n, nrhs, generator=g, dtype=torch.float64, device=DEV)
    X = jmg.potrs_(jmg.colmajor_copy(L), jmg.colmajor_copy(B))
    R = (L @ (L.t() @ X) - B).abs()
    La = L.abs_()
    # n u of |L| |L^T| |X| for either substitution, twice that for the products here
    bound = La @ (La.t() @ X.abs()) + B.abs()
    assert bool((R <= 4 * (n + 2) * U64 * bound).all())


def test_solve_behind_a_failed_factor_leaves_the_right_hand_sides():
    n, nrhs = 4100, 70
    g = torch.Generator(device=DEV).manual_seed(1)
    A = _gram(n, g)
    A[3000, 3000] = -1.0
    B = torch.randn(n, nrhs, generator=g, dtype=torch.float64, device=DEV)
    Ad, X = jmg.colmajor_copy(A), jmg.colmajor_copy(B)
    work = jmg.workspace(jmg.OP_POSV, n, nrhs, None, DEV)
    info = torch.zeros(1, dtype=torch.int32, device=DEV)
    st = jmg.load().jmg_posv(n, nrhs, Ad.data_ptr(), n, X.data_ptr(), n, jmg.JMG_F64, info.data_ptr(),
                             None, None, work.data_ptr(), work.numel(),
                             torch.cuda.current_stream().cuda_stream)
    assert st == 0
    assert int(info.item()) == 3001
    assert torch.equal(X, B)


def _spiky(n, g):
    """A lower factor with dense rows, every fifth one spiky (one large entry in sixteen)."""
    L = torch.randn(n, n, generator=g, dtype=torch.float64, device=DEV).mul_(n ** -0.5).tril_(-1)
    small = torch.rand(n, n, generator=g, dtype=torch.float64, device=DEV) > 1 / 16
    small[torch.arange(n, device=DEV) % 5 != 3] = False
    L[small] *= 1e-9
    L.diagonal().copy_(2.0 + torch.rand(n, generator=g, dtype=torch.float64, device=DEV))
    return L


@pytest.mark.parametrize("n", [777, 2600])
def test_factor_with_some_spread_rows(n):
    # the entries of a tile are shared out: those of spread rows and columns to the FMAs
    # (other CTAs), the rest to the slices
    g = torch.Generator(device=DEV).manual_seed(n)
    L0 = _spiky(n, g)
    A = L0 @ L0.t()
    W = jmg.colmajor_copy(A)
    assert int(jmg.potrf_(W).item()) == 0
    L = torch.tril(W)
    R = (A - L @ L.t()).abs().tril()
    s = A.diagonal().sqrt()
    # (2 n + 2) u s_i s_j as above, n u s_i s_j for this product
    assert bool((R <= (3 * n + 2) * U64 * s[:, None] * s[None, :]).all())


@pytest.mark.parametrize("n,nrhs", [(4230, 70), (8192, 19)])
def test_solve_with_some_spread_rows_and_columns(n, nrhs):
    g = torch.Generator(device=DEV).manual_seed(n)
    L = _spiky(n, g)
    B = torch.randn(n, nrhs, generator=g, dtype=torch.float64, device=DEV)
    B[:, ::3] = 0.0
    B[torch.randint(0, n, (40,), generator=g, device=DEV), 0] = 1.0  # sparse ones
    B[n - 1, ::3] = 1.0
    X = jmg.potrs_(jmg.colmajor_copy(L), jmg.colmajor_copy(B))
    R = (L @ (L.t() @ X) - B).abs()
    La = L.abs()
    assert bool((R <= 4 * (n + 2) * U64 * (La @ (La.t() @ X.abs()) + B.abs())).all())
