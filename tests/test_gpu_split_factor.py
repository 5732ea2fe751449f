"""FP64 factorisation with its updates in error-free slices on the tensor cores
(the route of jmg_potrf / jmg_posv when `work` holds jmg_workspace_fast bytes),
against its input and against the general route, at the edges of its tiles
(panels of 64 columns, tiles of 128 rows, blocks of 512 columns).

Tolerance: Cholesky in FP64 gives |A - L L^T|_ij <= gamma_(n+1) (|L| |L^T|)_ij,
and (|L| |L^T|)_ij <= sqrt(a_ii a_jj); the slices keep 2^-56 of each row's largest
element of the block, below sqrt(a_ii), and the products left out stay below
6 * 2^-56 of them, so n u sqrt(a_ii a_jj) covers both: (2 n + 2) u in all.
"""
from __future__ import annotations

import ctypes

import numpy as np
import pytest
import torch

import oracle
from helpers import DEV, U64, host, to_dev_colmajor
from paper_2601_14466_gb300 import inputs, jmg


def _factor(A: torch.Tensor, route: str, lda=None):
    view, _ = to_dev_colmajor(A, lda=lda)
    n = A.shape[0]
    info = torch.full((1,), 77, dtype=torch.int32, device=DEV)
    o = jmg.default_options()
    lib = jmg.load()
    nbytes = int(lib.jmg_workspace_fast(jmg.OP_POTRF, n, 1, jmg.JMG_F64, ctypes.byref(o)))
    work = torch.empty(max(nbytes, 256), dtype=torch.uint8, device=DEV)
    wp, wl = (work.data_ptr(), nbytes) if route == "split" else (None, 0)
    st = lib.jmg_potrf(n, view.data_ptr(), view.stride(1), jmg.JMG_F64, info.data_ptr(),
                       ctypes.byref(o), wp, wl, torch.cuda.current_stream().cuda_stream)
    assert st == 0
    torch.cuda.synchronize()
    return host(view), int(info.item())


def _backward(A: np.ndarray, L: np.ndarray) -> float:
    L = np.tril(L)
    s = np.sqrt(np.diag(A))
    R = (A - (L.astype(np.longdouble) @ L.T.astype(np.longdouble))) / np.outer(s, s)
    return float(np.max(np.abs(R)))


@pytest.mark.gpu
@pytest.mark.parametrize("n,lda", [(65, 65), (127, 130), (128, 128), (192, 193), (257, 257),
                                   (512, 512), (513, 515), (577, 577), (641, 641)])
@pytest.mark.parametrize("kind", ["gram", "graded", "ones"])
def test_split_factor_reproduces_its_input(n, lda, kind):
    A = inputs.gram_shift(n, 1.0, seed=inputs.seed_for("split", n))
    if kind == "graded":  # rows 16 decades apart
        d = torch.logspace(-8, 8, n, dtype=torch.float64)
        A = A * d[:, None] * d[None, :]
    elif kind == "ones":  # every digit of a row of L the same: the largest level sums
        A = torch.ones(n, n, dtype=torch.float64) + torch.eye(n, dtype=torch.float64)
    An = A.numpy()
    Lower = torch.tril(A) + torch.triu(torch.full_like(A, float("nan")), 1)
    L, info = _factor(Lower, "split", lda)
    assert info == 0
    assert np.isnan(L[np.triu_indices(n, 1)]).all()  # the upper triangle is neither read nor written
    assert _backward(An, L) <= (2 * n + 2) * U64


@pytest.mark.gpu
@pytest.mark.parametrize("n", [65, 640, 1100])
def test_split_factor_is_exact_on_integer_factors(n):
    Lt, A = inputs.integer_factor(n, seed=3)
    L, info = _factor(A, "split")
    assert info == 0
    np.testing.assert_array_equal(np.tril(L), Lt.numpy())


@pytest.mark.gpu
@pytest.mark.parametrize("n,k", [(130, 0), (130, 63), (130, 64), (700, 129), (700, 512), (700, 699)])
@pytest.mark.parametrize("bad", ["negative", "nan", "nan_below"])
def test_split_factor_reports_the_first_bad_pivot(n, k, bad):
    A = inputs.gram_shift(n, 1.0, seed=5)
    if bad == "negative":
        A[k, k] = -1.0
    elif bad == "nan":
        A[k, k] = float("nan")
    else:
        if k == 0:
            pytest.skip("no element left of the first pivot")
        A[k, k // 2] = A[k // 2, k] = float("nan")  # reaches pivot k through the updates
    want = _factor(A, "general")[1]
    assert want == k + 1
    assert _factor(A, "split")[1] == want


@pytest.mark.gpu
def test_posv_routes_agree_by_scratch():
    n, nrhs = 600, 5
    A = inputs.gram_shift(n, 1.0, seed=8)
    B = inputs.uniform(n, nrhs, seed=9)
    o = jmg.default_options()
    lib = jmg.load()
    X = {}
    for route, nbytes in (("general", jmg.workspace_size(jmg.OP_POSV, n, nrhs, o)),
                          ("split", int(lib.jmg_workspace_fast(jmg.OP_POSV, n, nrhs, jmg.JMG_F64,
                                                               ctypes.byref(o))))):
        work = torch.empty(nbytes, dtype=torch.uint8, device=DEV)
        x, _ = jmg.posv(to_dev_colmajor(A)[0], to_dev_colmajor(B)[0], prec="fp64", work=work)
        X[route] = host(x)
    for x in X.values():
        assert oracle.bwd_err(A.numpy(), x, B.numpy())[0] <= n * U64
    assert np.max(np.abs(X["split"] - X["general"])) <= 1e-12 * np.max(np.abs(X["general"]))


def test_fast_scratch_is_never_less_and_only_more_where_it_helps():
    lib = jmg.load()
    for prec, dt in (("fp64", jmg.JMG_F64), ("fp64", jmg.JMG_F32), ("bf16", jmg.JMG_F64),
                     ("fp32", jmg.JMG_F64)):
        o = jmg.default_options(prec=prec)
        for op in (jmg.OP_POTRF, jmg.OP_POTRS, jmg.OP_POSV, jmg.OP_POSV_HOST):
            for n in (0, 1, 64, 65, 1000, 65536):
                need = jmg.workspace_size(op, n, 3, o, dt)
                fast = int(lib.jmg_workspace_fast(op, n, 3, dt, ctypes.byref(o)))
                assert fast >= need
                more = prec == "fp64" and dt == jmg.JMG_F64 and n > 64 and op != jmg.OP_POTRS
                # (three right-hand sides: the solves never want more)
                assert (fast > need + 255) == more


def test_fast_scratch_of_the_solves_follows_their_shape():
    lib = jmg.load()
    for n, nrhs, more in ((4095, 100, False), (4096, 61, False), (4096, 62, True), (8192, 16, False),
                          (8192, 17, True), (65536, 17, True), (100000, 1, False)):
        need = jmg.workspace_size(jmg.OP_POTRS, n, nrhs)
        fast = int(lib.jmg_workspace_fast(jmg.OP_POTRS, n, nrhs, jmg.JMG_F64, None))
        assert (fast > need) == more and fast >= need
        assert int(lib.jmg_workspace_fast(jmg.OP_POTRS, n, nrhs, jmg.JMG_F32, None)) == \
            jmg.workspace_size(jmg.OP_POTRS, n, nrhs, None, jmg.JMG_F32)


@pytest.mark.gpu
@pytest.mark.parametrize("n,nrhs,pad", [(4096, 62, 0), (4097, 64, 1), (4608, 65, 0), (5121, 49, 2)])
@pytest.mark.parametrize("scaled", [False, True])
def test_split_solve_matches_substitution(n, nrhs, pad, scaled):
    # rows of L eight decades apart leave D X as it is for L -> D L, B -> D B: the same
    # bound holds for it (substitution: 64 n u as in the other solve tests; the slices
    # keep 2^-56 of a row's and a column's largest element in each block of 512)
    L = inputs.lower_factor(n, seed=3)
    B = inputs.uniform(n, nrhs, seed=4)
    Xo = oracle.potrs(np.asfortranarray(L.numpy()), B.numpy())
    d = torch.logspace(-4, 4, n, dtype=torch.float64)[torch.randperm(n, generator=torch.Generator().manual_seed(1))] \
        if scaled else torch.ones(n, dtype=torch.float64)
    lda, ldb = n + pad, n + 3
    Lb = torch.full((n, lda), float("nan"), dtype=torch.float64, device=DEV)
    Lb[:, :n] = (torch.tril(d[:, None] * L) + torch.triu(torch.full_like(L, float("nan")), 1)).t().to(DEV)
    Bb = torch.full((nrhs, ldb), float("nan"), dtype=torch.float64, device=DEV)
    Bb[:, :n] = (d[:, None] * B).t().to(DEV)
    lib = jmg.load()
    nbytes = int(lib.jmg_workspace_fast(jmg.OP_POTRS, n, nrhs, jmg.JMG_F64, None))
    assert nbytes > jmg.workspace_size(jmg.OP_POTRS, n, nrhs)
    work = torch.empty(nbytes, dtype=torch.uint8, device=DEV)
    st = lib.jmg_potrs(n, nrhs, Lb.data_ptr(), lda, Bb.data_ptr(), ldb, jmg.JMG_F64, work.data_ptr(),
                       nbytes, torch.cuda.current_stream().cuda_stream)
    assert st == 0
    torch.cuda.synchronize()
    assert int(work[:4].view(torch.int32).item()) == 0
    assert torch.isnan(Bb[:, n:]).all()
    X = Bb[:, :n].t().cpu().numpy() * d.numpy()[:, None]
    assert np.abs(X - Xo).max() <= 64 * n * U64 * max(1.0, np.abs(Xo).max())
