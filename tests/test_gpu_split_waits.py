"""The bounded waits of the FP64 kernels that form their products in slices: with a copy
producer that stays idle the first wait runs out, the kernel returns and reports it, what
it had not started on is untouched, and the next ordinary call is right."""
from __future__ import annotations

import numpy as np
import pytest
import torch

from helpers import DEV, U64, host, to_dev_colmajor
from paper_2601_14466_gb300 import inputs, jmg

pytestmark = pytest.mark.gpu
JMG_ERR_TIMEOUT = 5


@pytest.fixture
def short_waits():
    old = jmg.set_wait_limit_ns(1_000_000)  # 1 ms
    try:
        yield
    finally:
        jmg.set_wait_limit_ns(old)


def _fast(op, n, nrhs):
    nbytes = int(jmg.load().jmg_workspace_fast(op, n, nrhs, jmg.JMG_F64, None))
    return torch.empty(nbytes, dtype=torch.uint8, device=DEV)


def _stream():
    return torch.cuda.current_stream().cuda_stream


@pytest.mark.parametrize("n", [65, 700, 2600])
def test_factor_update_wait_runs_out(short_waits, n):
    A = inputs.gram_shift(n, 1.0, seed=inputs.seed_for("splitwait", n))
    Ad, _ = to_dev_colmajor(A)
    info = torch.full((1,), 77, dtype=torch.int32, device=DEV)
    work = _fast(jmg.OP_POTRF, n, 1)
    st = jmg.load().jmg_dev_oz_factor_idle_producer(n, Ad.data_ptr(), n, info.data_ptr(),
                                                    work.data_ptr(), work.numel(), _stream())
    assert st == 0
    torch.cuda.synchronize()  # returns: every wait gave up after the limit
    assert int(info.item()) == -1
    assert np.array_equal(host(Ad)[:, 64:], A.numpy()[:, 64:])
    jmg.set_wait_limit_ns(2_000_000_000)
    Ad, _ = to_dev_colmajor(A)
    assert int(jmg.potrf_(Ad).item()) == 0
    L = torch.tril(Ad)
    s = A.diagonal().sqrt().to(DEV)
    R = (A.to(DEV) - L @ L.t()).abs() / (s[:, None] * s[None, :])
    assert float(R.max()) <= (3 * n + 2) * U64  # (2 n + 2) u of the factor, n u of this product


def test_solve_update_wait_runs_out(short_waits):
    n, nrhs = 4096, 62
    L = inputs.lower_factor(n, seed=3)
    B = inputs.uniform(n, nrhs, seed=4)
    Ld, Bd = jmg.colmajor_copy(L.to(DEV)), jmg.colmajor_copy(B.to(DEV))
    work = _fast(jmg.OP_POTRS, n, nrhs)
    assert work.numel() > jmg.workspace_size(jmg.OP_POTRS, n, nrhs)
    st = jmg.load().jmg_dev_oz_solve_idle_producer(n, nrhs, Ld.data_ptr(), n, Bd.data_ptr(), n,
                                                   work.data_ptr(), work.numel(), _stream())
    assert st == 0
    torch.cuda.synchronize()
    assert int(work[:4].view(torch.int32).item()) == JMG_ERR_TIMEOUT
    assert torch.equal(Bd[512:].cpu(), B[512:])
    jmg.set_wait_limit_ns(2_000_000_000)
    Bd = jmg.colmajor_copy(B.to(DEV))
    st = jmg.load().jmg_potrs(n, nrhs, Ld.data_ptr(), n, Bd.data_ptr(), n, jmg.JMG_F64,
                              work.data_ptr(), work.numel(), _stream())
    assert st == 0
    Y = torch.linalg.solve_triangular(Ld, B.to(DEV), upper=False)
    X = torch.linalg.solve_triangular(Ld.mT, Y, upper=True)
    assert int(work[:4].view(torch.int32).item()) == 0
    assert float((Bd - X).abs().max()) <= 64 * n * U64 * max(1.0, float(X.abs().max()))


@pytest.mark.parametrize("n,nrhs", [(65, 12), (300, 35)])
def test_adjoint_wait_runs_out(short_waits, n, nrhs):
    Y, X = inputs.uniform(n, nrhs, seed=5).to(DEV), inputs.uniform(n, nrhs, seed=6).to(DEV)
    Yc, Xc = jmg.colmajor_copy(Y), jmg.colmajor_copy(X)
    G = torch.full((n, n), float("nan"), dtype=torch.float64, device=DEV)
    st = jmg.load().jmg_dev_sym_grad_no_products(n, nrhs, Yc.data_ptr(), n, Xc.data_ptr(), n,
                                                 G.data_ptr(), n, _stream())
    assert st == 0
    torch.cuda.synchronize()
    jmg.set_wait_limit_ns(2_000_000_000)
    want = -0.5 * (Y @ X.t() + X @ Y.t())
    tol = (2 * nrhs + 2) * U64 * (Y.abs() @ X.abs().t() + X.abs() @ Y.abs().t())
    assert bool(((G - want).abs() <= tol).all())
    assert bool(((jmg.sym_grad(Yc, Xc) - want).abs() <= tol).all())
