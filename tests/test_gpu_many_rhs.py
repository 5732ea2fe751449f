"""FP64 solves with many right-hand sides: the one-launch solves in batches of groups (the
scratch of jmg_workspace_size) and the blocked route from its line on, against
the system itself."""
from __future__ import annotations

import pytest
import torch

from helpers import DEV, U64
from paper_2601_14466_gb300 import inputs, jmg


@pytest.mark.gpu
@pytest.mark.parametrize("fast", [False, True])
@pytest.mark.parametrize("n,nrhs", [(33, 2000), (96, 1100), (97, 1100), (500, 700), (513, 1170),
                                    (1000, 150), (1025, 333), (2050, 101)])
def test_solve_satisfies_its_system(n, nrhs, fast):
    L = inputs.lower_factor(n, seed=n).to(DEV)
    B = inputs.uniform(n, nrhs, seed=nrhs).to(DEV)
    Ld, X = jmg.colmajor_copy(L), jmg.colmajor_copy(B)
    size = jmg.load().jmg_workspace_fast if fast else jmg.load().jmg_workspace_size
    work = torch.empty(int(size(jmg.OP_POTRS, n, nrhs, jmg.JMG_F64, None)), dtype=torch.uint8, device=DEV)
    st = jmg.load().jmg_potrs(n, nrhs, Ld.data_ptr(), n, X.data_ptr(), n, jmg.JMG_F64,
                              work.data_ptr(), work.numel(), torch.cuda.current_stream().cuda_stream)
    assert st == 0
    torch.cuda.synchronize()
    assert int(work[:4].view(torch.int32).item()) == 0
    La = L.abs()
    R = (L @ (L.t() @ X) - B).abs()
    # n u of |L| |L^T| |X| for either substitution, twice that for the products here
    assert bool((R <= 4 * (n + 2) * U64 * (La @ (La.t() @ X.abs()) + B.abs())).all())


def test_where_the_blocked_route_begins():
    def more(n, nrhs):
        return int(jmg.load().jmg_workspace_fast(jmg.OP_POTRS, n, nrhs, jmg.JMG_F64, None)) > \
            jmg.workspace_size(jmg.OP_POTRS, n, nrhs)

    for n, nrhs, want in ((512, 5000, False), (513, 1169, False), (513, 1170, True), (1000, 149, False),
                          (1000, 150, True), (4000, 100, False), (4000, 101, True)):
        assert more(n, nrhs) == want
