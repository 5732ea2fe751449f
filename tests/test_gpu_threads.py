"""Mixed solves issued by several threads on streams of their own: each prologue (norm and
slices of A, on a side stream that the threads share) has to wait for its own caller's
stream, where A is written just before the call."""
from __future__ import annotations

import threading

import pytest
import torch

from helpers import DEV
from paper_2601_14466_gb300 import inputs, jmg

pytestmark = pytest.mark.gpu


def test_prologue_follows_its_own_stream():
    n, nrhs, rounds = 700, 3, 6
    systems = [(inputs.gram_shift(n, 1.0, seed=60 + t).to(DEV), inputs.uniform(n, nrhs, seed=70 + t).to(DEV))
               for t in range(4)]
    big = torch.randn(3000, 3000, device=DEV)
    torch.cuda.synchronize()
    errors = []

    def work(t):
        A, B = systems[t]
        s = torch.cuda.Stream()
        with torch.cuda.stream(s):
            for _ in range(rounds):
                Ad = torch.full((n, n), float("nan"), dtype=torch.float64, device=DEV).t()
                for _ in range(4):
                    big @ big  # keeps the stream busy, so that A is written late
                Ad.copy_(A)
                X, info = jmg.posv(Ad, jmg.colmajor_copy(B), prec="bf16", words=2)
                s.synchronize()
                R = (B - A @ X).abs().amax(0)
                anorm = A.abs().sum(1).max()
                eta = float((R / (anorm * X.abs().amax(0) + B.abs().amax(0))).max())
                # the solve's target, and n u for the product of this check
                if not (info.status == 0 and eta <= 1e-13 + n * 2.0 ** -53
                        and abs(info.anorm - float(anorm)) <= n * 2.0 ** -52 * float(anorm)):
                    errors.append((t, info.status, eta, info.anorm, float(anorm)))

    threads = [threading.Thread(target=work, args=(t,)) for t in range(4)]
    for th in threads:
        th.start()
    for th in threads:
        th.join()
    assert not errors, errors
