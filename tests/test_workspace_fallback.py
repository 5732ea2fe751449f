"""Scratch of a call when the device has no room for the fastest route's: the call still
gets what it needs, and says that it takes the slower route."""
from __future__ import annotations

import warnings

import pytest
import torch

from paper_2601_14466_gb300 import jmg

N = 4096


def _sizes(op, nrhs):
    need = jmg.workspace_size(op, N, nrhs)
    return need, int(jmg.load().jmg_workspace_fast(op, N, nrhs, jmg.JMG_F64, None))


@pytest.mark.parametrize("op,nrhs", [(jmg.OP_POTRF, 1), (jmg.OP_POTRS, 64), (jmg.OP_POSV, 3)])
def test_the_slower_route_is_announced(monkeypatch, op, nrhs):
    need, fast = _sizes(op, nrhs)
    assert fast > need
    empty = torch.empty

    def full_device(n, **kw):
        if n > max(need, 256):
            raise torch.cuda.OutOfMemoryError("no room")
        return empty(n, **kw)

    monkeypatch.setattr(torch, "empty", full_device)
    with pytest.warns(RuntimeWarning, match=str(fast)):
        w = jmg.workspace(op, N, nrhs, None, "cpu")
    assert w.numel() == max(need, 256)


def test_no_warning_with_room_or_without_a_faster_route():
    with warnings.catch_warnings():
        warnings.simplefilter("error")
        assert jmg.workspace(jmg.OP_POTRF, N, 1, None, "cpu").numel() == _sizes(jmg.OP_POTRF, 1)[1]
        assert jmg.workspace(jmg.OP_POTRS, 100, 1, None, "cpu").numel() >= 256
