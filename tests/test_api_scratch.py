"""Scratch of the Python calls (no GPU: the C calls are replaced by a record of
what they are given): scratch down to the least that the library accepts is
passed on, and without memory for the row buffer the least is allocated."""
import pytest
import torch

from paper_1912_07704_gb300 import abi
from paper_1912_07704_gb300.api import Plan

N, W = 20000, 64


class _Stream:
    cuda_stream = 0


@pytest.fixture
def plan(monkeypatch):
    p = Plan(1024, 1508.0, -300.0 / 1024, 64e-6, [(0.0, 0.1, 256, 1), (60.0, 0.2, 128, 2)])
    monkeypatch.setattr(Plan, "bind", lambda self: None)
    monkeypatch.setattr(Plan, "alloc_output", lambda self, n: torch.empty(self.query(n).dd_elems))
    yield p
    p.close()


@pytest.fixture
def given(monkeypatch):
    """ws_bytes of the C calls made"""
    seen = []
    monkeypatch.setattr(abi, "aa_dedisperse_device", lambda *a: seen.append(a[6]))
    return seen


def _least(plan):
    for r in range(2):  # what the direct kernels take: no row buffer
        plan.set_strategy(r, abi.AA_DEDISP_DIRECT)
    least = plan.query(N).dedisp_ws_bytes, plan.fused_ws_bytes(N, W)[0]
    for r in range(2):
        plan.set_strategy(r, abi.AA_DEDISP_GROUPED)
    return least


def test_least_scratch_is_known_and_passed_on(plan, given):
    least, fused = _least(plan)
    assert least < plan.query(N).dedisp_ws_bytes and fused <= plan.fused_ws_bytes(N, W)[0]
    ws = torch.empty(least, dtype=torch.uint8)
    plan.dedisperse_device(torch.empty((1024, N), dtype=torch.uint8), N, ws=ws, stream=_Stream())
    assert given == [least]
    assert abi.aa_dedisperse_least_ws_bytes(plan.handle, N) == least
    assert abi.aa_search_fused_least_ws_bytes(plan.handle, N, W) == fused
    with pytest.raises(abi.AAError):
        abi.aa_dedisperse_least_ws_bytes(plan.handle, -1)
    with pytest.raises(abi.AAError):
        abi.aa_search_fused_least_ws_bytes(plan.handle, N, 0)


def test_without_memory_for_the_row_buffer(plan, given, monkeypatch):
    least, _ = _least(plan)
    asked = []

    def alloc(self, nbytes):
        asked.append(nbytes)
        if nbytes > least:
            raise torch.cuda.OutOfMemoryError("full")
        return torch.empty(nbytes, dtype=torch.uint8)
    monkeypatch.setattr(Plan, "alloc_workspace", alloc)
    plan.dedisperse_device(torch.empty((1024, N), dtype=torch.uint8), N, stream=_Stream())
    assert asked == [plan.query(N).dedisp_ws_bytes, least] and given == [least]
    # nothing smaller to fall back to: the error stays
    for r in range(2):
        plan.set_strategy(r, abi.AA_DEDISP_DIRECT)
    monkeypatch.setattr(Plan, "alloc_workspace", lambda self, n: (_ for _ in ()).throw(torch.cuda.OutOfMemoryError("full")))
    with pytest.raises(torch.cuda.OutOfMemoryError):
        plan.dedisperse_device(torch.empty((1024, N), dtype=torch.uint8), N, stream=_Stream())
