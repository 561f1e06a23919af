"""Two host threads, each with its own plan, buffers and stream, call the same
kernels with different amounts of dynamic shared memory: every call is
accepted (the limit is a property of the kernel, not of the launch) and gives
the result of the plan alone."""
import threading

import pytest
import torch

from paper_1912_07704_gb300 import abi, synth
from paper_1912_07704_gb300.api import Plan

pytestmark = pytest.mark.gpu

CALLS = 1500


def _dedisp(nchans, ranges, nsamp, prepare):
    plan = Plan(nchans, 1508.0, -300.0 / nchans, 64e-6, ranges)
    for r in range(len(ranges)):
        prepare(plan, r)
    x, n = plan.device_input(synth.noise_filterbank(nchans, nsamp, 5, device="cuda"))
    plan.bind()
    q = plan.query(n)
    out = torch.zeros(q.dd_elems, device="cuda")
    ws = plan.alloc_workspace(q.dedisp_ws_bytes)

    def call(stream):
        plan.dedisperse_device(x, n, out=out, ws=ws, stream=stream)
    return plan, call, lambda: torch.cat([v.flatten() for v in plan.range_views(out, n)])


def _boxcar(width, dec):
    L = 5000
    plan = Plan(16, 1400.0, -1.0, 64e-6, [(0.0, 0.0, 2, 1)])
    plan.bind()
    plan.set_sps_decimated(dec)
    q = plan.query(L, width)
    dd = torch.zeros(q.dd_elems, device="cuda")
    plan.range_views(dd, L)[0].copy_((torch.arange(2 * L, device="cuda").view(2, L) * 37 % 101 + 4000).float())
    ws, snr = plan.alloc_workspace(q.sps_ws_bytes), torch.zeros_like(dd)
    cands, count = torch.empty(16 * L, dtype=torch.uint8, device="cuda"), torch.zeros(1, dtype=torch.int64, device="cuda")

    def call(stream):
        plan.sps_search_device(dd, L, width, 50.0, L, snr_out=snr, ws=ws, cands=cands, count=count, stream=stream)
    return plan, call, lambda: plan.range_views(snr, L)[0].flatten()


def _float(step):
    plan = Plan(64, 1508.0, -300.0 / 64, 64e-6, [(0.0, step, 32, 1)])
    plan.bind()
    n = 4096
    x, w = torch.arange(64.0 * n, device="cuda").remainder(97).view(64, n), torch.ones(64, device="cuda")
    out = plan.alloc_output(n).zero_()

    def call(stream):
        plan.f32_forward(x, w, out=out, stream=stream)
    return plan, call, lambda: torch.cat([v.flatten() for v in plan.range_views(out, n)])


def _pair(kind):
    if kind == "tree":
        fdmt = lambda p, r: p.set_fdmt(r)
        return (_dedisp(16, [(0.0, 0.5, 8, 1)], 600, fdmt), _dedisp(256, [(0.0, 0.5, 64, 1), (32.0, 1.0, 20, 2)], 4000, fdmt))
    if kind == "bands":
        grouped = lambda p, r: p.set_strategy(r, abi.AA_DEDISP_GROUPED)
        return (_dedisp(512, [(0.0, 0.1, 64, 1)], 2000, grouped), _dedisp(1024, [(0.0, 0.3, 128, 1)], 4000, grouped))
    if kind == "grouped":  # without the row buffer's bands: trials below half a block
        grouped = lambda p, r: p.set_strategy(r, abi.AA_DEDISP_GROUPED)
        return (_dedisp(64, [(0.0, 0.1, 16, 1)], 2000, grouped), _dedisp(256, [(0.0, 5.0, 16, 1)], 4000, grouped))
    if kind == "direct":
        direct = lambda p, r: p.set_strategy(r, abi.AA_DEDISP_DIRECT)
        return (_dedisp(8, [(0.0, 0.1, 320, 1)], 2000, direct), _dedisp(8, [(0.0, 3.0, 320, 1)], 18000, direct))
    if kind == "sub-band":
        return (_dedisp(64, [(0.0, 0.1, 16, 1)], 2000, lambda p, r: p.set_subband(r, 8, 4)),
                _dedisp(64, [(0.0, 2.0, 64, 1)], 6000, lambda p, r: p.set_subband(r, 32, 16)))
    if kind == "boxcar":
        return _boxcar(16, 0), _boxcar(2048, 0)
    if kind == "boxcar-decimated":
        return _boxcar(64, 16), _boxcar(2048, 64)
    return _float(0.1), _float(2.0)


@pytest.mark.parametrize("kind", ["tree", "bands", "grouped", "direct", "sub-band", "boxcar", "boxcar-decimated", "float"])
def test_two_threads_with_different_shared_memory(kind):
    if kind == "bands":  # (also where the grouped kernel would be the faster side)
        abi.aa_debug_inject(4, 1)
    try:
        _run(_pair(kind))
    finally:
        abi.aa_debug_inject(0, 0)


def _run(pairs):
    want = []
    for _, call, result in pairs:
        call(None)
        torch.cuda.synchronize()
        want.append(result().clone())
    failures = []
    start = threading.Barrier(2)

    def work(call):
        stream = torch.cuda.Stream()
        start.wait()
        try:
            for _ in range(CALLS):
                call(stream)
        except Exception as e:  # noqa: BLE001 (reported below)
            failures.append(e)
        stream.synchronize()

    torch.cuda.synchronize()
    threads = [threading.Thread(target=work, args=(call,)) for _, call, _ in pairs]
    for t in threads:
        t.start()
    for t in threads:
        t.join()
    assert not failures, failures
    torch.cuda.synchronize()
    for (plan, _, result), w in zip(pairs, want):
        assert torch.equal(result(), w)
        plan.close()
