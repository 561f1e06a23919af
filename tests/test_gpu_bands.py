"""Band rows of the grouped strategy against the direct kernel (bit for bit):
last bands of 1 to 8 channels, parts of blocks and segments, one tile and
several slabs, both halves of a word past the series end, and the least
scratch, with which the grouped kernel runs instead.  Short outputs included:
band rows run here wherever they fit, not only where they are the faster side."""
import time

import pytest
import torch

from paper_1912_07704_gb300 import abi, synth
from paper_1912_07704_gb300.api import Plan

pytestmark = pytest.mark.gpu


@pytest.fixture(autouse=True)
def _wherever_they_fit():
    abi.aa_debug_inject(4, 1)
    yield
    abi.aa_debug_inject(0, 0)


CASES = [  # nchans, foff, ranges, output samples of the first range
    (1024, -300.0 / 1024, ((0.0, 0.1, 600, 1), (60.0, 0.2, 70, 2)), 1),
    (1001, -0.3, ((0.0, 0.1, 65, 1), (7.0, 0.1, 513, 3)), 511),
    (1004, -0.3, ((3.0, 0.2, 64, 1), (300.0, 0.5, 100, 4)), 513),
    (1005, -0.3, ((0.0, 0.05, 1025, 1),), 20001),
    (1007, -0.3, ((0.0, 0.0, 70, 1), (50.0, 0.3, 200, 16)), 33000),
    (800, 0.375, ((0.0, 0.1, 300, 1), (30.0, 0.4, 150, 5)), 12345),  # rising band
    (4096, -300.0 / 4096, ((0.0, 0.1, 130, 1), (600.0, 1.0, 66, 8)), 40000),
]


def _run(plan, x, nsamp, ws_bytes):
    out = torch.full((plan.query(nsamp).dd_elems,), -1.0, device="cuda")
    ws = torch.full((ws_bytes,), 0xA5, dtype=torch.uint8, device="cuda")  # the row buffer starts as garbage
    abi.aa_dedisperse_device(plan.handle, x.data_ptr(), nsamp, x.stride(0), out.data_ptr(), ws.data_ptr(), ws.numel(),
                             torch.cuda.current_stream().cuda_stream)
    assert abi.aa_workspace_status(ws.data_ptr(), torch.cuda.current_stream().cuda_stream) == abi.AA_OK
    return out


@pytest.mark.parametrize("case", range(len(CASES)))
@pytest.mark.parametrize("data", ["noise", "saturated"])
def test_bands_equal_the_direct_kernel(case, data):
    C, foff, ranges, length = CASES[case]
    plan = Plan(C, 1508.0 if foff < 0 else 1208.0, foff, 64e-6, ranges)
    nsamp = length + int(plan.shifts(0).max())
    plan.bind()
    x, n = plan.device_input(synth.noise_filterbank(C, nsamp, 31 + case, device="cuda"))
    if data == "saturated":  # the largest sums in every 16-bit lane, and whatever lies behind the rows' ends
        x.fill_(255)
    for r in range(len(ranges)):
        plan.set_strategy(r, abi.AA_DEDISP_DIRECT)
    base = plan.query(n).dedisp_ws_bytes
    want = _run(plan, x, n, base)
    for r in range(len(ranges)):
        plan.set_strategy(r, abi.AA_DEDISP_GROUPED)
    full = plan.query(n).dedisp_ws_bytes
    assert full > base
    for nbytes in (full, base + (full - base) // 3, base):
        got = _run(plan, x, n, nbytes)
        for a, b in zip(plan.range_views(got, n), plan.range_views(want, n)):
            assert torch.equal(a, b), nbytes


@pytest.mark.parametrize("band", [0, 1, 34, 99])
@pytest.mark.parametrize("length, ranges", [(700, ((0.0, 0.1, 70, 1),)), (40000, ((0.0, 0.1, 700, 1),)),
                                            (1500, ((160.0, 2.0, 70, 16),))])
def test_bounded_wait_reports_timeout(length, ranges, band):
    """Copies of a band that are never issued make every CTA of the sums give up
    after the wait limit without writing output (halves and whole tiles, two
    pairs of bands a round and one); the next call is clean."""
    plan = Plan(800, 1508.0, -0.375, 64e-6, ranges)
    plan.bind()
    nsamp = (length + int(plan.shifts(0).max())) * ranges[0][3]
    x, n = plan.device_input(synth.noise_filterbank(800, nsamp, 3, device="cuda"))
    plan.set_strategy(0, abi.AA_DEDISP_DIRECT)
    want = _run(plan, x, n, plan.query(n).dedisp_ws_bytes)
    plan.set_strategy(0, abi.AA_DEDISP_GROUPED)
    nbytes = plan.query(n).dedisp_ws_bytes
    assert nbytes > abi.aa_dedisperse_least_ws_bytes(plan.handle, n)
    out, ws = torch.full_like(want, -1.0), plan.alloc_workspace(nbytes)
    stream = torch.cuda.current_stream().cuda_stream
    try:
        abi.aa_debug_inject(2, 20_000_000)  # 20 ms
        abi.aa_debug_inject(1, band)
        torch.cuda.synchronize()
        t0 = time.perf_counter()
        plan.dedisperse_device(x, n, out=out, ws=ws)
        assert abi.aa_workspace_status(ws.data_ptr(), stream) == abi.AA_ERR_TIMEOUT
        assert time.perf_counter() - t0 < 1.5  # six waves of CTAs at most, two limits each; the default limit is 2 s
    finally:
        abi.aa_debug_inject(0, 0)
        abi.aa_debug_inject(4, 1)
    assert torch.all(out == -1.0)
    got = _run(plan, x, n, nbytes)
    assert torch.equal(plan.range_views(got, n)[0], plan.range_views(want, n)[0])


@pytest.mark.parametrize("stripe", [16, 64, 0])
def test_bands_in_the_fused_search(stripe):
    """Stripes on band rows (every decimation, read from the decimated input
    or decimated by the row kernel; row sums added by its epilogue) give the
    unfused direct path's candidates and B(t); also with the least scratch."""
    from paper_1912_07704_gb300.api import candidates_from_device
    C, nsamp, W, thr, cap = 1003, 30011, 24, 4.5, 1 << 18
    ranges = ((0.0, 0.1, 70, 1), (10.0, 0.2, 64, 2), (30.0, 0.5, 40, 3), (60.0, 1.0, 64, 4), (100.0, 1.0, 64, 8), (160.0, 2.0, 70, 16))
    plan = Plan(C, 1508.0, -0.3, 64e-6, ranges)
    x, n = plan.device_input(synth.noise_filterbank(C, nsamp, 77, device="cuda"))
    for r in range(len(ranges)):
        plan.set_strategy(r, abi.AA_DEDISP_DIRECT)
    least = plan.fused_ws_bytes(n, W, stripe)[0]
    dd = plan.dedisperse_device(x, n)
    snr = torch.zeros_like(dd)
    c, count, _ = plan.sps_search_device(dd, n, W, thr, cap, snr_out=snr)
    want = candidates_from_device(c, count, cap)
    assert len(want) > 0
    for r in range(len(ranges)):
        plan.set_strategy(r, abi.AA_DEDISP_GROUPED)
    for nbytes in (plan.fused_ws_bytes(n, W, stripe)[0], plan.fused_ws_bytes(n, W, stripe)[0] + (64 << 20), least):
        got = torch.zeros_like(dd)
        ws = torch.full((nbytes,), 0x5A, dtype=torch.uint8, device="cuda")
        c, count, _ = plan.search_fused_device(x, n, W, thr, cap, stripe, snr_out=got, ws=ws)
        assert (candidates_from_device(c, count, cap) == want).all()
        for a, b in zip(plan.range_views(got, n), plan.range_views(snr, n)):
            assert torch.equal(a, b)
