"""The boxcar search's pruning, at the widths where its groups of chunks begin
and end (16, 128, 1024, 8192 widths and one more or less) and where the map's
widths cease to be evaluated in turn (2048 for so few series): the B(t) map equals
the maximum over every width in 64 bits, and the pruned search (no map) finds
exactly the peaks of the map at widths that have their SNR, for a usual threshold
and one below zero."""
import math

import numpy as np
import pytest
import torch

from paper_1912_07704_gb300 import abi
from paper_1912_07704_gb300.api import Plan, candidates_from_device

pytestmark = pytest.mark.gpu

ROWS, L = 3, 21007


def _series(kind):
    g = torch.Generator(device="cuda")
    g.manual_seed(5)
    y = (torch.randn((ROWS, L), generator=g, device="cuda") * 50 + 4000).round()
    if kind == "pulses":  # narrow, a block wide, and wider than a group of 64 chunks
        y[0, 5000:5007] += 400
        y[0, 12000:12300] += 120
        y[1, 3000:6500] += 25
        y[1, 15000:15020] += 300
        y[2, 9000:9001] += 2000
    elif kind == "ramp":  # rising then falling: long stretches of negative sums
        y += torch.linspace(-40, 40, L, device="cuda").round() * torch.tensor([[1.0], [-1.0], [0.0]], device="cuda")
    elif kind == "flat":  # from one start on sums grow like sqrt(w): it has hundreds of chunks to evaluate
        y = 4000 + ((y - 4000) / 25).round()
        for row, s in enumerate((100, 5003, 12000)):
            k = torch.arange(L - s + 1, device="cuda", dtype=torch.float64)
            y[row, s:] += torch.diff((2000 * k.sqrt()).round()).float()
    return y


def _prefix(y):
    y = y.double()
    mu, sigma = y.mean(1, keepdim=True), y.std(1, keepdim=True, unbiased=False)
    P = torch.zeros((ROWS, L + 1), dtype=torch.float64, device="cuda")
    torch.cumsum(y - mu, 1, out=P[:, 1:])
    return P, sigma


def _best(y, W):
    """max over every width in 64 bits"""
    P, sigma = _prefix(y)
    best = torch.full_like(P[:, :L], -math.inf)
    for w in range(1, min(W, L) + 1):
        v = (P[:, w:] - P[:, :L + 1 - w]) / (sigma * math.sqrt(w))
        torch.maximum(best[:, :L + 1 - w], v, out=best[:, :L + 1 - w])
    return best


def _snr_at(y, rec):
    """of each record's window, in 64 bits"""
    P, sigma = _prefix(y)
    row, t, w = (torch.from_numpy(rec[k].astype(np.int64)).cuda() for k in ("dm_index", "t", "width"))
    assert bool(((w >= 1) & (t + w <= L)).all())
    return (P[row, t + w] - P[row, t]) / (sigma[row, 0] * w.double().sqrt())


@pytest.mark.parametrize("W", [1, 16, 17, 127, 129, 1024, 1025, 2048, 2049, 4100, 8191, 8193, 9000])
@pytest.mark.parametrize("kind", ["noise", "pulses", "ramp", "flat"])
def test_pruned_search_equals_the_map(W, kind):
    """Whatever the tiles a CTA takes (1, 3 and 7 of the 6 of a series: sliding
    the staged sums, the new samples copied ahead)."""
    plan = Plan(16, 1400.0, -1.0, 64e-6, [(0.0, 0.0, ROWS, 1)])
    plan.bind()
    info = plan.query(L, W)
    dd = torch.zeros(info.dd_elems, device="cuda")
    y = _series(kind)
    plan.range_views(dd, L)[0].copy_(y)
    want = _best(y, W)
    cap = ROWS * L
    for thr in (4.0, -0.5):
        first = None
        for tiles in (1, 3, 7):
            try:
                abi.aa_debug_inject(3, tiles)
                snr = torch.full_like(dd, float("nan"))
                with_map, count, _ = plan.sps_search_device(dd, L, W, thr, cap, snr_out=snr)
                pruned, n2, _ = plan.sps_search_device(dd, L, W, thr, cap)
            finally:
                abi.aa_debug_inject(0, 0)
            got = plan.range_views(snr, L)[0]
            rec = candidates_from_device(pruned, n2, cap)
            assert int(count) == int(n2)
            assert np.array_equal(candidates_from_device(with_map, count, cap), rec)  # widths included
            if first is None:
                assert torch.allclose(got.double(), want, rtol=2e-6, atol=1e-4)
                b = got.cpu().numpy()
                left = np.concatenate([np.full((ROWS, 1), -np.inf, np.float32), b[:, :-1]], 1)
                right = np.concatenate([b[:, 1:], np.full((ROWS, 1), -np.inf, np.float32)], 1)
                rows, ts = np.nonzero((b >= thr) & (b > left) & (b >= right))
                assert np.array_equal(rec["dm_index"], rows) and np.array_equal(rec["t"], ts)
                assert np.array_equal(rec["snr"], b[rows, ts])
                # the record's width is one that has its SNR (FP32 of the same sum)
                at = _snr_at(y, rec)
                assert torch.allclose(torch.from_numpy(rec["snr"].copy()).cuda().double(), at, rtol=2e-6, atol=1e-4)
                first = rec, got.clone()
            else:
                assert np.array_equal(rec, first[0]) and torch.equal(got, first[1]), tiles
    plan.close()
