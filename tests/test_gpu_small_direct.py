"""The direct strategy's kernel for few output samples (one trial x 128 samples
a block): exact sums at the edges of its tiles, for channel counts around its
warps and its 16-bit accumulators' limit, both input types, and the row sums of
the fused search."""
import numpy as np
import pytest
import torch

from gpu_common import run_gpu
from paper_1912_07704_gb300 import abi
from paper_1912_07704_gb300.api import Plan

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("nchans,nsamp,ndm,step,dec", [
    (1, 1, 1, 0.0, 1), (7, 129, 3, 1.0, 1), (8, 1000, 17, 2.0, 1), (9, 4096, 33, 4.0, 2),
    (65, 6001, 20, 4.0, 3), (2049, 2050, 5, 3.0, 1), (2100, 1999, 9, 0.5, 16), (300, 40000, 1, 0.0, 1),
])
def test_small_direct_sums_are_exact(nchans, nsamp, ndm, step, dec):
    rng = np.random.default_rng(nchans + nsamp)
    x = rng.integers(0, 256, size=(nchans, nsamp), dtype=np.uint8)
    x[:, nsamp // 2:] = 255  # full lanes
    with Plan(nchans, 1400.0, -200.0 / nchans, 64e-6, [(0.0, step, ndm, dec)]) as plan:
        plan.set_strategy(0, abi.AA_DEDISP_DIRECT)
        out, _, cands, total, _ = run_gpu(plan, x, 8, 6.0)
        s = plan.shifts(0)
        z = x[:, :nsamp // dec * dec].reshape(nchans, -1, dec).sum(2, dtype=np.int64)
        n = z.shape[1] - int(s.max())
        want = np.stack([sum(z[c, s[i, c]:s[i, c] + n] for c in range(nchans)) for i in range(ndm)])
        got = plan.range_views(out, nsamp)[0]
        assert n > 0 and np.array_equal(got.double().cpu().numpy(), want.astype(np.float64))
        # the fused search takes its statistics from the same kernel's sums
        pitch = (nsamp + 15) // 16 * 16
        d = torch.zeros((nchans, pitch), dtype=torch.uint8, device="cuda")
        d[:, :nsamp] = torch.from_numpy(x).cuda()
        cap = ndm * n + 1
        nbytes, _ = plan.fused_ws_bytes(nsamp, 8)
        ws = plan.alloc_workspace(nbytes)
        fc = torch.zeros(cap * 16, dtype=torch.uint8, device="cuda")
        count = torch.zeros(1, dtype=torch.int64, device="cuda")
        plan.search_fused_device(d, nsamp, 8, 6.0, cap, ws=ws, cands=fc, count=count)
        assert int(count) == total
