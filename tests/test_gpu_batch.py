"""Batched beams (one CUDA graph: each beam's kernels on concurrent branches,
or persistent work-queue kernels per stage) against the same beams run one
at a time, and the autotuner."""
import os

import numpy as np
import pytest
import torch

from paper_1912_07704_gb300 import abi, synth
from paper_1912_07704_gb300.api import Batch, Plan, candidates_from_device

pytestmark = pytest.mark.gpu

BEAMS = [
    (64, 1400.0, -4.0, 21001, [(0.0, 4.0, 23, 1), (92.0, 6.0, 17, 2)]),
    (128, 1500.0, -2.0, 30011, [(0.0, 3.0, 40, 1), (120.0, 5.0, 9, 4), (165.0, 9.0, 7, 16)]),
    (64, 1300.0, -3.0, 9000, [(10.0, 2.0, 5, 2)]),
    (96, 1450.0, -2.5, 17777, [(0.0, 1.0, 33, 1), (33.0, 2.0, 12, 8)]),
]
W, THR = 64, 5.0


def make_beams(oracle):
    plans, data = [], []
    for k, (C, fch1, foff, T, ranges) in enumerate(BEAMS):
        w = synth.Workload(f"b{k}", C, fch1, foff, 64e-6, T, tuple(ranges), W, THR, 20 + k)
        pulses = [synth.Pulse(ranges[0][0] + ranges[0][1] * 2, T // 3, 6, 30.0)]
        x = synth.make_filterbank(w, pulses, lambda dm: oracle.shifts(C, fch1, foff, 64e-6, dm, 1))
        plans.append(Plan(C, fch1, foff, 64e-6, ranges))
        data.append(x.numpy())
    return plans, data


def single(plan, x):
    d, nsamp = plan.device_input(x)
    out = plan.dedisperse_device(d, nsamp)
    cands, count, _ = plan.sps_search_device(out, nsamp, W, THR, 1 << 16)
    torch.cuda.synchronize()
    return candidates_from_device(cands, count, 1 << 16)


def batched(plans, data, budget=0):
    b = Batch(plans, [x.shape[1] for x in data], W, THR, capacity=1 << 18, wave_budget=budget)
    for i, x in enumerate(data):
        b.input_view(i)[:, : x.shape[1]].copy_(torch.from_numpy(x))
    b.run()
    arr, total = b.candidates()
    return b, arr, total


def split(arr, n):
    out = []
    for i in range(n):
        a = arr[arr["reserved"] == i].copy()
        a["reserved"] = 0
        out.append(a)
    return out


@pytest.mark.parametrize("budget", [0, 1], ids=["one-wave", "wave-per-beam"])
def test_batch_equals_beams_alone(oracle, budget):
    plans, data = make_beams(oracle)
    b, arr, total = batched(plans, data, budget)
    assert b.info()[0] == (1 if budget == 0 else len(BEAMS))
    per = split(arr, len(BEAMS))
    assert sum(len(a) for a in per) == total == len(arr)
    n_nonempty = 0
    for i, (p, x) in enumerate(zip(plans, data)):
        ref = single(p, x)
        assert np.array_equal(per[i], ref), f"beam {i}"
        n_nonempty += len(ref) > 0
    assert n_nonempty >= 3
    # a second replay of the graph gives the same list
    b.run()
    arr2, total2 = b.candidates()
    assert total2 == total and np.array_equal(arr2, arr)
    b.close()


@pytest.mark.parametrize("budget", [0, 1], ids=["one-wave", "wave-per-beam"])
@pytest.mark.parametrize("branches", [1, 3])
def test_branched_graph_equals_persistent(oracle, budget, branches):
    """Every graph form (8 branches at creation, 1 or 3 branches, the
    persistent work-queue kernels) finds the same candidates and the same
    dedispersed series; switching re-records the graph without touching the
    buffers."""
    plans, data = make_beams(oracle)
    b, arr, total = batched(plans, data, budget)
    b.set_branches(branches)
    b.run()
    arr_b, total_b = b.candidates()
    assert total_b == total and np.array_equal(arr_b, arr)
    for i, (p, x) in enumerate(zip(plans, data)):
        if b.info()[0] == 1 or i == len(BEAMS) - 1:  # series kept by the last wave only
            d, nsamp = p.device_input(x)
            ref = p.range_views(p.dedisperse_device(d, nsamp), nsamp)
            got = p.range_views(b.dd_view(i), nsamp)
            assert all(torch.equal(u, v) for u, v in zip(got, ref)), f"beam {i}"
    b.set_branches(0)
    b.run()
    arr_p, total_p = b.candidates()
    assert total_p == total and np.array_equal(arr_p, arr)
    with pytest.raises(Exception):
        b.set_branches(65)
    b.close()


def test_autotune_keeps_results_and_caches(tmp_path, oracle):
    C, fch1, foff, T, ranges = BEAMS[1]
    x = synth.noise_filterbank(C, T, seed=3).numpy()
    p0 = Plan(C, fch1, foff, 64e-6, ranges)
    d, nsamp = p0.device_input(x)
    ref = p0.dedisperse_device(d, nsamp).clone()
    cache = tmp_path / "tune.txt"
    p1 = Plan(C, fch1, foff, 64e-6, ranges)
    p1.autotune(nsamp, str(cache))
    assert cache.exists() and len(cache.read_text().strip().splitlines()) == len(ranges)
    out1 = p1.dedisperse_device(d, nsamp)
    p2 = Plan(C, fch1, foff, 64e-6, ranges)
    p2.autotune(nsamp, str(cache))  # served from the cache
    assert len(cache.read_text().strip().splitlines()) == len(ranges)
    out2 = p2.dedisperse_device(d, nsamp)
    torch.cuda.synchronize()
    for a, b_, c in zip(p0.range_views(ref, nsamp), p1.range_views(out1, nsamp),
                        p2.range_views(out2, nsamp)):
        assert torch.equal(a, b_) and torch.equal(a, c)


@pytest.mark.parametrize("thr", [6.0, -0.25])
def test_persistent_search_prunes(thr):
    """The work-queue form's search skips widths by bounds as the branches' does
    (with every width evaluated noise took it four times their time), and below
    a threshold of zero finds what they find."""
    plans = [Plan(64, 1508.0, -300.0 / 64, 64e-6, [(0.0, 1.0, 64, 1)]) for _ in range(4)]
    xs = [synth.noise_filterbank(64, 30000 + 999 * i, 3 + i, device="cuda") for i in range(4)]
    b = Batch(plans, [x.shape[1] for x in xs], 1024, thr, capacity=1 << 22)
    for i, x in enumerate(xs):
        b.input_view(i)[:, : x.shape[1]].copy_(x)
    ms, found = {}, {}
    e = [torch.cuda.Event(enable_timing=True) for _ in range(2)]
    for branches in (8, 0):
        b.set_branches(branches)
        b.run()
        e[0].record()
        for _ in range(5):
            b.run()
        e[1].record()
        torch.cuda.synchronize()
        ms[branches] = e[0].elapsed_time(e[1]) / 5
        found[branches] = b.candidates()
    assert found[0][1] == found[8][1] and np.array_equal(found[0][0], found[8][0])
    assert thr < 0 or ms[0] < 2 * ms[8], ms
    assert thr > 0 or found[0][1] > 0
    b.close()


@pytest.mark.parametrize("C, step, trials, kernel", [(256, 1.0, 256, abi.AA_DEDISP_DIRECT),      # hardly a shared delay pattern
                                                     (1024, 0.1, 300, abi.AA_DEDISP_GROUPED)])
def test_autotune_leaves_band_rows_to_the_launch(tmp_path, C, step, trials, kernel):
    """The tuner chooses among the strategies' own kernels (at DM step 1 over
    256 channels the grouped one is the slower), and neither its choice nor a
    cached "direct" takes band rows from the plan."""
    make = lambda: Plan(C, 1508.0, -300.0 / C, 64e-6, [(0.0, step, trials, 1)])
    n, cache = 40000, tmp_path / "tune.txt"
    p = make()
    least = abi.aa_dedisperse_least_ws_bytes(p.handle, n)
    assert p.query(n).dedisp_ws_bytes > least
    p.autotune(n, str(cache))
    assert abi.aa_plan_range(p.handle, n, 0).strategy == kernel
    assert p.query(n).dedisp_ws_bytes > least
    p.close()
    key, _, cc, ns, ms = cache.read_text().split()
    cache.write_text(f"{key} {abi.AA_DEDISP_DIRECT} 8 2 {ms}\n")
    p = make()
    p.autotune(n, str(cache))
    assert abi.aa_plan_range(p.handle, n, 0).strategy == abi.AA_DEDISP_DIRECT  # served from the cache
    assert p.query(n).dedisp_ws_bytes > least
    p.close()
    cache.write_text(f"{key.replace(';v2', '')} {abi.AA_DEDISP_DIRECT} 8 2 {ms}\n")  # a line of an older library
    p = make()
    p.autotune(n, str(cache))
    assert len(cache.read_text().splitlines()) == 2  # timed again
    p.close()


def test_autotune_times_the_shapes_on_a_short_probe(tmp_path):
    """Calls of a few blocks run on a kernel without shapes; the tuner times the
    staged one all the same (there about three times the small one's time)."""
    p = Plan(1024, 1508.0, -300.0 / 1024, 64e-6, [(0.0, 5.0, 20, 1)])
    x, n = p.device_input(synth.noise_filterbank(1024, 6000 + int(p.shifts(0).max()), 4, device="cuda"))
    p.set_strategy(0, abi.AA_DEDISP_DIRECT)
    out, ws = p.alloc_output(n), p.alloc_workspace(p.query(n).dedisp_ws_bytes)
    e = [torch.cuda.Event(enable_timing=True) for _ in range(2)]
    for _ in range(2):
        e[0].record()
        for _ in range(20):
            p.dedisperse_device(x, n, out=out, ws=ws)
        e[1].record()
        torch.cuda.synchronize()
    small_ms = e[0].elapsed_time(e[1]) / 20
    p.autotune(n, str(tmp_path / "tune.txt"))
    line = (tmp_path / "tune.txt").read_text().split()
    assert int(line[1]) == abi.AA_DEDISP_DIRECT and float(line[4]) > 1.5 * small_ms
    p.close()


@pytest.mark.parametrize("step, nsamp", [(0.3, 100000), (1.0, 110000)])
def test_row_buffers_hold_what_band_rows_take(step, nsamp):
    """4096 channels whose rows take 0.8 GB at least: the branches that such
    beams run on get that much, so that they run on band rows (a wait left to
    run out by a copy that is never issued shows it: the grouped kernel has no
    such copy); results are those of the beams alone, for any number of branches."""
    wide = [(0.0, step, 1500, 1)]
    specs = [(4096, wide, nsamp), (1024, [(0.0, 0.5, 100, 1), (50.0, 1.0, 64, 2)], 30000), (4096, wide, nsamp - 999), (256, [(0.0, 1.0, 40, 1)], 5000)]
    plans = [Plan(C, 1508.0, -300.0 / C, 64e-6, ranges) for C, ranges, _ in specs]
    for i in (0, 2):
        plans[i].set_strategy(0, abi.AA_DEDISP_GROUPED)
    xs = [synth.noise_filterbank(C, n, 8 + i, device="cuda") for i, (C, _, n) in enumerate(specs)]
    cap, thr = 1 << 20, 5.5

    def batch(which):
        b = Batch([plans[i] for i in which], [specs[i][2] for i in which], 16, thr, capacity=cap)
        for k, i in enumerate(which):
            b.input_view(k)[:, : specs[i][2]].copy_(xs[i])
        return b
    try:
        abi.aa_debug_inject(2, 2_000_000)  # 2 ms
        abi.aa_debug_inject(1, 5)
        b = batch([0, 2])
        b.run()
        with pytest.raises(abi.AAError, match="AA_ERR_TIMEOUT"):
            b.candidates()
        b.close()
    finally:
        abi.aa_debug_inject(0, 0)
    alone = []
    for p, x, (_, _, n) in zip(plans, xs, specs):
        d, _ = p.device_input(x)
        c, count, _ = p.sps_search_device(p.dedisperse_device(d, n), n, 16, thr, cap)
        alone.append(candidates_from_device(c, count, cap))
    assert sum(len(a) for a in alone) > 0
    b = batch([0, 1, 2, 3])
    for branches in (8, 1, 3, 64):
        b.set_branches(branches)
        b.run()
        arr, total = b.candidates()
        assert total == sum(len(a) for a in alone)
        for a, want in zip(split(arr, 4), alone):
            assert np.array_equal(a, want)
    b.close()
