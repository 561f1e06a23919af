"""What the library's speed is measured on: calls a user's program makes, through the public entry points.

A case is one call (or the short chain of calls that belongs together) on inputs of one size.  The listed cases stand for
the ways the library is used -- blocks from a receiver searched one at a time, many short beams at once, host blocks through
the pipeline, a streaming server's blocks, the differentiable form in training, file input -- from calls that are launch
latency alone to the 4096-channel plan at full length; ``draw`` gives other sizes of the same kinds, odd ones among them,
and the search's and the dedispersion's options.

Kinds:
  search    8-bit filterbank -> dedispersed series -> single-pulse candidates in (dm_index, t) order (optionally their
            2-D peaks); "fused" takes the one-call form that never holds the series of the whole plan
  snr       single-pulse search of dedispersed series with the B(t) map (the largest SNR at every start) asked for
  batch     several uneven beams in one graph, candidates read back
  pipeline  page-locked host blocks in, candidate lists out, two blocks in flight
  approx    sub-band or tree dedispersion of every range
  train     differentiable form: the forward and both gradients, or the loss against a template and its gradients
  corner    time-major file block -> channel-major rows
"""
from __future__ import annotations

import math

import numpy as np
import torch

from paper_1912_07704_gb300 import synth
from paper_1912_07704_gb300.api import Batch, Pipeline, Plan, corner_turn
from paper_1912_07704_gb300.autograd import Dedisperse, DedispersionMSE

TSAMP = 64e-6
SKA = ",".join("%g:%g:%d:%d" % r for r in synth.SKA_4096.ranges)


def _ranges(text):
    """ "lo:step:trials:decimation,..." as the plan takes it."""
    out = []
    for part in text.split(","):
        lo, step, ndm, dec = part.split(":")
        out.append((float(lo), float(step), int(ndm), int(dec)))
    return tuple(out)


def _text(ranges):
    return ",".join("%r:%r:%d:%d" % tuple(r) for r in ranges)


def listed():
    ska = synth.SKA_4096
    plain = synth.PLAIN_256
    return [
        # a smoke-sized block: the call is launches and latency
        {"name": "tiny-64ch", "kind": "search", "nchans": 64, "fch1": 1400.0, "foff": -4.0, "nsamp": 6000,
         "ranges": "0:4:20:1,80:8:10:2", "width": 16, "opt": "none", "peaks": 0, "fused": 0},
        # the 256-channel workload: a 2 s block of a small receiver, coarse DM steps
        {"name": "plain-256ch", "kind": "search", "nchans": 256, "fch1": plain.fch1, "foff": plain.foff, "nsamp": plain.nsamp,
         "ranges": _text(plain.ranges), "width": plain.max_width, "opt": "none", "peaks": 0, "fused": 0},
        # one beam of a multi-beam receiver: 3 s, 1024 channels, fine DM steps, wide boxcars, 2-D peaks of the candidates
        {"name": "beam-1024ch", "kind": "search", "nchans": 1024, "fch1": 1508.0, "foff": -300.0 / 1024, "nsamp": 48611,
         "ranges": _text(synth.clipped_ska_ranges(250.0)), "width": 8192, "opt": "none", "peaks": 1, "fused": 0},
        # what a streaming server's slot runs per chunk on the 4096-channel plan: 2^16 new samples behind their history
        {"name": "block-4096ch-fused", "kind": "search", "nchans": 4096, "fch1": ska.fch1, "foff": ska.foff, "nsamp": (1 << 16) + 97536,
         "ranges": SKA, "width": 8192, "opt": "none", "peaks": 0, "fused": 1},
        # the benchmark's step: 67 s of 4096 channels, 4250 trials in four decimated ranges, widths 1..8192
        {"name": "ska-4096ch", "kind": "search", "nchans": 4096, "fch1": ska.fch1, "foff": ska.foff, "nsamp": ska.nsamp,
         "ranges": SKA, "width": 8192, "opt": "none", "peaks": 0, "fused": 0},
        # a search whose user wants the SNR map as well as the candidates
        {"name": "snr-map", "kind": "snr", "nchans": 256, "fch1": 1500.0, "foff": -1.171875, "nsamp": 65537,
         "ranges": "0:1:96:1", "width": 1024},
        # blocks of a few seconds from many beams, searched together
        {"name": "batch-12-short", "kind": "batch", "beams": 12, "mix": 3, "width": 8192, "threshold": 20.0},
        # host blocks through the whole path, copies and all
        {"name": "host-blocks", "kind": "pipeline", "nchans": 4096, "fch1": ska.fch1, "foff": ska.foff, "nsamp": 70001,
         "ranges": _text(synth.clipped_ska_ranges(300.0)), "width": 1024, "blocks": 2, "threshold": 10.0},
        # the tree strategy on 8 s of the 4096-channel plan
        {"name": "tree-4096ch", "kind": "approx", "nchans": 4096, "fch1": ska.fch1, "foff": ska.foff, "nsamp": 1 << 17,
         "ranges": SKA, "method": "tree"},
        # training through the forward: y and both gradients at the size the gradients are checked at
        {"name": "train-256ch", "kind": "train", "nchans": 256, "foff": -1.171875, "nsamp": 4096, "trials": 256, "step": 0.5, "loss": 0},
        # training on the loss: recomputed residuals, gradients of input and weights
        {"name": "train-1024ch-mse", "kind": "train", "nchans": 1024, "foff": -0.29296875, "nsamp": 65536, "trials": 1024, "step": 0.5, "loss": 1},
        # a file block's corner turn
        {"name": "corner-4096ch", "kind": "corner", "nchans": 4096, "nsamp": 1 << 20},
    ]


def _log_int(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def draw(rng):
    kind = rng.choice(["search", "search", "search", "snr", "batch", "pipeline", "approx", "train", "corner"])
    if kind == "corner":
        return {"kind": kind, "nchans": _log_int(rng, 64, 4096), "nsamp": _log_int(rng, 5000, 1 << 20)}
    if kind == "train":
        nchans, nsamp, step = _log_int(rng, 64, 1024), _log_int(rng, 4096, 65536), rng.choice([0.1, 0.5])
        most = int(nsamp / 2 / (16.0 * step))  # the largest delay takes half the block at most: 16 samples per unit of DM over 300 MHz
        return {"kind": kind, "nchans": nchans, "foff": -300.0 / nchans, "nsamp": nsamp, "trials": min(most, _log_int(rng, 16, 1024)),
                "step": step, "loss": rng.randint(0, 1)}
    if kind == "batch":
        return {"kind": kind, "beams": rng.randint(3, 12), "mix": rng.randint(1, 1 << 20), "width": rng.choice([512, 8192]),
                "threshold": 20.0}
    if kind == "snr":
        return {"kind": kind, "nchans": 256, "fch1": 1500.0, "foff": -1.171875, "nsamp": _log_int(rng, 8192, 65537),
                "ranges": "0:1:%d:1" % rng.randint(8, 128), "width": _log_int(rng, 16, 1024)}
    # a few configurations keep to 256 channels and coarse steps; the others are 300 MHz bands under the four-range plan
    dm_max = rng.uniform(60.0, 2000.0)
    if kind == "search" and rng.random() < 0.3:
        nchans, trials, step = _log_int(rng, 32, 300), rng.randint(16, 256), rng.choice([1.0, 2.0, 4.0])
        ranges = [(0.0, step, trials, 1)] + ([(trials * step, 2 * step, rng.randint(8, 64), rng.choice([2, 3]))] if rng.random() < 0.5 else [])
        nsamp, fch1, foff, widths = _log_int(rng, 24000, 65536), 1500.0, -300.0 / nchans, (16, 512)
        text = _text(ranges)
    else:
        nchans = rng.choice([512, 1000, 1024, 2048, 4096])
        text, fch1, foff, widths = _text(synth.clipped_ska_ranges(dm_max)), 1508.0, -300.0 / nchans, (64, 8192)
        most = {512: 1 << 18, 1000: 1 << 18, 1024: 1 << 18, 2048: 1 << 18, 4096: 1 << 18}[nchans]
        nsamp = _log_int(rng, 40000 + 8192, most)
    base = {"kind": kind, "nchans": nchans, "fch1": fch1, "foff": foff, "ranges": text}
    if kind == "approx":
        return {**base, "nsamp": min(nsamp, 1 << 17), "method": rng.choice(["tree", "sub-band"])}
    if kind == "pipeline":
        return {**base, "nsamp": min(nsamp, 70001), "width": _log_int(rng, 32, 1024), "blocks": rng.randint(1, 3), "threshold": 10.0}
    return {**base, "nsamp": nsamp, "width": _log_int(rng, *widths), "opt": rng.choice(["none", "none", "clip", "ladder", "decimated"]),
            "peaks": rng.randint(0, 1), "fused": rng.randint(0, 1)}


# ---------------------------------------------------------------- inputs --

def _workload(case, seed, nsamp=None):
    return synth.Workload("case", case["nchans"], case["fch1"], case["foff"], TSAMP, nsamp or case["nsamp"], _ranges(case["ranges"]),
                          case.get("width", 0), 6.0, int(seed))


def _delays(w):
    def of(dm):
        with Plan(w.nchans, w.fch1, w.foff, w.tsamp, [(float(dm), 0.0, 1, 1)]) as p:
            return p.shifts(0)[0]
    return of


def _filterbank(w, pitch):
    """Noise and dispersed pulses: DMs over the plan's range, widths 64 us to 16 ms (log-uniform), matched-filter SNRs of
    8 to 150, one pulse per 3.3 s but at least two and at most twenty, starting anywhere they fit."""
    rng = np.random.Generator(np.random.PCG64(w.pulse_seed))
    delays = _delays(w)
    dm_max = max(lo + (n - 1) * step for lo, step, n, _ in w.ranges)
    pulses = []
    for _ in range(max(2, min(20, w.nsamp // 52000))):
        dm = float(rng.uniform(0.02, 1.0)) * dm_max
        n_w = max(1, int(round(math.exp(rng.uniform(math.log(64e-6), math.log(16e-3))) / w.tsamp)))
        room = w.nsamp - int(delays(dm).max()) - n_w
        amplitude = rng.uniform(8.0, 150.0) * 16.0 / math.sqrt(w.nchans * n_w)
        pulses.append(synth.Pulse(dm, int(rng.uniform(0.0, 1.0) * max(0, room)), n_w, float(amplitude)))
    return synth.make_filterbank(w, pulses, delays, device="cuda", pitch=pitch)


def _options(plan, opt):
    if opt == "clip":
        plan.set_sps_clip(48, 4)
    elif opt == "ladder":
        plan.set_sps_ladder(24)
    elif opt == "decimated":
        plan.set_sps_decimated(32)


def _records(cands, ints, floats):
    """Columns of a candidate buffer: (dm_index, t, width and range) and the SNR."""
    rec = cands.view(torch.int32).view(-1, 4)
    return {ints: rec[:, :3], floats: cands.view(torch.float32).view(-1, 4)[:, 3]}


def _prepare_search(case, seed):
    w = _workload(case, seed)
    plan = Plan.from_workload(w)
    plan.bind()
    _options(plan, case["opt"])
    info = plan.query(w.nsamp, w.max_width)
    cap = max(1 << 14, min(info.dm_trial_samples // 8, 1 << 26))  # the list never overflows
    s = {"plan": plan, "nsamp": w.nsamp, "width": w.max_width, "cap": cap, "x": _filterbank(w, info.in_pitch_min),
         "count": torch.zeros(1, dtype=torch.int64, device="cuda"), "tmp": plan.postprocess_scratch(w.nsamp, w.max_width, cap)}
    for name in ("cands", "sorted") + (("peaks",) if case["peaks"] else ()):
        s[name] = torch.zeros(cap * 16, dtype=torch.uint8, device="cuda")
    s["npeaks"] = torch.zeros(1, dtype=torch.int64, device="cuda")
    if case["fused"]:
        nbytes, off = plan.fused_ws_bytes(w.nsamp, w.max_width)
        s["ws"] = plan.alloc_workspace(nbytes)
        s["ws_sps"] = s["ws"][off:]
    else:
        s["ws_dd"] = plan.alloc_workspace(info.dedisp_ws_bytes)
        s["ws_sps"] = plan.alloc_workspace(info.sps_ws_bytes)
        s["out"] = torch.zeros(info.dd_elems, dtype=torch.float32, device="cuda")
        s["views"] = plan.range_views(s["out"], w.nsamp)
    return s


def _run_search(case, s):
    plan, nsamp, width, cap = s["plan"], s["nsamp"], s["width"], s["cap"]
    out = {}
    if case["fused"]:
        plan.search_fused_device(s["x"], nsamp, width, 6.0, cap, ws=s["ws"], cands=s["cands"], count=s["count"])
    else:
        plan.dedisperse_device(s["x"], nsamp, out=s["out"], ws=s["ws_dd"])
        plan.sps_search_device(s["out"], nsamp, width, 6.0, cap, ws=s["ws_sps"], cands=s["cands"], count=s["count"])
        out["series"] = s["views"]
    plan.sps_order_device(nsamp, width, s["ws_sps"], s["cands"], s["count"], cap, out=s["sorted"], tmp=s["tmp"])
    out.update(_records(s["sorted"], "cand", "snr"), count=s["count"])
    if case["peaks"]:
        plan.peaks2d_device(nsamp, width, s["sorted"], s["count"], cap, 8, 256, out=s["peaks"], npeaks=s["npeaks"], tmp=s["tmp"])
        # the list's length is npeaks; the records behind it are not written by every call
        out["npeaks"] = s["npeaks"]
        out.update(_records(s["peaks"], "peak", "peak_snr"))
    return out


def _prepare_snr(case, seed):
    w = _workload(case, seed)
    plan = Plan.from_workload(w)
    plan.bind()
    info = plan.query(w.nsamp, w.max_width)
    cap = max(1 << 14, min(info.dm_trial_samples // 8, 1 << 26))  # the list never overflows
    dd = plan.dedisperse_device(_filterbank(w, info.in_pitch_min), w.nsamp)
    snr = torch.zeros(info.dd_elems, dtype=torch.float32, device="cuda")
    return {"plan": plan, "nsamp": w.nsamp, "width": w.max_width, "cap": cap, "dd": dd, "snr": snr, "views": plan.range_views(snr, w.nsamp),
            "ws": plan.alloc_workspace(info.sps_ws_bytes), "cands": torch.zeros(cap * 16, dtype=torch.uint8, device="cuda"),
            "count": torch.zeros(1, dtype=torch.int64, device="cuda")}


def _run_snr(case, s):
    s["plan"].sps_search_device(s["dd"], s["nsamp"], s["width"], 6.0, s["cap"], snr_out=s["snr"], ws=s["ws"], cands=s["cands"], count=s["count"])
    return {"snr": s["views"], "count": s["count"]}  # the candidate records are unordered: their number stands for them


def _beams(case):
    return synth.small_beams(case["beams"], seed=case["mix"])


def _prepare_batch(case, seed):
    beams = _beams(case)
    plans = [Plan.from_workload(w) for w in beams]
    cap = sum(p.query(w.nsamp).dm_trial_samples for p, w in zip(plans, beams)) // 100
    batch = Batch(plans, [w.nsamp for w in beams], case["width"], case["threshold"], capacity=cap)
    for i, w in enumerate(beams):
        base = {"nchans": w.nchans, "fch1": w.fch1, "foff": w.foff, "ranges": _text(w.ranges), "nsamp": w.nsamp}
        v = batch.input_view(i)
        v[:, :w.nsamp].copy_(_filterbank(_workload(base, 1000 * int(seed) + i), None))
    return {"plans": plans, "batch": batch, "store": np.zeros((cap, 4), dtype=np.int32)}


def _host_records(recs, total, store):
    """A host list is the library's: the program copies the records it keeps, at these thresholds far fewer than one in a
    thousand samples, into its own store."""
    store[:len(recs)] = recs.view(np.int32).reshape(-1, 4)
    return {"cand": store[:, :3], "snr": store.view(np.float32)[:, 3], "total": total}


def _run_batch(case, s):
    s["batch"].run()
    return _host_records(*s["batch"].candidates(), s["store"])


def _prepare_pipeline(case, seed):
    w = _workload(case, seed)
    plan = Plan.from_workload(w)
    cap = max(1 << 14, plan.query(w.nsamp).dm_trial_samples // 100)
    hosts = []
    for k in range(case["blocks"]):
        h = torch.empty((w.nchans, w.nsamp), dtype=torch.uint8, pin_memory=True)
        h.copy_(_filterbank(_workload(case, 1000 * int(seed) + k), None))
        hosts.append(h)
    return {"plan": plan, "pipeline": Pipeline(plan, w.nsamp, w.max_width, case["threshold"], capacity=cap, depth=2), "hosts": hosts,
            "stores": [np.zeros((cap, 4), dtype=np.int32) for _ in hosts]}


def _run_pipeline(case, s):
    pipe, tickets, out = s["pipeline"], [], []
    for h in s["hosts"]:
        if len(tickets) - len(out) == 2:  # as many in flight as it has slots
            out.append(_host_records(*pipe.wait(tickets[len(out)]), s["stores"][len(out)]))
        tickets.append(pipe.submit(h))
    while len(out) < len(tickets):
        out.append(_host_records(*pipe.wait(tickets[len(out)]), s["stores"][len(out)]))
    return out


def _sub_band(dec):
    """Channels per band of the sub-band strategy: as many as its 16-bit partial sums allow, 64 at most."""
    return min(64, 65535 // (255 * dec) // 8 * 8)


def _prepare_approx(case, seed):
    w = _workload(case, seed)
    plan = Plan.from_workload(w)
    for r, g in enumerate(w.ranges):
        if case["method"] == "tree":
            plan.set_fdmt(r)
        else:
            plan.set_subband(r, _sub_band(g[3]), 16)
    plan.bind()
    info = plan.query(w.nsamp)
    out = torch.zeros(info.dd_elems, dtype=torch.float32, device="cuda")
    return {"plan": plan, "nsamp": w.nsamp, "x": _filterbank(w, info.in_pitch_min), "out": out, "views": plan.range_views(out, w.nsamp),
            "ws": plan.alloc_workspace(info.dedisp_ws_bytes)}


def _run_approx(case, s):
    s["plan"].dedisperse_device(s["x"], s["nsamp"], out=s["out"], ws=s["ws"])
    return s["views"]


def _train_inputs(case, seed):
    """Float filterbank ~N(0, 1) with one pulse, positive channel weights, and the upstream gradient or the template."""
    g = torch.Generator(device="cuda")
    g.manual_seed(int(seed))
    C, T = case["nchans"], case["nsamp"]
    x = torch.randn((C, T), generator=g, device="cuda")
    shift = _table(C, 1508.0, case["foff"], 0.0, case["step"], case["trials"], 1)
    mid = shift[case["trials"] // 2]
    at = torch.from_numpy(np.minimum(T // 4 + mid[:, None] + np.arange(16), T - 1)).cuda()
    x.scatter_add_(1, at, torch.ones(at.shape, device="cuda"))
    w = torch.rand(C, generator=g, device="cuda") + 0.5
    L = max(0, T - int(shift.max()))
    return x, w, torch.randn((case["trials"], L), generator=g, device="cuda"), shift


def _prepare_train(case, seed):
    plan = Plan(case["nchans"], 1508.0, case["foff"], TSAMP, [(0.0, case["step"], case["trials"], 1)])
    plan.bind()
    x, w, t, _ = _train_inputs(case, seed)
    flat = torch.zeros(plan.query(case["nsamp"]).dd_elems, device="cuda")
    plan.range_views(flat, case["nsamp"])[0].copy_(t)
    return {"plan": plan, "x": x.requires_grad_(), "w": w.requires_grad_(), "t": flat}


def _run_train(case, s):
    if case["loss"]:
        loss = DedispersionMSE.apply(s["x"], s["w"], s["t"], s["plan"])
        gx, gw = torch.autograd.grad(loss, (s["x"], s["w"]))
        return {"loss": loss.detach(), "gx": gx, "gw": gw}
    y = Dedisperse.apply(s["x"], s["w"], s["plan"])
    gx, gw = torch.autograd.grad(y, (s["x"], s["w"]), s["t"])
    return {"y": s["plan"].range_views(y.detach(), case["nsamp"])[0], "gx": gx, "gw": gw}


def _prepare_corner(case, seed):
    g = torch.Generator(device="cuda")
    g.manual_seed(int(seed))
    return {"tm": torch.randint(0, 256, (case["nsamp"], case["nchans"]), dtype=torch.uint8, generator=g, device="cuda")}


def _run_corner(case, s):
    return corner_turn(s["tm"])


KINDS = {"search": (_prepare_search, _run_search), "snr": (_prepare_snr, _run_snr), "batch": (_prepare_batch, _run_batch),
         "pipeline": (_prepare_pipeline, _run_pipeline), "approx": (_prepare_approx, _run_approx), "train": (_prepare_train, _run_train),
         "corner": (_prepare_corner, _run_corner)}


def prepare(case, seed):
    s = KINDS[case["kind"]][0](case, seed)
    s["case"] = case
    return s


def run(state):
    return KINDS[state["case"]["kind"]][1](state["case"], state)


# ------------------------------------------------------------ what it takes --

def _shapes(nchans, fch1, foff, ranges, nsamp):
    """(trials, output length) of every range, from the delay formula at the largest DM."""
    f = np.array([fch1, fch1 + (nchans - 1) * foff])
    span = abs(f[0] ** -2 - f[1] ** -2)
    return [(n, max(0, nsamp // dec - int(round(4.148808e3 * (lo + (n - 1) * step) * span / (TSAMP * dec))))) for lo, step, n, dec in ranges]


def work(case):
    """Each input read once, each output written once; one add per channel, trial and sample of the dedispersion's definition
    (the exact strategies share partial sums and do fewer), one multiply-add for the weighted form."""
    kind = case["kind"]
    if kind == "corner":
        return {"bytes": 2.0 * case["nchans"] * case["nsamp"], "flops": 0.0}
    if kind == "train":
        (n, L), = _shapes(case["nchans"], 1508.0, case["foff"], [(0.0, case["step"], case["trials"], 1)], case["nsamp"])
        x, y = 4.0 * case["nchans"] * case["nsamp"], 4.0 * n * L
        fma = 2.0 * n * L * case["nchans"]
        # x read by the forward and the backward and its gradient written; y (or the template) once each way
        return {"bytes": 3 * x + 2 * y, "flops": 2 * fma if not case["loss"] else 3 * fma}
    beams = [case] * case.get("blocks", 1) if kind != "batch" else [
        {"nchans": w.nchans, "fch1": w.fch1, "foff": w.foff, "ranges": _text(w.ranges), "nsamp": w.nsamp} for w in _beams(case)]
    nbytes = flops = 0.0
    for b in beams:
        shapes = _shapes(b["nchans"], b["fch1"], b["foff"], _ranges(b["ranges"]), b["nsamp"])
        out = sum(n * L for n, L in shapes)
        if kind == "snr":
            nbytes += 8.0 * out
            flops += 2.0 * out * case["width"]
            continue
        nbytes += b["nchans"] * b["nsamp"] + (0 if case.get("fused") or kind in ("batch", "pipeline") else 4.0 * out)
        if kind == "approx":  # a tree's adds: one per sample and level for each row of a level of ndm rows
            flops += out * math.log2(b["nchans"])
        else:
            flops += out * b["nchans"]
    return {"bytes": nbytes, "flops": flops}


def tolerance(case):
    kind = case["kind"]
    if kind in ("corner", "approx"):
        return "exact"  # bytes moved; whole sums below 2^24
    if kind == "train":
        # sums of up to 1024 channels or trials and 65536 samples in 32 bits: 3.5e-7 off their 64-bit values
        return {"rel": 1.5e-6}
    # the series are whole sums below 2^24; SNRs are one 32-bit multiply-add of an exact sum, 4e-8 off their 64-bit values
    return {"rel": 2e-7, "differ": 0.0}


# ------------------------------------------------------- the same in 64 bits --

def _table(nchans, fch1, foff, lo, step, ndm, dec):
    """Delays [ndm][nchans] in decimated samples, from the formula."""
    f = fch1 + np.arange(nchans) * foff
    delta = f ** -2.0 - np.max(f) ** -2.0
    dm = lo + np.arange(ndm) * step
    return np.floor(4.148808e3 * dm[:, None] * delta[None, :] / (TSAMP * dec) + 0.5).astype(np.int64)


def _exact_series(x, nchans, fch1, foff, ranges):
    """y[i][t] = sum over channels of x[c][t + s(c, i)], summed in 64 bits."""
    out = []
    for lo, step, ndm, dec in ranges:
        n = x.shape[1] // dec
        xd = x[:, :n * dec].view(nchans, n, dec).to(torch.int32).sum(-1)
        shift = torch.from_numpy(_table(nchans, fch1, foff, lo, step, ndm, dec)).cuda()
        L = max(0, n - int(shift.max()))
        y = torch.zeros((ndm, L), dtype=torch.int64, device="cuda")
        for i in range(ndm):  # a window of every channel at once, in slices of time
            for a in range(0, L, 1 << 16):
                b = min(L, a + (1 << 16))
                at = shift[i][:, None] + torch.arange(a, b, device="cuda")[None, :]
                y[i, a:b] = torch.gather(xd, 1, at).sum(0)
        out.append(y.double())
    return out


def exact(case, seed):
    kind = case["kind"]
    if kind == "search":
        if case["fused"] or work(case)["flops"] > 1e11:
            return None  # no computed number but the candidates' own, or minutes of sums
        w = _workload(case, seed)
        x = _filterbank(w, None)
        return {"series": _exact_series(x, w.nchans, w.fch1, w.foff, w.ranges)}
    if kind == "snr":
        w = _workload(case, seed)
        ys = _exact_series(_filterbank(w, None), w.nchans, w.fch1, w.foff, w.ranges)
        maps = []
        for y in ys:
            mu, sigma = y.mean(1, keepdim=True), y.std(1, keepdim=True, unbiased=False)
            n, L = y.shape
            P = torch.zeros((n, L + 1), dtype=torch.float64, device="cuda")
            torch.cumsum(y, 1, out=P[:, 1:])
            best = torch.full_like(y, -math.inf)
            for k in range(1, min(case["width"], L) + 1):  # only full windows
                v = (P[:, k:] - P[:, :L + 1 - k] - k * mu) / (sigma * math.sqrt(k))
                torch.maximum(best[:, :L + 1 - k], v, out=best[:, :L + 1 - k])
            maps.append(best)
        return {"snr": maps}
    if kind == "train":
        C, T, n = case["nchans"], case["nsamp"], case["trials"]
        x, w, t, shift = _train_inputs(case, seed)
        x, w, t, shift = x.double(), w.double(), t.double(), torch.from_numpy(shift).cuda()
        L = t.shape[1]
        if not L:
            return None
        xw = x * w[:, None]
        gx = torch.zeros_like(x)  # sum over trials of the upstream gradient at u - s(c, d): scattered window by window
        y = torch.empty_like(t)
        loss = 0.0
        for d in range(n):
            at = shift[d][:, None] + torch.arange(L, device="cuda")[None, :]
            y[d] = torch.gather(xw, 1, at).sum(0)
            g = t[d]
            if case["loss"]:
                loss += float((y[d] - t[d]).square().sum())
                g = 2.0 * (y[d] - t[d]) / (n * L)
            gx.scatter_add_(1, at, g[None, :].expand(C, L))
        gw = (x * gx).sum(1)
        gx *= w[:, None]
        return {"loss": loss / (n * L), "gx": gx, "gw": gw} if case["loss"] else {"y": y, "gx": gx, "gw": gw}
    return None
