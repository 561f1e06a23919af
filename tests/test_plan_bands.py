"""Band rows of the grouped strategy, host side (no GPU): the delays that the
tables add up to, read back entry by entry as the kernels read them
(aa_plan_effective_shifts), are the brute-force delays."""
import numpy as np
import pytest

from paper_1912_07704_gb300 import abi, synth
from paper_1912_07704_gb300.api import Plan

PLANS = {
    "ska": (4096, 1508.0, -300.0 / 4096, synth.SKA_4096.ranges),
    "1024ch-dec16": (1024, 1508.0, -300.0 / 1024, synth.clipped_ska_ranges(2300.0)),
    "512ch": (512, 1508.0, -300.0 / 512, synth.clipped_ska_ranges(400.0)),
    # a last band of 1, 4, 5 and 7 channels; one, two and a part of a segment; 64 k + 1 trials
    "ragged-1001": (1001, 1508.0, -0.3, ((0.0, 0.1, 65, 1), (7.0, 0.1, 513, 3))),
    "ragged-1004": (1004, 1508.0, -0.3, ((3.0, 0.2, 64, 2),)),
    "ragged-1005": (1005, 1508.0, -0.3, ((0.0, 0.05, 1025, 1),)),
    "ragged-1007": (1007, 1508.0, -0.3, ((0.0, 0.0, 70, 1), (50.0, 0.3, 200, 16))),
    # rising band: delays fall with the channel index
    "rising": (800, 1208.0, 0.375, ((0.0, 0.1, 300, 1), (30.0, 0.4, 150, 5))),
}


# nchans, DM step, trials, samples, band rows faster (measured, us with / without)
SIDES = [
    (1024, 1.0, 1600, 300, False),   # 540 / 160
    (1024, 1.0, 1600, 16000, True),
    (256, 0.3, 1600, 300, False),    # 98 / 39
    (256, 1.0, 700, 1000, False),    # 85 / 45
    (64, 0.3, 64, 4000, False),      # 18 / 14
    (64, 0.1, 1500, 64000, True),
    (4096, 0.1, 1500, 16000, True),
]


@pytest.mark.parametrize("C, step, ndm, length, bands", SIDES)
def test_row_buffer_is_asked_for_where_band_rows_are_faster(C, step, ndm, length, bands):
    p = Plan(C, 1508.0, -300.0 / C, 64e-6, [(0.0, step, ndm, 1)])
    n = length + int(p.shifts(0).max())
    least = abi.aa_dedisperse_least_ws_bytes(p.handle, n)
    assert (p.query(n).dedisp_ws_bytes > least) == bands
    try:
        abi.aa_debug_inject(4, 1)
        assert p.query(n).dedisp_ws_bytes > least
    finally:
        abi.aa_debug_inject(0, 0)
    p.set_strategy(0, abi.AA_DEDISP_DIRECT)
    assert p.query(n).dedisp_ws_bytes == least
    with pytest.raises(abi.AAError, match="AA_ERR_ARG"):
        abi.aa_debug_inject(4, 2)


@pytest.fixture
def wherever_they_fit():
    abi.aa_debug_inject(4, 1)
    yield
    abi.aa_debug_inject(0, 0)


@pytest.mark.parametrize("name", PLANS)
def test_band_tables_add_up_to_the_delays(name, wherever_they_fit):
    C, fch1, foff, ranges = PLANS[name]
    p = Plan(C, fch1, foff, 64e-6, ranges)
    banded = 0
    for r, g in enumerate(ranges):
        abi.aa_plan_set_strategy(p.handle, r, abi.AA_DEDISP_GROUPED)
        assert np.array_equal(abi.aa_plan_effective_shifts(p.handle, r, g[2], C), p.shifts(r))
        p.set_strategy(r, abi.AA_DEDISP_DIRECT)
    base = p.query(1 << 17).dedisp_ws_bytes
    for r in range(len(ranges)):
        p.set_strategy(r, abi.AA_DEDISP_GROUPED)
        banded += p.query(1 << 17).dedisp_ws_bytes > base
        p.set_strategy(r, abi.AA_DEDISP_DIRECT)
    assert banded == len(ranges)  # every range here has band rows
