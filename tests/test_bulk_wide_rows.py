"""Tilings of the bulk fold for the widest rows (long periods with few factors of two: a row is up to 16 periods of up
to 2^20 samples).  Column groups that several CTAs share hand out their boxes through one of 8192 counters, and the
kernel's counter index is the column group: a tiling with more groups must leave every CTA its boxes statically, with
nothing left to grab.  (Host arithmetic; every plan within the limits of pcal_plan_geometry.)"""
import pytest

import paper_2501_05993_gb300 as pcal

COUNTERS = 8192

# L 1048575, 703125, 953125, 781250, 390625, 102400
PLANS = [(1048575, 1025, 1), (45e6, 1e6, 64), (61e6, 1e6, 64), (50e6, 1e6, 448), (25e6, 1e6, 64), (1024e6, 1e6, 10e3)]


@pytest.fixture(scope="module")
def lib():
    from paper_2501_05993_gb300 import build as libbuild

    libbuild.build()
    return pcal.load()


@pytest.mark.parametrize("fmt", [pcal.PCAL_2BIT, pcal.PCAL_I8, pcal.PCAL_F32])
@pytest.mark.parametrize("num_sms", [152, 148, 64, 1])
def test_no_counter_beyond_the_last(lib, fmt, num_sms):
    wide = 0
    for fs, fc, fo in PLANS:
        N = int(fs) // int(fc)
        for n_rows in (1, 2, 57, 129, 1000, 5000, 40_000, 1_000_000):
            try:
                t = pcal.pcal_bulk_tiling(fs, fc, fo, N, fmt, num_sms, n_rows)
            except pcal.PcalError:
                continue  # no tile plan: the call takes another fold
            if t.row_groups == 1:
                assert t.static_boxes == t.max_boxes == t.total_boxes  # (no grab follows)
            else:
                assert t.col_groups <= COUNTERS, (fs, fo, n_rows, t.col_groups)
            wide += t.col_groups > COUNTERS
    assert wide > 0  # the plans do reach such rows
