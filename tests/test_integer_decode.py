"""Finalizes of integer bins: the decode and rotation in exact integer sums, over every level weight they can need
(antisymmetric, biased, with a (h AND l) term), packed and spilled counts, short and long periods, few and many
tones, and periods of more samples per bin than the integer sums take (the FP64 path), against the oracle's FP64
tones of the oracle's counts.  Tolerance: the library's for phasors, 1e-5 of the largest (an FP32 DFT of the bins)."""
import numpy as np
import pytest

import oracle
import synth

pytestmark = pytest.mark.gpu

RTOL = 1e-5
MHZ = 1_000_000
DEFAULT = (-3.3359, -1.0, 1.0, 3.3359)


@pytest.fixture(scope="module")
def pcal():
    import torch

    from paper_2501_05993_gb300 import build as libbuild

    libbuild.build()
    import paper_2501_05993_gb300 as pkg

    pkg.load()
    torch.cuda.set_device(0)
    return pkg


def _check(pcal, fs, fc, fo, fmt, host, levels=DEFAULT, repeat=1, periods=2):
    import torch

    dev = torch.from_numpy(host).cuda()
    n1 = host.size * (4 if fmt == "2bit" else 1)
    with pcal.Plan(fs, fc, fo, fmt) as plan:
        if fmt == "2bit":
            plan.set_levels(levels)
        at = 0
        for _ in range(periods):  # the second period starts off the bins' origin
            count = 0
            for _ in range(repeat):
                plan.accumulate(dev)
                c = oracle.counts_2bit(host, at % plan.L, plan.L) if fmt == "2bit" else \
                    oracle.sums_i8(host, at % plan.L, plan.L)
                count = count + c
                at += n1
            assert np.array_equal(plan.bins(), count)
            T = plan.finalize()
            S = oracle.decode_counts(count, levels) if fmt == "2bit" else count.astype(np.float64)
            ref = oracle.tones_from_bins(S, fs, fc, fo)
            assert np.max(np.abs(T - ref)) <= RTOL * np.max(np.abs(ref))


@pytest.mark.parametrize("levels", [DEFAULT, (-2.5, -1.0, 1.0, 3.0), (0.0, 1.0, 2.0, 3.0), (1e-3, 0.0, 0.0, -7.25),
                                    (1e26, -1e26, 2e26, 3e26)],
                         ids=["antisymmetric", "biased", "linear", "and-term", "beyond-floats"])
@pytest.mark.parametrize("geom", [(64 * MHZ, MHZ, 10_000), (16, 4, 1), (256 * MHZ, MHZ, 7_000),
                                  (500 * MHZ, MHZ, 10_000)], ids=["L6400", "L16", "L256000", "N500"])
def test_2bit_levels(pcal, geom, levels):
    if levels[0] == 1e26 and geom[1] != 4:
        pytest.skip("one period is enough for the path itself")
    fs, fc, fo = geom
    host = synth.Stream(fs=fs, fc=fc, fo=fo, amp=0.05, td=0.0, seed=3).bits2(0, 4 * 300_007)
    _check(pcal, fs, fc, fo, "2bit", host, levels)


@pytest.mark.parametrize("geom", [(16, 4, 1), (128 * MHZ, MHZ, 30_000), (256 * MHZ, MHZ, 1_000), (MHZ, MHZ, 3),
                                  (272 * MHZ, MHZ, 10_000), (1000 * MHZ, MHZ, 10_000), (1024 * MHZ, MHZ, 10_000)],
                         ids=["N4", "N128", "L256000", "N1-L1000000", "N272", "N1000", "N1024"])
def test_i8_geometries(pcal, geom):
    fs, fc, fo = geom
    host = synth.Stream(fs=fs, fc=fc, fo=fo, amp=0.05, td=0.0, seed=4).i8(0, 2_100_003)
    _check(pcal, fs, fc, fo, "i8", host)


def test_many_samples_per_bin(pcal):
    """Packed counts that spilled (2^21 per bin), and counts beyond the integer sums' bounds (2^26 2-bit, 2^19 int8)."""
    s = synth.Stream(fs=16, fc=4, fo=1, amp=0.05, td=0.0, seed=5)
    _check(pcal, 16, 4, 1, "2bit", s.bits2(0, 4 * 4_000_000), repeat=3, periods=1)
    _check(pcal, 16, 4, 1, "2bit", np.tile(s.bits2(0, 4 * 4_000_000), 68), periods=1)
    _check(pcal, 16, 4, 1, "i8", np.tile(s.i8(0, 3_000_000), 3), periods=1)
