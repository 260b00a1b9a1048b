"""The ways a finalize decodes integer bins that its plan's size decides between, each on plans that do take it:
larger plans (more than 256 tones here) and batches decode in exact integer sums, from packed 2-bit words, from packed
words and the arrays they spilled into, or from the wide arrays alone (batches), and in FP64 where a bin's samples or
the level weights are beyond the integer sums (2^19 int8 or 2^26 2-bit samples a bin; weights of 1e25 and more).
Streams of billions of samples repeat one buffer of whole periods, so the oracle's counts of it add up.  Tolerance: the
library's for phasors, 1e-5 of the largest."""
import numpy as np
import pytest

import oracle

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


def _stream(fmt, n, seed):
    """n samples with a tone in them (a drifting threshold), so that no phasor is rounding alone."""
    rng = np.random.default_rng(seed)
    if fmt == "2bit":
        return rng.integers(0, 256, n // 4, dtype=np.uint8)
    return np.clip(np.round(20 * rng.standard_normal(n) + 3 * np.sin(np.arange(n))), -128, 127).astype(np.int8)


def _close(T, ref):
    assert np.max(np.abs(T - ref)) <= RTOL * np.max(np.abs(ref)), np.max(np.abs(T - ref)) / np.max(np.abs(ref))


# fs, f_offset (300 tones: L 300; 500 tones: L 50000), format, samples of a call, calls, levels
PLANS = {
    "spilled": (300 * MHZ, 0, "2bit", 4 * 16_000_200, 11, DEFAULT),        # 2.3M samples a bin: past the 21-bit fields
    "spilled-biased": (300 * MHZ, 0, "2bit", 4 * 16_000_200, 11, (-2.5, -1.0, 1.5, 3.0)),
    "i8-many": (300 * MHZ, 0, "i8", 15_000_000, 11, DEFAULT),              # 2^19 samples a bin and more: FP64
    "i8-most": (300 * MHZ, 0, "i8", 14_000_100, 11, DEFAULT),              # just below: integer sums
    "weights": (300 * MHZ, 0, "2bit", 4 * 300_300, 1, (1e26, -1e26, 2e26, 3e26)),  # FP64 over the fixed-point table
    "weights-long": (500 * MHZ, 10_000, "2bit", 4 * 300_000, 1, (1e26, -1e26, 2e26, 3e26)),
}


@pytest.mark.parametrize("name", list(PLANS))
def test_larger_plans(pcal, name):
    import torch

    fs, fo, fmt, n, calls, levels = PLANS[name]
    host = _stream(fmt, n, 21)
    dev = torch.from_numpy(host).cuda()
    with pcal.Plan(fs, MHZ, fo, fmt) as p:
        assert n % p.L == 0 and p.N > 256
        if fmt == "2bit":
            p.set_levels(levels)
        once = oracle.counts_2bit(host, 0, p.L) if fmt == "2bit" else oracle.sums_i8(host, 0, p.L)
        S = oracle.decode_counts(once * calls, levels) if fmt == "2bit" else (once * calls).astype(np.float64)
        for _ in range(2):  # the second period finds the bins cleared
            for _ in range(calls):
                p.accumulate(dev)
            assert np.array_equal(p.bins(), once * calls)
            _close(p.finalize(), oracle.tones_from_bins(S, fs, MHZ, fo))


def test_batches_beyond_the_integer_sums(pcal):
    """Both formats in one batch, below and beyond the bounds: L 16 channels of 2^19 and 2^26 samples a bin and more."""
    import torch

    chans = [(16, 4, 1, "i8"), (16, 4, 1, "2bit"), (16, 4, 1, "i8"), (300 * MHZ, MHZ, 0, "i8")]
    n = [16 * 60_000, 4 * 27_000_000, 16 * 20_000, 300 * 50_000]
    hosts = [_stream(c[3], m, 40 + i) for i, (c, m) in enumerate(zip(chans, n))]
    dev = [torch.from_numpy(h).cuda() for h in hosts]
    calls = 11  # 660,000, 74,250,000, 220,000 and 550,000 samples a bin
    with pcal.Batch(chans) as b:
        for _ in range(2):
            for _ in range(calls):
                b.accumulate(dev, n)
            b.finalize_device()
            for c, (ch, h) in enumerate(zip(chans, hosts)):
                L = int(b.geometry[c].L)
                S = oracle.decode_counts(oracle.counts_2bit(h, 0, L) * calls) if ch[3] == "2bit" else \
                    (oracle.sums_i8(h, 0, L) * calls).astype(np.float64)
                _close(b.results(c)["phasors"], oracle.tones_from_bins(S, *ch[:3]))


@pytest.mark.parametrize("N", [129, 256, 700, 1021, 1024])
@pytest.mark.parametrize("fmt", ["i8", "f32"])
def test_long_period_products_of_many_tones(pcal, fmt, N):
    """Everything a long-period plan's finalize gives for more than 128 tones, against the oracle's products of its own
    phasors: a strong comb, so that no step of the unwrapped phase is near half a turn."""
    import torch

    import synth

    fs, fo, n = N * MHZ, 10_007.25, 40_000
    host = synth.Stream(fs=fs, fc=MHZ, fo=fo, amp=0.2, td=4e-9, seed=31).samples("f32", 0, n)
    if fmt == "i8":
        host = np.round(host * (127 / np.max(np.abs(host)))).astype(np.int8)
    dev = torch.from_numpy(host).cuda()
    ref = oracle.direct_any(host, fmt, 0, fs, MHZ, fo)
    pr = oracle.products(ref, n, fs, MHZ, fo)
    with pcal.RotPlan(fs, MHZ, fo, fmt) as rp:
        rp.accumulate(dev, n)
        rp.finalize_device()
        r = rp.results()
    _close(r["phasors"], ref)
    weak = np.abs(ref) < 1e-2 * np.max(np.abs(ref))
    assert np.allclose(r["amp"], pr["amp"], rtol=0, atol=RTOL * np.max(pr["amp"]))
    # a phasor error of 1e-5 of the largest turns a tone of 1e-2 of it by 1e-3 rad
    assert np.all(np.abs(oracle.wrap(r["phase"] - pr["phase"]))[~weak] <= 1e-3)
    steps = np.abs(oracle.wrap(np.diff(pr["phase"])))
    assert not np.any(weak) and np.max(steps) < np.pi - 2e-3  # (so the unwrapped phases are comparable)
    assert np.max(np.abs(r["unwrapped"] - pr["unwrapped"])) <= 1e-3
    assert abs(r["td"] - pr["td"]) <= 1e-3 * pr["sigma_td"]
    assert abs(r["sigma_td"] - pr["sigma_td"]) <= 1e-3 * pr["sigma_td"]
    assert abs(r["td_peak"] - pr["td_peak"]) <= 1e-3 / fs
    assert np.max(np.abs(r["bandpass_phase"] - pr["bandpass_phase"])) <= 1e-3
