"""Long-period plans at the sizes where the stripe cut can go wrong: tone counts that are odd, prime or the
largest (wide blocks), streams shorter than a 16-byte word, starts and ends off 16 bytes, streams that end inside
a stripe or a stage, many blocks of stripes, and periods handed over in uneven calls, against the oracle's direct
definition.  The tolerance is the library's for phasors (an FP32 DFT of exact sums): 1e-5 of the largest phasor; a
lost or doubled sample of these streams is 1e-4 of it or more."""
import numpy as np
import pytest

import oracle
import synth

pytestmark = pytest.mark.gpu

PHASOR_RTOL = 1e-5
MHZ = 1_000_000

# fs / f_comb = N, sample counts of the calls (2-bit: multiples of 4), byte offset of each call's buffer
CASES = [
    ("i8", 16, [1], 0), ("i8", 16, [3, 40_001], 7), ("i8", 1, [9_000], 1), ("i8", 50, [20_016, 15], 0),
    ("i8", 1024, [16_384, 16_383], 9), ("i8", 1021, [30_000], 3), ("i8", 513, [16, 20_000], 15), ("i8", 7, [70_001], 0),
    ("f32", 16, [2], 4), ("f32", 16, [4_096, 30_001], 8), ("f32", 1, [9_001], 0), ("f32", 1000, [24_000], 12),
    ("f32", 1021, [30_001], 4), ("f32", 350, [5, 30_000], 0), ("f32", 1024, [20_479], 0),
    ("2bit", 16, [4], 0), ("2bit", 16, [60, 65_536], 3), ("2bit", 50, [40_004], 1), ("2bit", 1021, [40_000], 5),
    ("2bit", 1024, [65_536, 65_532], 0), ("2bit", 3, [30_000], 2),
]


@pytest.fixture(scope="module")
def pcal():
    import torch

    from paper_2501_05993_gb300 import build as libbuild

    libbuild.build()
    import paper_2501_05993_gb300 as pkg

    pkg.load()
    torch.cuda.set_device(0)
    return pkg


def _dev(host, offset):
    import torch

    raw = host.view(np.uint8)
    # what surrounds the samples must not matter
    buf = torch.full((raw.size + 64,), 0xA5, dtype=torch.uint8, device="cuda")
    buf[offset:offset + raw.size].copy_(torch.from_numpy(raw))
    return buf, buf.data_ptr() + offset


@pytest.mark.parametrize("case", CASES, ids=[f"{c[0]}-N{c[1]}-{sum(c[2])}-{c[3]}" for c in CASES])
def test_stripe_edges_match_direct_definition(pcal, case):
    fmt, N, calls, offset = case
    fs, fo = N * MHZ, 10_007.25
    s = synth.Stream(fs=fs, fc=MHZ, fo=fo, amp=0.1, td=4e-9, seed=77)
    with pcal.RotPlan(fs, MHZ, fo, fmt) as rp:
        at = 0
        for period in range(2):  # the second one starts off every boundary
            first, keep, parts = at, [], []
            for n in calls:
                host = s.samples(fmt, at, n)
                parts.append(host)
                buf, addr = _dev(host, offset)
                keep.append(buf)
                rp.accumulate(addr, n)
                at += n
            rp.finalize_device()
            T = rp.results()["phasors"]
            ref = oracle.direct_any(np.concatenate(parts), fmt, first, fs, MHZ, fo)
            err = np.max(np.abs(T - ref)) / np.max(np.abs(ref))
            assert err <= PHASOR_RTOL, (period, err)


@pytest.mark.parametrize("fmt", ["i8", "f32", "2bit"])
def test_one_call_equals_many(pcal, fmt):
    """A long call runs through many blocks of stripes per CTA; the same stream in uneven calls sums to the same
    bins (double-float sums, so equal to an FP32 DFT's rounding)."""
    fs, fo, n = 16 * MHZ, 333_333.3125, 4 * 10_000_003
    one = synth.Stream(fs=fs, fc=MHZ, fo=fo, amp=0.1, td=4e-9, seed=5).samples(fmt, 0, 4 * 1_000_003)
    host = np.tile(one, 10)
    n = host.size * (4 if fmt == "2bit" else 1)
    buf, addr = _dev(host, 0)
    esize = 4 if fmt == "f32" else 1
    out = []
    for cuts in ([0, n], [0, 4 * 999, 4 * 5_000_001, 4 * 5_000_002, n]):
        with pcal.RotPlan(fs, MHZ, fo, fmt) as rp:
            for a, b in zip(cuts, cuts[1:]):
                rp.accumulate(addr + (a // 4 if fmt == "2bit" else a * esize), b - a)
            rp.finalize_device()
            out.append(rp.results()["phasors"])
    # 16 FP32 products and sums of each P, at most 16 * 2^-23 of the largest phasor apart
    assert np.max(np.abs(out[0] - out[1])) <= 16 * 2.0**-23 * np.max(np.abs(out[0]))


def test_float_buffer_off_its_elements_is_refused(pcal):
    with pcal.RotPlan(16 * MHZ, MHZ, 10_007.0, "f32") as rp:
        with pytest.raises(pcal.PcalError) as ei:
            rp.accumulate(2, 16)  # an address that is no multiple of 4: no access is made
        assert ei.value.code == pcal.PCAL_EINVAL
