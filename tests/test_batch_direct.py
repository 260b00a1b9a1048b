"""The fold of a batch without a schedule (small CTAs on column blocks of row blocks) at the sizes where its cut can
go wrong: rows narrower than a block and not a multiple of one, one row and none, row counts around a warp's batch
and a task's chunk, periods shorter than a block's bins, starts off 16 bytes, ends inside a row and inside a 16-byte
word.  The bins are exact integers, so they equal the oracle's, and the persistent fold's, exactly."""
import numpy as np
import pytest

import oracle
import synth

pytestmark = pytest.mark.gpu

# fs, f_comb, f_offset, format, samples, byte offset of the buffer
CHANNELS = [
    (16, 4, 1, "i8", 256 * 40_000 + 77, 3),            # L 16, 64-word rows, several chunks of rows
    (16, 4, 1, "2bit", 4 * (256 * 33_000 + 9), 1),     # L 16, more rows than one task takes
    (32_000_000, 1_000_000, 0, "2bit", 4 * 256 * 32, 0),           # 64-word rows, 32 of them
    (32_000_000, 1_000_000, 0, "i8", 256 * 8 + 16, 0),             # 8 rows and one 16-byte word
    (20_000_000, 1_000_000, 10_000, "i8", 2000 * 65, 15),          # 500-word rows
    (20_000_000, 1_000_000, 10_000, "2bit", 2000 * 4 * 129 + 4, 2),
    (7_000_000, 1_000_000, 10_000, "i8", 2800 * 5 - 1, 0),         # rows of 2800 samples, the last one short
    (7_000_000, 1_000_000, 10_000, "2bit", 4 * 7, 5),              # under 16 bytes
    (64_000_000, 1_000_000, 30_000, "i8", 6_399, 4),               # under one row
    (64_000_000, 1_000_000, 30_000, "2bit", 640_000, 0),
    (50_000_000, 1_000_000, 130_000, "i8", 500_001, 9),
    (1_024_000_000, 1_000_000, 10_000, "2bit", 10_240_000, 0),
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
    buf = torch.full((raw.size + 64,), 0x5A, dtype=torch.uint8, device="cuda")  # (the surroundings must not count)
    buf[offset:offset + raw.size].copy_(torch.from_numpy(raw))
    return buf, buf.data_ptr() + offset


def test_direct_fold_bins_are_exact(pcal):
    hosts = [synth.Stream(fs=c[0], fc=c[1], fo=c[2], amp=0.02, td=0.0, seed=60 + i).samples(c[3], 0, c[4])
             for i, c in enumerate(CHANNELS)]
    dev = [_dev(h, c[5]) for h, c in zip(hosts, CHANNELS)]
    n = [c[4] for c in CHANNELS]
    with pcal.Batch([c[:4] for c in CHANNELS]) as b, pcal.Batch([c[:4] for c in CHANNELS]) as p:
        p.set_schedule(min_chunk=4)  # any schedule: the persistent fold
        for _ in range(2):  # the second call starts at every channel's own index
            for x in (b, p):
                x.accumulate([a for _, a in dev], n)
        for c, (ch, h) in enumerate(zip(CHANNELS, hosts)):
            L = int(b.geometry[c].L)
            count = oracle.counts_2bit if ch[3] == "2bit" else oracle.sums_i8
            ref = count(h, 0, L) + count(h, ch[4], L)
            bins = b.bins(c)
            assert np.array_equal(bins, ref), (c, np.argwhere(bins != ref)[:4].tolist())
            assert np.array_equal(bins, p.bins(c))


def test_finalize_order_of_many_channels(pcal):
    """45 channels whose clusters cannot all run at once, the shortest finalizes first in channel order (the launch
    starts the longest first): every channel gets its own results, twice.  Bound: the phasor bound of the other
    paths, 1e-5 of the largest."""
    chans = [(fs, 1_000_000, 10_000 * (1 + i % 3), "i8" if i % 2 else "2bit")
             for fs in (16_000_000, 64_000_000, 1_024_000_000) for i in range(15)]
    n = [400_000 + 4 * i for i in range(len(chans))]
    hosts = [synth.Stream(fs=c[0], fc=c[1], fo=c[2], amp=0.05, td=1e-9, seed=90 + i).samples(c[3], 0, n[i])
             for i, c in enumerate(chans)]
    dev = [_dev(h, 0) for h in hosts]
    with pcal.Batch(chans) as b:
        plans = [pcal.Plan(*c[:3], fmt=c[3]) for c in chans]
        for _ in range(2):
            b.accumulate([a for _, a in dev], n)
            b.finalize_device()
            for i, p in enumerate(plans):
                pcal.pcal_accumulate(p.handle, dev[i][1], n[i], 0)
                T = p.finalize()
                got = b.results(i)["phasors"]
                assert np.max(np.abs(got - T)) <= 1e-5 * np.max(np.abs(T)), i
        for p in plans:
            p.close()
