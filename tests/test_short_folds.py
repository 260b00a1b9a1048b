"""Single calls too short for the bulk fold: every format around the sizes where the cut changes (a few KB, one row,
a warp's batch and a chunk of rows, just below the bulk kernel), short and long periods, starts and ends off 16-byte
words and rows.  Integer bins equal the oracle's exactly; float32 bins are double-float sums: an addition errs by at
most 2^-46 of the partial sum, so n of them by n * 2^-46 * sum|x| / n per bin at worst."""
import numpy as np
import pytest

import oracle
import synth

pytestmark = pytest.mark.gpu
MHZ = 1_000_000

GEOMS = [(64 * MHZ, MHZ, 10_000), (16, 4, 1), (16 * MHZ, MHZ, 0), (20 * MHZ, MHZ, 130_000), (7 * MHZ, MHZ, 10_000),
         (256 * MHZ, MHZ, 7_000)]  # L 6400, 16, 16, 2000, 700, 256000
BYTES = [8_191, 8_192, 8_200, 25_600, 102_417, 160_000, 409_601, 1_048_575, 1_048_576 + 300]


@pytest.fixture(scope="module")
def pcal():
    import torch

    from paper_2501_05993_gb300 import build as libbuild

    libbuild.build()
    import paper_2501_05993_gb300 as pkg

    pkg.load()
    torch.cuda.set_device(0)
    return pkg


@pytest.mark.parametrize("geom", GEOMS, ids=[f"L{g[0] // np.gcd.reduce(g)}" for g in GEOMS])
@pytest.mark.parametrize("fmt", ["2bit", "i8", "f32"])
def test_short_folds(pcal, geom, fmt):
    import torch

    fs, fc, fo = geom
    s = synth.Stream(fs=fs, fc=fc, fo=fo, amp=0.05, td=0.0, seed=8)
    per = {"2bit": 4, "i8": 1, "f32": 0.25}[fmt]
    for i, nbytes in enumerate(BYTES):
        n = int(nbytes * per)
        host = s.samples(fmt, 0, n)
        raw = host.view(np.uint8)
        off = (0, 4, 8, 12)[i % 4] if fmt == "f32" else (0, 1, 15, 6)[i % 4]
        buf = torch.full((raw.size + 64,), 0x6D, dtype=torch.uint8, device="cuda")  # the surroundings must not count
        buf[off:off + raw.size].copy_(torch.from_numpy(raw))
        with pcal.Plan(fs, fc, fo, fmt) as plan:
            for _ in range(3):  # the later calls start inside a period
                plan.accumulate(buf.data_ptr() + off, n)
            got = plan.bins()
            L = plan.L
        if fmt == "f32":
            ref = sum(oracle.sums_f32(host, k * n, L) for k in range(3))
            bound = 3 * np.sum(np.abs(host.astype(np.float64))) * 2.0**-46
            assert np.max(np.abs(got - ref)) <= bound, (nbytes, np.max(np.abs(got - ref)), bound)
        else:
            count = oracle.counts_2bit if fmt == "2bit" else oracle.sums_i8
            ref = sum(count(host, k * n, L) for k in range(3))
            assert np.array_equal(got, ref), nbytes
