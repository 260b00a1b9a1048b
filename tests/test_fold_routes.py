"""Which fold takes a call (Plan.fold_counts, Batch.fold_counts), on both sides of the lines between them, and the
bulk fold of long float32 periods, whose partial sums go through four slots and a reduction with one thread per bin."""
import numpy as np
import pytest

import oracle
import synth

pytestmark = pytest.mark.gpu
MHZ = 1_000_000


@pytest.fixture(scope="module")
def pcal():
    import torch

    from paper_2501_05993_gb300 import build as libbuild

    libbuild.build()
    import paper_2501_05993_gb300 as pkg

    pkg.load()
    torch.cuda.set_device(0)
    return pkg


def counts(**kw):
    return dict({"bulk": 0, "short_folds": 0, "ragged": 0, "persistent": 0, "direct": 0}, **kw)


# fmt, fs, f_offset, samples, byte offset, folds
ROUTES = [
    ("i8", 16, 1, 8_191, 0, counts(ragged=1)),                           # under 8 KB (L 16)
    ("i8", 16, 1, 8_192, 0, counts(short_folds=1)),
    ("2bit", 64 * MHZ, 10_000, 640_000, 3, counts(short_folds=1)),       # 10 ms
    ("f32", 16 * MHZ, 10_000, 160_000, 4, counts(short_folds=1)),
    ("i8", 64 * MHZ, 10_000, 245_760, 1, counts(ragged=1)),              # short calls and few samples a bin
    ("i8", 64 * MHZ, 10_000, 245_761, 1, counts(short_folds=1)),
    ("i8", 16 * MHZ, 10_000, 128 * 1_600, 0, counts(ragged=1)),
    ("i8", 16 * MHZ, 10_000, 128 * 1_600 + 1, 0, counts(short_folds=1)),
    ("2bit", 64 * MHZ, 10_000, 4 * 40_960, 0, counts(ragged=1)),
    ("2bit", 64 * MHZ, 10_000, 4 * 40_961, 0, counts(short_folds=1)),
    ("2bit", 16 * MHZ, 10_000, 48 * 1_600, 5, counts(ragged=1)),
    ("2bit", 16 * MHZ, 10_000, 48 * 1_600 + 4, 5, counts(short_folds=1)),
    ("f32", 64 * MHZ, 10_000, 4 * 6_400, 4, counts(ragged=1)),           # up to four periods
    ("f32", 64 * MHZ, 10_000, 4 * 6_400 + 1, 4, counts(short_folds=1)),
    ("f32", 256 * MHZ, 7_000, 4 * 256_000, 0, counts(ragged=1)),
    ("f32", 256 * MHZ, 7_000, 4 * 256_000 + 1, 0, counts(short_folds=1)),
    ("f32", 1024 * MHZ, 1_000, 40_000, 0, counts(short_folds=1)),        # (not of the longest)
    ("f32", 16, 1, 64, 0, counts(ragged=1)),
    ("f32", 16, 1, 65, 0, counts(short_folds=1)),
    ("i8", 1024 * MHZ, 1_000, 3 * 1_024_000 - 1, 0, counts(ragged=1)),   # fewer than three whole rows
    ("i8", 1024 * MHZ, 1_000, 3 * 1_024_000, 0, counts(short_folds=1)),
    ("2bit", 1024 * MHZ, 1_000, 4 * 767_999, 0, counts(ragged=1)),
    ("2bit", 1024 * MHZ, 1_000, 4 * 768_000, 0, counts(short_folds=1)),
    ("2bit", 25 * MHZ, 64, 4 * 1_000_000, 2, counts(ragged=1)),          # (rows of 6.25 MB)
    ("i8", 25 * MHZ, 64, 6_249_999, 0, counts(ragged=1)),                # none, however long
    ("i8", 25 * MHZ, 64, 6_250_000, 0, counts(short_folds=1)),
    ("2bit", 64 * MHZ, 10_000, 4 * 1_100_000, 1, counts(bulk=1)),        # 1 MB of rows, edges inside
    ("i8", 64 * MHZ, 10_000, 1_100_000, 0, counts(bulk=1)),
    ("f32", 64 * MHZ, 10_000, 245 * 6_400, 0, counts(short_folds=1)),
    ("f32", 64 * MHZ, 10_000, 257 * 6_400 + 1, 0, counts(bulk=1, ragged=1)),
    ("f32", 256 * MHZ, 10_000, 61 * 25_600, 0, counts(short_folds=1)),   # up to 6 MB where the rows fit the SMs
    ("f32", 256 * MHZ, 10_000, 62 * 25_600, 0, counts(bulk=1)),
    ("f32", 64 * MHZ, 10_000, 246 * 6_400, 0, counts(bulk=1)),
    ("f32", 256 * MHZ, 7_000, 256 * 256_000, 0, counts(short_folds=1)),  # at most 256 periods of wider rows
    ("f32", 256 * MHZ, 7_000, 257 * 256_000, 0, counts(bulk=1)),
    ("2bit", 1024 * MHZ, 7_000, 4 * 18 * 256_000, 0, counts(bulk=1)),    # wide 2-bit rows all the same
    ("2bit", 45 * MHZ, 64, 4 * 2 * 11_250_000, 0, counts(bulk=1)),       # (10,987 column groups)
    ("i8", 256 * MHZ, 7_000, 128 * 256_000, 0, counts(short_folds=1)),   # at most 128 wide rows
    ("i8", 256 * MHZ, 7_000, 129 * 256_000, 0, counts(bulk=1)),
]


@pytest.mark.parametrize("route", ROUTES, ids=[f"{r[0]}-fs{r[1]}-{r[2]}-{r[3]}" for r in ROUTES])
def test_fold_of_a_call(pcal, route):
    import torch

    fmt, fs, fo, n, offset, expect = route
    nbytes = {"2bit": n // 4, "i8": n, "f32": 4 * n}[fmt]
    gen = torch.Generator(device="cuda").manual_seed(n)
    if fmt == "f32":
        buf = torch.randn(n + 8, generator=gen, device="cuda").view(torch.uint8)
    else:
        buf = torch.randint(0, 256, (nbytes + 32,), dtype=torch.uint8, generator=gen, device="cuda")
    with pcal.Plan(fs, MHZ if fs > 16 else 4, fo, fmt) as p:
        p.accumulate(buf.data_ptr() + offset, n)
        assert p.fold_counts() == expect
        bins = p.bins()
        host = buf[offset:offset + nbytes].cpu().numpy()
        if fmt == "2bit":
            assert np.array_equal(bins, oracle.counts_2bit(host, 0, p.L))
        elif fmt == "i8":
            assert np.array_equal(bins, oracle.sums_i8(host.view(np.int8), 0, p.L))
        else:
            x = host.view(np.float32)
            # compensated FP32 sums of at most 257 samples a bin: 257^2 * 2^-48 < 2^-31 of their magnitudes
            mag = oracle.fold_real(np.abs(x), "f32", 0, p.L)
            assert np.all(np.abs(bins - oracle.sums_f32(x, 0, p.L)) <= 2.0**-31 * mag)


# fmt, fs, f_offset (L 390625, 140625 and 703125: rows of 6.25, 2.25 and 11.25 MB), samples, fold, its ragged edges
LARGE = [
    ("i8", 25 * MHZ, 64, 300_000_007, "short_folds", 0),   # 256 MB and more of few wide rows
    ("i8", 1125 * MHZ, 8_000, 270_000_000, "short_folds", 0),
    ("i8", 25 * MHZ, 64, 130 * 6_250_000, "bulk", 2),      # (13 bytes before, most of a row behind)
    ("i8", 45 * MHZ, 64, 130 * 11_250_000, "bulk", 2),     # 10,987 column groups
    ("f32", 45 * MHZ, 64, 257 * 703_125, "bulk", 1),
    ("f32", 45 * MHZ, 64, 256 * 703_125, "short_folds", 0),
]


@pytest.mark.parametrize("case", LARGE, ids=[f"{c[0]}-{c[3]}" for c in LARGE])
def test_large_calls_of_wide_rows(pcal, case):
    import torch

    fmt, fs, fo, n, fold, ragged = case
    gen = torch.Generator(device="cuda").manual_seed(n)
    if fmt == "i8":
        x = torch.randint(-128, 128, (n + 3,), dtype=torch.int8, generator=gen, device="cuda")[3:]
    else:
        x = torch.randn(n, generator=gen, device="cuda")
    with pcal.Plan(fs, MHZ, fo, fmt) as p:
        p.accumulate(x.data_ptr(), n)
        f = p.fold_counts()
        assert f[fold] == 1 and f["bulk"] + f["short_folds"] == 1, f
        assert f["ragged"] == ragged, f
        bins, L = torch.from_numpy(p.bins()).cuda(), p.L

    def fold_of(v, dtype):
        s = torch.zeros(L, dtype=dtype, device="cuda")
        for at in range(0, n // L * L, 32 * L):
            s += v[at:min(at + 32 * L, n // L * L)].view(-1, L).sum(0, dtype=dtype)
        s[:n % L] += v[n // L * L:].to(dtype)
        return s

    if fmt == "i8":
        assert torch.equal(bins, fold_of(x, torch.int64))
    else:
        # compensated FP32 sums of at most 257 samples a bin: 257^2 * 2^-48 < 2^-31 of their magnitudes
        assert bool(torch.all((bins - fold_of(x, torch.float64)).abs() <= 2.0**-31 * fold_of(x.abs(), torch.float64)))


@pytest.mark.parametrize("geom", [(64 * MHZ, 10_000), (256 * MHZ, 10_000), (1024 * MHZ, 10_000), (256 * MHZ, 1_000)],
                         ids=["L6400", "L25600", "L102400", "L256000"])
def test_bulk_float32_of_long_periods(pcal, geom):
    """Six bulk folds of 257 periods and a few samples each: the slots fill, are reduced, and fill again; then the
    bins (a reduction of what is pending), and the same once more through the finalize."""
    import torch

    fs, fo = geom
    with pcal.Plan(fs, MHZ, fo, "f32") as p:
        L, calls = p.L, 6
        n = 257 * L + 37
        x = np.random.default_rng(L).standard_normal(n).astype(np.float32)
        dev = torch.from_numpy(x).cuda()
        for _ in range(calls):
            p.accumulate(dev)
        f = p.fold_counts()
        assert f["bulk"] == calls and f["short_folds"] == 0, f
        bins = p.bins()
        ref, mag = np.zeros(L), np.zeros(L)
        once, once_mag = oracle.sums_f32(x, 0, L), oracle.fold_real(np.abs(x), "f32", 0, L)
        for c in range(2 * calls):  # (a call's bins start at its first sample's)
            if c == calls:
                # compensated FP32 sums of at most 258 samples a bin and call (258^2 * 2^-48 < 2^-31 of their
                # magnitudes), added in double-float
                assert np.all(np.abs(bins - ref) <= 2.0**-31 * mag)
                p.finalize_device()
                for _ in range(calls):
                    p.accumulate(dev)
                ref, mag = np.zeros(L), np.zeros(L)
            ref += np.roll(once, c * n % L)
            mag += np.roll(once_mag, c * n % L)
        T = p.finalize()
        want = oracle.tones_from_bins(ref, fs, MHZ, fo)
        assert np.max(np.abs(T - want)) <= 1e-5 * np.max(np.abs(want))  # the library's bound for phasors


# fs, f_offset, bulk folds before the finalize (0: one short fold), kernels of the finalize
FINALIZES = [
    (128 * MHZ, 10_000, 1, 1),   # L 12800: one fold's partials are added by the finalize,
    (128 * MHZ, 10_000, 2, 2),   # more by a reduction before it
    (48 * MHZ, 10_000, 3, 1),    # (not for short periods)
    (64 * MHZ, 1_000, 2, 1),     # L 64000: the finalize of all SMs adds them
    (300 * MHZ, 10_000, 1, 1),   # L 30000, 300 tones: one cluster
    (300 * MHZ, 10_000, 3, 2),
    (512 * MHZ, 10_000, 0, 1),   # L 51200, 512 tones: one cluster where no partials wait,
    (512 * MHZ, 10_000, 1, 2),   # else two kernels on all SMs
    (512 * MHZ, 5_000, 0, 1),    # L 102400
    (512 * MHZ, 1_000, 0, 2),    # L 512000
]


@pytest.mark.parametrize("case", FINALIZES, ids=[f"L{c[0] // np.gcd(MHZ, c[1])}-{c[2]}" for c in FINALIZES])
def test_float32_finalizes(pcal, case):
    """The finalize that a float32 period takes, and its phasors (the library's bound, 1e-5 of the largest), twice."""
    import torch

    fs, fo, folds, kernels = case
    with pcal.Plan(fs, MHZ, fo, "f32") as p:
        L = p.L
        n = 257 * L + 3 * L // 7 if folds else 5 * L // 2
        gen = torch.Generator(device="cuda").manual_seed(L)
        x = torch.randn(n, generator=gen, device="cuda")
        once = torch.zeros(L, dtype=torch.float64, device="cuda")
        once += x[:n // L * L].view(-1, L).sum(0, dtype=torch.float64)
        once[:n % L] += x[n // L * L:]
        once = once.cpu().numpy()
        at = 0
        for _ in range(2):
            S = np.zeros(L)
            for _ in range(max(folds, 1)):
                p.accumulate(x)
                S += np.roll(once, at % L)
                at += n
            assert (p.fold_counts()["bulk"] > 0) == (folds > 0)
            before = p.stats()["kernel_launches"]
            T = p.finalize()
            assert p.stats()["kernel_launches"] - before == kernels
            ref = oracle.tones_from_bins(S, fs, MHZ, fo)
            assert np.max(np.abs(T - ref)) <= 1e-5 * np.max(np.abs(ref))


def test_fold_of_a_batch(pcal):
    import torch

    chans = [(64 * MHZ, MHZ, 10_000, "2bit"), (32 * MHZ, MHZ, 30_000, "i8")]
    n = [4 * 300_000, 500_001]
    xs = [torch.randint(0, 256, (300_000,), dtype=torch.uint8, device="cuda"),
          torch.randint(-128, 128, (500_001,), dtype=torch.int8, device="cuda")]
    with pcal.Batch(chans) as b:
        b.accumulate(xs, n)
        assert b.fold_counts() == counts(direct=1)
        b.finalize_device()
        for _ in range(3):
            b.step_graph(xs, n)
        assert b.fold_counts() == counts(direct=4)
        want = [b.results(c)["phasors"] for c in range(2)]
        b.set_schedule(min_chunk=4)
        b.accumulate(xs, n)
        assert b.fold_counts() == counts(direct=4, persistent=1)
        assert all(np.all(np.isfinite(w)) for w in want)
    with pcal.Batch(chans) as b:
        b.accumulate(xs, [0, 0])  # no samples: no fold
        b.step_graph(xs, [0, 0])
        assert b.fold_counts() == counts()


def test_captured_steps_follow_the_schedule(pcal):
    """A step that was captured before its batch's schedule changed is captured again: it runs the new fold, with the
    same exact bins and so the same phasors."""
    import torch

    chans = [(64 * MHZ, MHZ, 10_000, "2bit"), (32 * MHZ, MHZ, 30_000, "i8")]
    n = [64 * 80_000, 32 * 20_000]  # whole periods: every step's phasors are the first one's
    xs = [torch.randint(0, 256, (n[0] // 4,), dtype=torch.uint8, device="cuda"),
          torch.randint(-128, 128, (n[1],), dtype=torch.int8, device="cuda")]
    with pcal.Batch(chans) as b:
        def step():
            before = b.fold_counts()
            b.step_graph(xs, n)
            torch.cuda.synchronize()
            now = b.fold_counts()
            got = [b.results(c)["phasors"] for c in range(2)]
            return {k for k in now if now[k] != before[k]}, got

        kind, want = step()
        assert kind == {"direct"}
        for kw in (dict(min_chunk=4), dict(box_rows=64), dict(box_rows=64)):
            b.set_schedule(**kw)
            kind, got = step()
            assert kind == {"persistent"}
            assert all(np.array_equal(x, y) for x, y in zip(got, want))
        b.autotune(xs, n)
        kind, got = step()
        b.accumulate(xs, n)  # the fold of an uncaptured call is the one that autotune kept
        last = b.fold_counts()
        b.accumulate(xs, n)
        now = b.fold_counts()
        assert kind == {k for k in now if now[k] != last[k]}
        assert all(np.array_equal(x, y) for x, y in zip(got, want))


def test_the_fold_that_runs_is_the_one_reported(pcal):
    import torch

    chans = [(64 * MHZ, MHZ, 10_000, "2bit"), (32 * MHZ, MHZ, 30_000, "i8")]
    n = [64 * 80_000, 32 * 20_000]
    xs = [torch.randint(0, 256, (n[0] // 4,), dtype=torch.uint8, device="cuda"),
          torch.randint(-128, 128, (n[1],), dtype=torch.int8, device="cuda")]
    with pcal.Batch(chans) as b:
        def runs():
            before = b.fold_counts()
            b.step_graph(xs, n)
            b.accumulate(xs, n)
            now = b.fold_counts()
            b.finalize_device()
            return {k: now[k] - before[k] for k in now if now[k] != before[k]}

        kernel = {"direct": "direct", "schedule": "persistent"}
        assert b.fold == "direct"
        assert runs() == {"direct": 2}
        for change in (lambda: b.autotune(xs, n), lambda: b.set_schedule(min_chunk=8), lambda: b.set_fold("direct"),
                       lambda: b.set_fold("schedule"), lambda: b.autotune(xs, n)):
            change()
            assert runs() == {kernel[b.fold]: 2}
        b.set_schedule(min_chunk=8)
        assert b.fold == "schedule"
        b.set_fold("direct")
        assert b.fold == "direct" and b.schedule["min_chunk"] == 8
        with pytest.raises(ValueError):
            b.set_fold("fast")
        assert pcal.load().pcal_batch_set_fold(b.handle, 2) == pcal.PCAL_EINVAL
