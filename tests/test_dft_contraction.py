"""The tensor-core contraction (and the direct FP32 sum) of the tone DFT on the tone counts that take it, those with a
prime factor above 7: against the definition over a tile's rows and K chunks, a closed form, a channel alone and among
others, and in a batch's finalize, direct and as a replayed step.  Bounds: those of the tone DFT tests (1e-5 of a
channel's largest phasor for FP32 sums, 2e-6 for the split operands, whose chunk sums are added in FP32), and a batch's,
1e-5 of the largest phasor and 1e-3 of the delay's sigma."""
import numpy as np
import pytest

import oracle
import synth

pytestmark = pytest.mark.gpu

MHZ = 1_000_000
BOUND = {"fp32": 1e-5, "tf32x3": 2e-6, "bf16x6": 2e-6}
# channels around a tile's 128 rows; 2N around a chunk of 32 values and a tile of 256 columns
SHAPES = [(1, 11), (127, 13), (128, 33), (129, 66), (300, 121), (64, 130), (257, 253), (130, 506), (129, 1012), (5, 1023)]


@pytest.fixture(scope="module")
def pcal():
    import torch

    from paper_2501_05993_gb300 import build as libbuild

    libbuild.build()
    import paper_2501_05993_gb300 as pkg

    pkg.load()
    torch.cuda.set_device(0)
    return pkg


def _run(pcal, mode, P):
    import torch

    C, N = P.shape
    dT = torch.full((C, N), complex(np.nan, np.nan), dtype=torch.complex64, device="cuda")
    with pcal.Dft(N, mode) as d:
        d.execute(torch.from_numpy(P.astype(np.complex64)).cuda(), C, dT)
        assert d.check() == 0
    return dT.cpu().numpy()


def _rel_err(T, ref):
    return np.max(np.abs(T - ref), axis=1) / np.max(np.abs(ref), axis=1)


@pytest.mark.parametrize("mode", list(BOUND))
@pytest.mark.parametrize("shape", SHAPES, ids=[f"C{c}-N{n}" for c, n in SHAPES])
def test_matches_definition(pcal, mode, shape):
    C, N = shape
    rng = np.random.default_rng(C * 1000 + N)
    P = (rng.standard_normal((C, N)) + 1j * rng.standard_normal((C, N))) * 10.0 ** rng.uniform(-3, 6, (C, 1))
    P += 3 * np.sqrt(N) * np.exp(2j * np.pi * rng.integers(0, N, (C, 1)) * np.arange(N) / N)
    T = _run(pcal, mode, P)
    assert _rel_err(T, np.fft.fft(P.astype(np.complex64).astype(np.complex128), axis=1)).max() <= BOUND[mode]


@pytest.mark.parametrize("mode", list(BOUND))
def test_pure_tones(pcal, mode):
    N = 253
    i0 = np.arange(20) * 13 % N
    P = np.exp(2j * np.pi * i0[:, None] * np.arange(N)[None, :] / N)
    ref = np.zeros_like(P)
    ref[np.arange(20), i0] = N
    assert _rel_err(_run(pcal, mode, P), ref).max() <= BOUND[mode]


@pytest.mark.parametrize("mode", list(BOUND))
@pytest.mark.parametrize("N", [66, 253])
def test_a_channel_alone_and_among_others(pcal, mode, N):
    rng = np.random.default_rng(N)
    P = rng.standard_normal((200, N)) + 1j * rng.standard_normal((200, N))
    T_all = _run(pcal, mode, P)
    for c in (0, 127, 128, 199):
        assert np.array_equal(_run(pcal, mode, P[c:c + 1])[0], T_all[c])


def test_workspace_grows_and_is_kept(pcal):
    """Calls of one object with more channels, then fewer: the operand tiles of the earlier ones are not read."""
    import torch

    N = 66
    rng = np.random.default_rng(7)
    with pcal.Dft(N, "tf32x3") as d:
        for C in (3, 400, 130, 3):
            P = (rng.standard_normal((C, N)) + 1j * rng.standard_normal((C, N))).astype(np.complex64)
            dT = torch.empty((C, N), dtype=torch.complex64, device="cuda")
            d.execute(torch.from_numpy(P).cuda(), C, dT)
            assert d.check() == 0
            assert _rel_err(dT.cpu().numpy(), np.fft.fft(P.astype(np.complex128), axis=1)).max() <= BOUND["tf32x3"]


@pytest.mark.parametrize("graph", [False, True], ids=["calls", "graph"])
@pytest.mark.parametrize("mode", ["tf32x3", "bf16x6"])
def test_batch(pcal, mode, graph):
    """Two channels of 66 tones, one each of 253, 11 and 1012, beside two that take the FFT."""
    import torch

    chans = [(66 * MHZ, 10_000, "i8"), (253 * MHZ, 10_000, "2bit"), (66 * MHZ, 30_000, "2bit"), (11 * MHZ, 5_000, "i8"),
             (1012 * MHZ, 10_000, "i8"), (64 * MHZ, 10_000, "2bit"), (66 * MHZ, 0, "i8"), (25 * MHZ, 20_000, "i8")]
    n = [4 * (150_000 + 37 * i) for i in range(len(chans))]
    streams = [synth.Stream(fs=fs, fc=MHZ, fo=fo, amp=0.05, td=3e-9 * (i + 1), seed=70 + i)
               for i, (fs, fo, _) in enumerate(chans)]
    hosts = [s.samples(c[2], 0, m) for s, c, m in zip(streams, chans, n)]
    dev = [torch.from_numpy(h).cuda() for h in hosts]
    with pcal.Batch([(fs, MHZ, fo, fmt) for fs, fo, fmt in chans]) as b:
        b.set_dft(mode)
        for period in range(3):  # the same buffers again: each period starts at its own index
            if graph:
                b.step_graph(dev, n)
            else:
                b.accumulate(dev, n)
                b.finalize_device()
            for c, ((fs, fo, fmt), h) in enumerate(zip(chans, hosts)):
                r = b.results(c)
                ref = oracle.tones_from_bins(oracle.bins(h, fmt, period * n[c], int(b.geometry[c].L)), fs, MHZ, fo)
                assert np.max(np.abs(r["phasors"] - ref)) <= 1e-5 * np.max(np.abs(ref)), (period, c)
                pr = oracle.products(ref, n[c], fs, MHZ, fo)
                if period == 0 and fo:  # (without an offset a tone falls on its image's place)
                    assert abs(r["td"] - pr["td"]) <= 1e-3 * pr["sigma_td"], c
