"""The two ways the batched tone DFT runs: the FFT for tone counts whose prime factors are at most 7, and the
contraction or the direct sum for the others, at the smallest counts, one of each radix, mixed radices, the longest
radix lists, the largest counts, and channel counts around a block's tile.

Tolerance (max over channels of max|T - T_ref| / max|T_ref|, FP64 reference): the FFT makes at most about 20
consecutive FP32 roundings of 2^-24 (two per level of a butterfly) or, in the tensor-core modes below 500 tones,
one per pass; both stay below 20 * 2^-24 = 1.2e-6.  The other counts keep the bounds of the existing paths."""
import numpy as np
import pytest

pytestmark = pytest.mark.gpu

MODES = ["fp32", "tf32x3", "bf16x6"]
FFT_BOUND = 20 * 2.0**-24
OTHER_BOUND = {"fp32": 1e-5, "tf32x3": 2e-6, "bf16x6": 2e-6}
SMOOTH = [(3, 2), (1, 3), (5, 4), (9, 5), (2, 7), (700, 8), (129, 27), (64, 30), (3, 49), (77, 105), (153, 343),
          (17, 512), (5, 625), (40, 729), (305, 768), (11, 1000), (1, 1024), (311, 1024)]
OTHER = [(5, 1), (130, 11), (7, 17), (129, 253), (131, 1021)]


@pytest.fixture(scope="module")
def pcal():
    import torch

    from paper_2501_05993_gb300 import build as libbuild

    libbuild.build()
    import paper_2501_05993_gb300 as pkg

    pkg.load()
    torch.cuda.set_device(0)
    return pkg


@pytest.mark.parametrize("mode", MODES)
@pytest.mark.parametrize("shape", SMOOTH + OTHER, ids=[f"C{c}-N{n}" for c, n in SMOOTH + OTHER])
def test_both_ways_match_the_definition(pcal, mode, shape):
    import torch

    C, N = shape
    rng = np.random.default_rng(C * 2000 + N)
    P = ((rng.standard_normal((C, N)) + 1j * rng.standard_normal((C, N))) * 10.0 ** rng.uniform(-3, 6, (C, 1)))
    P = P.astype(np.complex64)
    dP = torch.from_numpy(P).cuda()
    # rows beyond C stay as they are
    dT = torch.full((C + 3, N), complex(7.0, -7.0), dtype=torch.complex64, device="cuda")
    with pcal.Dft(N, mode) as d:
        d.execute(dP, C, dT)
        assert d.check() == 0
    T = dT.cpu().numpy()
    assert np.all(T[C:] == complex(7.0, -7.0))
    ref = np.fft.fft(P.astype(np.complex128), axis=1)
    err = np.max(np.abs(T[:C] - ref), axis=1) / np.max(np.abs(ref), axis=1)
    assert err.max() <= (FFT_BOUND if shape in SMOOTH else OTHER_BOUND[mode]), err.max()
