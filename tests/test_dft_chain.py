"""The FP32 FFT of 32 to 128 tones, whose kernel stages its twiddles and divides by multiplication: the first and last
counts that take it, their neighbours, and every mix of radices between, with one channel, a CTA's tile of channels and
one more, and many.  Tolerance: the FFT's, 20 * 2^-24 of a channel's largest phasor (FP64 reference)."""
import numpy as np
import pytest

pytestmark = pytest.mark.gpu

COUNTS = [30, 32, 35, 36, 42, 45, 48, 49, 54, 60, 63, 64, 70, 72, 75, 80, 81, 84, 90, 96, 98, 100, 105, 108, 112, 120, 125,
          126, 128, 135]


@pytest.mark.parametrize("N", COUNTS)
def test_chain_kernel(N):
    import torch

    from paper_2501_05993_gb300 import build as libbuild

    libbuild.build()
    import paper_2501_05993_gb300 as pcal

    pcal.load()
    tile = 2048 // N
    rng = np.random.default_rng(N)
    with pcal.Dft(N, "fp32") as d:
        for C in (1, tile, 152 * tile + 1):
            P = ((rng.standard_normal((C, N)) + 1j * rng.standard_normal((C, N))) * 10.0 ** rng.uniform(-3, 6, (C, 1)))
            P = P.astype(np.complex64)
            dT = torch.full((C + 2, N), complex(7.0, -7.0), dtype=torch.complex64, device="cuda")
            d.execute(torch.from_numpy(P).cuda(), C, dT)
            assert d.check() == 0
            T = dT.cpu().numpy()
            assert np.all(T[C:] == complex(7.0, -7.0))  # rows beyond C stay as they are
            ref = np.fft.fft(P.astype(np.complex128), axis=1)
            err = np.max(np.abs(T[:C] - ref), axis=1) / np.max(np.abs(ref), axis=1)
            assert err.max() <= 20 * 2.0**-24, (C, err.max())
