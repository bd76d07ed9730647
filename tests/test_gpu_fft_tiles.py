"""The pipelined FFT on grids wide enough for its wide tiles (small grids take
16-point tiles whatever the choice): ragged last tiles, a tail of snapshots in no
block, every input type and arithmetic, against FP64 spectra and the narrow tiles."""
import numpy as np
import pytest
import torch

import oracle as O
from paper_2309_11808_gb300 import SPOD, _lib

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("dtype,precision", [(torch.float32, "bf16x3"), (torch.float32, "fp32"),
                                             (torch.bfloat16, "bf16x3"), (torch.float64, "fp32"),
                                             (torch.complex64, "fp32")])
@pytest.mark.parametrize("nfft", [256, 384, 512, 720])
def test_wide_tiles(nfft, dtype, precision):
    M, nov = 64 * 152 + 40, nfft // 2                # a ragged tile at 16, 32 and 64 points
    nt = nfft + 2 * (nfft - nov) + 7
    nb = 3
    g = torch.Generator(device="cuda").manual_seed(nfft)
    x = torch.randn(nt, M, generator=g, device="cuda", dtype=torch.complex64 if dtype.is_complex else torch.float32)
    X = (x + 3.0).to(dtype)
    W = 0.5 + np.random.default_rng(nfft).random(M)
    sp = SPOD(M, 1, nt, nfft, nov, dtype=dtype, precision=precision, weights=W)
    sp.fit(X)
    G = sp.gram()
    X64 = X.to(torch.complex128 if dtype.is_complex else torch.float64).cpu().numpy()
    Q = O.block_dft(X64, nfft, nov, O.window("hamming", nfft), O.time_mean(X64), method="fft")
    n2 = np.sqrt((np.abs(Q) ** 2 * W).sum(-1))
    # the spectra to a few FP32 roundings of the block's samples (the largest bin's
    # scale); bf16x3: 2^-15 of the row norms (hi + lo products without lo * lo)
    scale = n2[:, :, None] * n2[:, None, :] / nb
    tol = (2 * 2.0 ** -15 if precision == "bf16x3" else 0.0) * scale + 1e-6 * scale.max()
    assert (np.abs(G - O.gram(Q, W)) <= tol).all()
    if _lib.spod_plan_get_tuning(sp.handle).fft_tile_points == 32:
        _lib.spod_plan_set_tuning(sp.handle, fft_tile_points=16)
        sp.fit(X)
        assert (np.abs(sp.gram() - G) <= 1e-6 * scale.max()).all()
