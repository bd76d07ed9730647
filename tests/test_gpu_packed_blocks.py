"""Tensor-core Gram and modes over every row padding: several blocks of
few rows share an item of the Gram and several tiles a copy of the modes, so ragged point counts and
last chunks smaller than the ones before them (whose blocks still hold the
previous chunk's spectra) are where these kernels can go wrong."""
import numpy as np
import pytest
import torch

import oracle as O
from paper_2309_11808_gb300 import SPOD

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("npts,chunk", [(65, 0), (1000, 0), (1411, 640), (2000, 1024)])
@pytest.mark.parametrize("nb", [1, 3, 7, 8, 15, 16, 21, 24, 31, 32, 33])
def test_gram_and_modes_over_row_paddings(nb, npts, chunk):
    # every entry of the Gram and of the modes against FP64 arithmetic on the
    # oracle's spectra.  q = hi + lo leaves 2^-17 |q| (half an ulp of lo); of a
    # product of two such numbers lo * lo (2^-16) is dropped: with both operands
    # split, 2 x 2^-17 + 2^-16 = 2^-15 of the sum of absolute products, and as
    # much again for the FP32 transform, sums and coefficients
    nfft, nov = 32, 0
    nt = nfft * nb + 5
    g = torch.Generator().manual_seed(100 * nb + npts)
    X = (torch.randn(nt, npts, generator=g) + 3.0).float()
    W = (0.5 + torch.rand(npts, generator=g)).double().numpy()
    sp = SPOD(npts, 1, nt, nfft, nov, precision="bf16x3", weights=W, chunk_points=chunk)
    Xd = X.cuda()
    sp.fit(Xd)
    lam, psi = sp.eigs(vectors=True)
    nm = min(nb, 5)
    Phi = sp.modes(Xd, nm).cpu().numpy()
    G = sp.gram()
    X64 = X.double().numpy()
    Q = O.block_dft(X64, nfft, nov, O.window("hamming", nfft), O.time_mean(X64))       # [nf][nb][M]
    n2 = np.sqrt((np.abs(Q) ** 2 * W).sum(-1))                   # sqrt of the Gram's diagonal, nb kappa = 1
    assert (np.abs(G - O.gram(Q, W)) <= 2 * 2.0 ** -15 * n2[:, :, None] * n2[:, None, :] / nb).all()
    keep = lam[:, :nm] > 1e-12 * lam[:, :1]
    B = psi[:, :, :nm] / np.sqrt(nb * np.where(keep, lam[:, :nm], 1.0))[:, None, :] * keep[:, None, :]
    want = np.einsum("flk,flm->fkm", B, Q)
    scale = np.einsum("flk,flm->fkm", np.abs(B), np.abs(Q))
    # the spectra's own FP32 error is relative to the block's samples, not to one bin
    floor = np.einsum("flk,lm->fkm", np.abs(B), np.sqrt((np.abs(Q) ** 2).mean(0)))
    assert (np.abs(Phi - want) <= 2 * 2.0 ** -15 * (scale + floor)).all()
