"""The two-pass adjoint (nfft 256, 384, 720, FP32) at ragged and odd point counts,
overlaps from none to three quarters and one that is no multiple of its passes, and
records with a tail, against the oracle's analytic gradient."""
import numpy as np
import pytest
import torch

import oracle as O
from paper_2309_11808_gb300 import SPOD, _lib

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("npts", [37, 64, 301])
@pytest.mark.parametrize("nfft,nov", [(256, 0), (256, 128), (256, 192), (256, 101), (384, 192), (384, 96), (384, 7),
                                      (720, 360), (720, 540), (720, 11)])
def test_gradient_of_the_two_pass_adjoint(nfft, nov, npts):
    # L = sum of all eigenvalues, weighted by bin: G_f is then a multiple of the unit
    # matrix and the gradient smooth in the data (no eigen-gaps).  Gate: that of the
    # gradient tests, 1e-5 of the largest entry
    nt = nfft + 4 * (nfft - nov) + 5
    g = torch.Generator().manual_seed(nfft + nov + npts)
    X = torch.randn(nt, npts, generator=g) + 2.0
    W = (0.5 + torch.rand(npts, generator=g)).double().numpy()
    sp = SPOD(npts, 1, nt, nfft, nov, precision="fp32", weights=W)
    assert sp.nb == 5
    Xd = X.cuda()
    sp.fit(Xd)
    gl = np.repeat(1.0 + np.cos(np.arange(sp.nf))[:, None], sp.nb, 1)
    dX = torch.full((nt, npts), float("nan"), device="cuda")
    _lib.spod_backward(sp.handle, torch.from_numpy(gl).cuda(), Xd, dX)
    _lib.spod_sync(sp.handle)
    d = O.Desc(nt=nt, M=npts, nfft=nfft, noverlap=nov, weights=W)
    X64 = X.double().numpy()
    Q = O.block_dft(X64, nfft, nov, d.w(), O.time_mean(X64), method="fft")
    # sum_l' Qhat[f, l'] G_f[l', l] with G_f = (1 + cos f) I
    R = 2.0 / sp.nb * W * np.transpose(Q, (1, 0, 2)) * (1.0 + np.cos(np.arange(sp.nf)))[None, :, None]   # [nb][nf][M]
    H = np.concatenate([R, np.zeros((sp.nb, nfft - sp.nf, npts))], 1)
    z = np.fft.ifft(H, axis=1).real * nfft
    w = d.w()
    want = np.zeros((nt, npts))
    for l in range(sp.nb):
        want[l * (nfft - nov): l * (nfft - nov) + nfft] += (w / w.sum())[:, None] * z[l]
    want -= want.mean(0)
    assert np.abs(dX.cpu().numpy() - want).max() <= 1e-5 * np.abs(want).max()
