"""FP32 products at the edges of their tiles: the coefficient GEMMs (64 x 128 tiles,
16-byte loads where the sizes allow them, the product over the points in several
parts) against the oracle at the gate of the FP32 plan, and the modes in both forms
(packed pairs, or 8-byte coefficients for many blocks) against FP64 arithmetic."""
import numpy as np
import pytest
import torch

import oracle as O
from paper_2309_11808_gb300 import SPOD
from test_gpu_coeffs import _run

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("npts,nt,fsel,nr", [(773, 1100, [0, 6, 13], 1), (1540, 1027, [6, 13, 30], 2),
                                             (4100, 640, [0, 6, 13, 30, 64], 3), (2051, 1024, [13], 1)])
def test_coefficient_products(npts, nt, fsel, nr):
    A, Aref, Xr, Xref, X = _run("fp32", torch.float32, fsel, nr, npts=npts, nt=nt)
    assert np.abs(A - Aref).max() <= 1e-4 * np.abs(Aref).max()
    assert np.abs(Xr - Xref).max() <= 1e-4 * np.abs(X).max()


@pytest.mark.parametrize("nb,nmodes", [(5, 5), (19, 19), (20, 20), (38, 38), (39, 1), (60, 59), (64, 64),
                                       (100, 97), (170, 160)])
@pytest.mark.parametrize("npts", [257, 770])
def test_fp32_modes(nb, nmodes, npts):
    # Phi = Qhat B, B from the plan's own eigenpairs: the spectra to a few FP32
    # roundings of the block's samples, nb products and sums of two terms in FP32
    nfft = 16
    g = torch.Generator().manual_seed(nb + npts)
    X = torch.randn(nfft * nb, npts, generator=g)
    sp = SPOD(npts, 1, nfft * nb, nfft, 0, precision="fp32")
    sp.fit(X.cuda())
    lam, psi = sp.eigs(vectors=True)
    Phi = sp.modes(X.cuda(), nmodes).cpu().numpy()
    X64 = X.double().numpy()
    Q = O.block_dft(X64, nfft, 0, O.window("hamming", nfft), O.time_mean(X64))
    keep = lam[:, :nmodes] > 1e-12 * lam[:, :1]
    B = psi[:, :, :nmodes] / np.sqrt(nb * np.where(keep, lam[:, :nmodes], 1.0))[:, None, :] * keep[:, None, :]
    want = np.einsum("flk,flm->fkm", B, Q)
    rms = np.sqrt((np.abs(Q) ** 2).mean(0))
    bound = np.einsum("flk,flm->fkm", np.abs(B), np.abs(Q) * (2 * nb + 4) + 8 * rms[None]) * 2.0 ** -23
    assert (np.abs(Phi - want) <= bound).all()
