"""The eigen-solver on real symmetric Grams (DC and Nyquist of real data): the last
column of the reduction takes no reflection there, so its tau is converted straight
after it was written -- by another warp from nb = 34 on.  Gates, relative to lambda_1:
those of test_gpu_eigsolver.py (FP64 1e-13, double-FP32 1e-11)."""
import numpy as np
import pytest
import torch

from paper_2309_11808_gb300 import SPOD, _lib

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("nb", [2, 3, 33, 34, 35, 38, 48, 49, 64])
@pytest.mark.parametrize("prec,tol", [("fp64", 1e-13), ("fp32", 1e-11), ("bf16x3", 1e-11)])
def test_real_symmetric_grams(nb, prec, tol):
    nfft = 16
    dt = torch.float64 if prec == "fp64" else torch.float32
    sp = SPOD(16, 1, nfft * nb, nfft, 0, dtype=dt, precision=prec)
    assert sp.nb == nb
    st = torch.cuda.current_stream()
    X = torch.randn(nfft * nb, 16, dtype=dt, device="cuda")
    part = torch.empty((sp.nf, nb, nb, 2), dtype=torch.float64, device="cuda")
    _lib.spod_fit_partial(sp.handle, X, part, st)
    rng = np.random.default_rng(nb)
    m = np.empty((sp.nf, nb, nb))
    for f in range(sp.nf):
        q = np.linalg.qr(rng.standard_normal((nb, nb)))[0]
        a = (q * rng.uniform(0.05, 1.0, nb)) @ q.T * 10.0 ** (f % 5 - 2)
        m[f] = 0.5 * (a + a.T)
    g = torch.zeros((1, sp.nf, nb, nb, 2), dtype=torch.float64, device="cuda")
    g[0, ..., 0] = torch.from_numpy(m).cuda()
    for _ in range(3):
        _lib.spod_fit_from_grams(sp.handle, g, 1, st)
        lam, psi = sp.eigs(vectors=True)
        w = np.linalg.eigvalsh(m)[:, ::-1]
        scale = w[:, :1]
        assert (np.abs(lam - w) <= tol * scale).all()
        assert (np.linalg.norm(m @ psi - psi * lam[:, None, :], axis=1) <= tol * scale).all()
        assert np.abs(np.conj(psi.transpose(0, 2, 1)) @ psi - np.eye(nb)).max() <= tol
    sp.close()


@pytest.mark.parametrize("nb", [34, 41])
def test_dc_and_nyquist_of_real_data(nb):
    nfft = 32
    g = torch.Generator().manual_seed(nb)
    sp = SPOD(500, 1, nfft * nb, nfft, 0, precision="fp32")
    sp.fit(torch.randn(nfft * nb, 500, generator=g).cuda())
    lam, psi = sp.eigs(vectors=True)
    G = sp.gram()
    for f in (0, nfft // 2):
        assert np.abs(G[f].imag).max() <= 1e-12 * lam[f, 0]
        assert np.linalg.norm(G[f] @ psi[f] - psi[f] * lam[f], axis=0).max() <= 1e-11 * lam[f, 0]
        assert np.abs(psi[f].conj().T @ psi[f] - np.eye(nb)).max() <= 1e-11
    sp.close()
