"""The tensor-core Gram off its plain loop: more than 80 rows (one run per tensor-memory
buffer), and accumulation runs of several blocks (gram_flush_blocks), whose groups span
items when a CTA holds several of them; and the adjoint without R's extra column
(nb = 64), which sums the mean of the gradient from R itself."""
import numpy as np
import pytest
import torch

import oracle as O
from paper_2309_11808_gb300 import SPOD, _lib

pytestmark = pytest.mark.gpu


def _check(precision, nb, npts, chunk, flush, splits):
    # BF16X3: the bound of test_gpu_packed_blocks.py.  BF16: each factor is rounded to 2^-9
    # of itself, a product to 2^-8, and 2^-12 for the FP32 transform and sums.  A run
    # of R MMAs (four a block) rounds toward zero, R 2^-24 of the diagonal
    unit = 2 * 2.0 ** -15 if precision == "bf16x3" else 2.0 ** -8 + 2.0 ** -12
    nfft = 32
    nt = nfft * nb + 5
    g = torch.Generator().manual_seed(100 * nb + npts)
    X = (torch.randn(nt, npts, generator=g) + 3.0).float()
    W = (0.5 + torch.rand(npts, generator=g)).double().numpy()
    sp = SPOD(npts, 1, nt, nfft, 0, precision=precision, weights=W, chunk_points=chunk)
    assert sp.nb == nb
    _lib.spod_plan_set_tuning(sp.handle, gram_flush_blocks=flush, gram_splits=splits)
    Xd = X.cuda()
    sp.fit(Xd)
    lam, psi = sp.eigs(vectors=True)
    nm = min(nb, 5)
    Phi = sp.modes(Xd, nm).cpu().numpy()
    G = sp.gram()
    sp.close()
    X64 = X.double().numpy()
    Q = O.block_dft(X64, nfft, 0, O.window("hamming", nfft), O.time_mean(X64))
    n2 = np.sqrt((np.abs(Q) ** 2 * W).sum(-1))
    bound = (unit + 8 * flush * 2.0 ** -24) * n2[:, :, None] * n2[:, None, :] / nb
    assert (np.abs(G - O.gram(Q, W)) <= bound).all()
    keep = lam[:, :nm] > 1e-12 * lam[:, :1]
    B = psi[:, :, :nm] / np.sqrt(nb * np.where(keep, lam[:, :nm], 1.0))[:, None, :] * keep[:, None, :]
    want = np.einsum("flk,flm->fkm", B, Q)
    scale = np.einsum("flk,flm->fkm", np.abs(B), np.abs(Q))
    floor = np.einsum("flk,lm->fkm", np.abs(B), np.sqrt((np.abs(Q) ** 2).mean(0)))
    assert (np.abs(Phi - want) <= unit * (scale + floor)).all()


@pytest.mark.parametrize("precision", ["bf16x3", "bf16"])
@pytest.mark.parametrize("npts,chunk", [(1000, 0), (1411, 640)])
@pytest.mark.parametrize("nb", [7, 24, 40, 41, 48, 49, 56, 57, 63, 64])
def test_gram_and_modes_up_to_128_rows(nb, npts, chunk, precision):
    _check(precision, nb, npts, chunk, 0, 0)


@pytest.mark.parametrize("precision", ["bf16x3", "bf16"])
@pytest.mark.parametrize("flush", [2, 3, 16])
@pytest.mark.parametrize("nb", [3, 16, 20, 30, 40, 45, 64])
@pytest.mark.parametrize("npts,chunk,splits", [(2100, 0, 2), (1411, 640, 3), (2100, 0, 0)])
def test_runs_of_several_blocks(nb, flush, npts, chunk, splits, precision):
    _check(precision, nb, npts, chunk, flush, splits)


@pytest.mark.parametrize("nfft,npts", [(256, 37), (256, 64), (384, 70), (720, 33)])
def test_adjoint_without_the_extra_column(nfft, npts):
    nb = 64
    nt = nfft + (nb - 1) * (nfft // 2) + 5
    g = torch.Generator().manual_seed(nfft + npts)
    X = torch.randn(nt, npts, generator=g) + 2.0
    W = (0.5 + torch.rand(npts, generator=g)).double().numpy()
    sp = SPOD(npts, 1, nt, nfft, nfft // 2, precision="bf16x3", weights=W)
    assert sp.nb == nb
    Xd = X.cuda()
    sp.fit(Xd)
    gl = np.repeat(1.0 + np.cos(np.arange(sp.nf))[:, None], nb, 1)       # G_f a multiple of I, as in test_gpu_adjoint_two.py
    dX = torch.full((nt, npts), float("nan"), device="cuda")
    _lib.spod_backward(sp.handle, torch.from_numpy(gl).cuda(), Xd, dX)
    _lib.spod_sync(sp.handle)
    got = dX.double().cpu().numpy()
    sp.close()
    d = O.Desc(nt=nt, M=npts, nfft=nfft, noverlap=nfft // 2, weights=W)
    X64 = X.double().numpy()
    Q = O.block_dft(X64, nfft, nfft // 2, d.w(), O.time_mean(X64), method="fft")
    R = 2.0 / nb * W * np.transpose(Q, (1, 0, 2)) * (1.0 + np.cos(np.arange(Q.shape[0])))[None, :, None]
    z = np.fft.ifft(np.concatenate([R, np.zeros((nb, nfft - R.shape[1], npts))], 1), axis=1).real * nfft
    w = d.w() / d.w().sum()
    want = np.zeros((nt, npts))
    for l in range(nb):
        want[l * (nfft // 2): l * (nfft // 2) + nfft] += w[:, None] * z[l]
    sums = np.abs(want.sum(0)).max()
    want -= want.mean(0)
    # R's operands split into hi + lo leave 2^-15 of each entry; G_f comes from
    # eigenvectors orthogonal to 1e-11
    assert np.linalg.norm(got - want) <= 1e-4 * np.linalg.norm(want)
    # the mean is taken off: 1e-3 of the sums it removes
    assert np.abs(got.sum(0)).max() <= 1e-3 * sums
