"""The tile width of the pipelined FFT: the plan reports the form it runs, a width that was
set is the one that runs whatever the grid, and both forms give the spectra at overlaps
where the folded mean finds its new snapshots inside the passes and where it reads
them again (N - step no multiple of the first pass's stride)."""
import ctypes
import re

import numpy as np
import pytest
import torch

import oracle as O
from paper_2309_11808_gb300 import SPOD, _lib

pytestmark = pytest.mark.gpu


def _tiles_run(sp, X, path):
    """Tile widths of the pipelined FFT kernels that a fit launches, from their names in
    the dump of a graph it was captured into."""
    g = torch.cuda.CUDAGraph(keep_graph=True)
    with torch.cuda.graph(g):
        sp.fit(X)
    dump = ctypes.CDLL("libcuda.so.1").cuGraphDebugDotPrint
    assert dump(ctypes.c_void_p(g.raw_cuda_graph()), str(path).encode(), 1) == 0
    text = path.read_text()
    assert "k_fft_pipe" in text
    # <input, output kind, tile, nfft, ..>, mangled or not
    found = re.findall(r"k_fft_pipe(?:I\w+?Li\d+ELi(\d+)ELi\d+E|<[^,]+, [^,]+, [^,\d]*(\d+),)", text)
    return {int(a or b) for a, b in found}


@pytest.mark.parametrize("npts,first", [(300, 16), (32 * 152 + 44, 32)])
def test_the_width_that_was_set_runs(npts, first, tmp_path):
    nt, nfft = 1024, 256
    X = torch.randn(nt, npts, generator=torch.Generator().manual_seed(1)).cuda()
    sp = SPOD(npts, 1, nt, nfft, 128, precision="bf16x3")
    sms = torch.cuda.get_device_properties(0).multi_processor_count
    if sms == 152:
        assert _lib.spod_plan_get_tuning(sp.handle).fft_tile_points == first
    sp.fit(X)
    assert _tiles_run(sp, X, tmp_path / "g0") == {_lib.spod_plan_get_tuning(sp.handle).fft_tile_points}
    for tp in (32, 16, 32):
        _lib.spod_plan_set_tuning(sp.handle, fft_tile_points=tp)
        assert _lib.spod_plan_get_tuning(sp.handle).fft_tile_points == tp
        assert _tiles_run(sp, X, tmp_path / "g") == {tp}
    sp.close()


@pytest.mark.parametrize("dtype,precision", [(torch.float32, "bf16x3"), (torch.float32, "fp32"),
                                             (torch.bfloat16, "bf16x3"), (torch.complex64, "bf16x3")])
@pytest.mark.parametrize("nfft,nov", [(256, 0), (256, 192), (256, 100), (384, 288), (384, 92), (512, 384), (512, 12),
                                      (720, 540), (720, 44)])
def test_both_widths_at_all_overlaps(nfft, nov, dtype, precision):
    M, nb = 296, 3
    nt = nfft + (nb - 1) * (nfft - nov) + 5
    x = torch.randn(nt, M, generator=torch.Generator().manual_seed(nfft + nov),
                    dtype=torch.complex64 if dtype.is_complex else torch.float32)
    X = (x + 3.0).to(dtype)
    W = 0.5 + np.random.default_rng(nfft).random(M)
    sp = SPOD(M, 1, nt, nfft, nov, dtype=dtype, precision=precision, weights=W)
    assert sp.nb == nb
    X64 = X.to(torch.complex128 if dtype.is_complex else torch.float64).numpy()
    Q = O.block_dft(X64, nfft, nov, O.window("hamming", nfft), O.time_mean(X64), method="fft")
    n2 = np.sqrt((np.abs(Q) ** 2 * W).sum(-1))
    # the gate of test_gpu_fft_tiles.py
    scale = n2[:, :, None] * n2[:, None, :] / nb
    tol = (2 * 2.0 ** -15 if precision == "bf16x3" else 0.0) * scale + 1e-6 * scale.max()
    ran = 0
    for tp in (16, 32):
        try:
            _lib.spod_plan_set_tuning(sp.handle, fft_tile_points=tp)
        except _lib.SpodError:
            continue
        ran += 1
        sp.fit(X.cuda())
        assert (np.abs(sp.gram() - O.gram(Q, W)) <= tol).all(), tp
    assert ran
    sp.close()
