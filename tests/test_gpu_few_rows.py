"""The basis Gram of a few rows over many points: its sums are split over the points, so
row counts at the edges of the 4 x 4 tiles and of the split, ragged parts, and the
time of a call, which must fall with the rows."""
import numpy as np
import pytest
import torch

from paper_2309_11808_gb300 import SPOD, _lib
from test_gpu_coeffs import _run

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("fsel,nr", [([0], 1), ([6], 1), ([0, 6, 64], 1), ([6, 13], 1), ([0, 6, 13], 1),
                                     ([6, 13, 30], 2), (list(range(1, 21)), 1), (list(range(1, 23)), 1)])
@pytest.mark.parametrize("npts", [2047, 5003])
@pytest.mark.parametrize("prec,dtype,tol", [("fp64", torch.float64, 1e-9), ("fp32", torch.float32, 1e-4)])
def test_coefficients_of_few_rows(fsel, nr, npts, prec, dtype, tol):
    A, Aref, Xr, Xref, X = _run(prec, dtype, fsel, nr, npts=npts, nt=700)
    assert np.abs(A - Aref).max() <= tol * np.abs(Aref).max()
    assert np.abs(Xr - Xref).max() <= tol * np.abs(X).max()


def test_few_rows_take_a_fraction_of_the_time_of_many():
    # a short record on a large grid, where the Gram is most of the call.  On GB300:
    # 4 rows 0.47 of the time of 64 when each tile's CTA walked all the points
    M, nt, nfft = 262144, 300, 128
    X = torch.randn(nt, M, generator=torch.Generator(device="cuda").manual_seed(1), device="cuda")
    sp = SPOD(M, 1, nt, nfft, 0, precision="fp32")
    sp.fit(X)
    Phi = sp.modes(X, 1)

    def best(bins):
        A = torch.empty(len(bins), 1, nt, dtype=torch.complex128, device="cuda")
        ms = []
        for _ in range(8):
            a, b = torch.cuda.Event(enable_timing=True), torch.cuda.Event(enable_timing=True)
            a.record()
            _lib.spod_coeffs(sp.handle, X, Phi, 1, 1, bins, A)
            b.record()
            b.synchronize()
            ms.append(a.elapsed_time(b))
        return min(ms[2:])

    few, many = best([1, 2]), best(list(range(1, 33)))
    print("4 rows %.3f ms, 64 rows %.3f ms" % (few, many))
    sp.sync()
    sp.close()
    assert few <= 0.3 * many
