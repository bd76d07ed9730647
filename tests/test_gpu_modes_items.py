"""Tensor-core modes on small grids: how many tiles an item holds follows the CTAs
(one CTA: the most; more CTAs than tiles: one), and changes no bit of the result."""
import pytest
import torch

from paper_2309_11808_gb300 import SPOD, _lib

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("precision", ["bf16", "bf16x3"])
@pytest.mark.parametrize("npts", [65, 300, 1001, 2100])
@pytest.mark.parametrize("nb", [1, 7, 20])
def test_modes_do_not_depend_on_the_tiles_of_an_item(precision, npts, nb):
    nfft = 32
    X = torch.randn(nfft * nb + 3, npts, generator=torch.Generator().manual_seed(npts + nb)).cuda()
    sp = SPOD(npts, 1, nfft * nb + 3, nfft, 0, precision=precision)
    sp.fit(X)
    want = None
    for ctas in (1, 5, 40, 152, 4096):
        _lib.spod_plan_set_tuning(sp.handle, modes_ctas=ctas)
        phi = sp.modes(X, min(nb, 5))
        sp.sync()
        assert torch.isfinite(torch.view_as_real(phi)).all()
        if want is None:
            want = phi
        assert torch.equal(torch.view_as_real(phi), torch.view_as_real(want))
    sp.close()
