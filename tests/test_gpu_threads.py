"""Plans of different sizes used by several host threads at once, each on its own stream:
the kernels they share take shared memory by the plan's sizes, and one thread's launch
must not change what the other's may take."""
import threading

import pytest
import torch

from paper_2309_11808_gb300 import SPOD, _lib

pytestmark = pytest.mark.gpu


def _plan(npts, nt, nfft, nov, seed):
    g = torch.Generator().manual_seed(seed)
    X = torch.randn(nt, npts, generator=g).cuda()
    sp = SPOD(npts, 1, nt, nfft, nov, precision="fp32")
    sp.fit(X)
    sp.sync()
    return sp, X


@pytest.mark.parametrize("what,calls", [("coeffs", 8000), ("modes", 3000)])
def test_plans_of_different_sizes_from_three_threads(what, calls):
    # (basis rows, or modes x blocks: small for two threads and large for the third; in
    # 16 000 small calls the launches met about five times)
    jobs = []
    for seed, (nfft, nb, bins, nm) in enumerate(((32, 2, [0], 1), (32, 2, [0], 1),
                                                 (128, 2 if what == "coeffs" else 60, list(range(1, 47)),
                                                  1 if what == "coeffs" else 57))):
        sp, X = _plan(256, nfft * nb, nfft, 0, seed)
        Phi = sp.modes(X, nm)
        sp.sync()
        stream = torch.cuda.Stream()
        if what == "coeffs":
            A = torch.empty(len(bins), 1, X.shape[0], dtype=torch.complex128, device="cuda")

            def call(sp=sp, X=X, Phi=Phi, nm=nm, bins=bins, out=A, stream=stream):
                _lib.spod_coeffs(sp.handle, X, Phi, nm, 1, bins, out, stream)
        else:
            A = torch.empty_like(Phi)

            def call(sp=sp, X=X, nm=nm, out=A, stream=stream):
                sp.modes(X, nm, out=out, stream=stream)
        call()
        stream.synchronize()
        jobs.append((call, A, A.cpu().numpy(), stream, sp))
    errors = []

    def work(call, stream):
        try:
            for i in range(calls):
                call()
                if i % 50 == 49:
                    stream.synchronize()
        except Exception as e:      # reported by the main thread
            errors.append(e)

    threads = [threading.Thread(target=work, args=(j[0], j[3])) for j in jobs]
    for t in threads:
        t.start()
    for t in threads:
        t.join()
    torch.cuda.synchronize()
    assert not errors, errors
    for call, A, want, stream, sp in jobs:
        sp.sync()
        assert (A.cpu().numpy() == want).all()
