"""The calls that a program using this package makes, for measuring it.

Three kinds of pass, each through the package's public entry points:

* ``modes``: decompose a record -- ``SPOD.fit``, the eigenvalues, ``SPOD.modes``;
* ``grad``: differentiate a loss on eigenvalues -- ``spod_eigs`` and its backward pass;
* ``coeffs``: expand a record in modes found before -- ``spod_coeffs`` and ``spod_reconstruct``.

The records are those of the two analyses this package is built for, at their
sizes: a twin-jet field (512 x 256 points, 3 variables, 10 000 snapshots,
blocks of 512) and one-year reanalysis records on lat-lon grids (blocks of 256
to 720), with smaller grids, the FP64 correctness grid, the gradient and
coefficient workloads, and block lengths and grids that fit no tile.  The
fields are made of coherent patterns at a few tones, broadband turbulence (many
patterns of decreasing strength, each with a red spectrum of its own), a little
noise that is independent from point to point, and a mean that differs from
point to point.
"""
import math

import numpy as np
import torch

from paper_2309_11808_gb300 import SPOD, _lib, spod_eigs

DTYPES = {"f32": torch.float32, "f64": torch.float64, "bf16": torch.bfloat16, "c64": torch.complex64}
BYTES = {"f32": 4, "f64": 8, "bf16": 2, "c64": 8}


def _case(name, kind, npoints, nvars, nt, nfft, noverlap, dtype, precision, nmodes):
    return dict(name=name, kind=kind, npoints=npoints, nvars=nvars, nt=nt, nfft=nfft, noverlap=noverlap,
                dtype=dtype, precision=precision, nmodes=nmodes)


def listed():
    return [
        # a quick look at one variable on a coarse grid: launches and the eigen-solver's chain
        _case("quick_look", "modes", 64 * 32, 1, 2048, 256, 128, "f32", "bf16x3", 5),
        # the same grid in FP64, all modes: the reference run a user checks the others with
        _case("reference_f64", "modes", 64 * 32, 1, 2048, 256, 128, "f64", "fp64", 15),
        # a station network of ten daily years, blocks of 360 days with 75 % overlap: an odd
        # number of points and a block length that no kernel is compiled for
        _case("stations_f32", "modes", 9999, 1, 3650, 360, 270, "f32", "fp32", 8),
        # a quarter of the jet grid, every mode (a full basis for a reduced-order model)
        _case("jet_all_modes", "modes", 256 * 128, 3, 10000, 512, 256, "f32", "bf16x3", 38),
        # the whole jet grid, the leading modes (what an analysis plots): the largest record
        _case("jet_leading", "modes", 512 * 256, 3, 10000, 512, 256, "f32", "bf16x3", 5),
        # plain FP32 arithmetic, every mode
        _case("jet_f32", "modes", 128 * 128, 3, 10000, 512, 256, "f32", "fp32", 38),
        # half-degree reanalysis, three-hourly year in blocks of 90 days
        _case("year_720", "modes", 361 * 720, 2, 2920, 720, 360, "f32", "bf16x3", 3),
        # half-degree reanalysis, two-hourly year in blocks of 32 days
        _case("year_384", "modes", 361 * 720, 2, 4380, 384, 192, "f32", "bf16x3", 5),
        # the same record archived in BF16 and decomposed in BF16, shorter blocks
        _case("archive_bf16", "modes", 361 * 720, 2, 4380, 256, 128, "bf16", "bf16", 5),
        # a complex field (velocity components u + iv): the two-sided spectrum
        _case("complex_field", "modes", 128 * 128, 3, 6000, 512, 256, "c64", "bf16x3", 5),
        # sensitivities: the gradient of the leading eigenvalues with respect to the data
        _case("sensitivity", "grad", 256 * 128, 2, 4096, 256, 128, "f32", "bf16x3", 2),
        # compression: coefficients of a record in its modes, and the record from them
        _case("compression", "coeffs", 256 * 128, 2, 4096, 256, 128, "f32", "bf16x3", 2),
    ]


def _blocks(c):
    return (c["nt"] - c["noverlap"]) // (c["nfft"] - c["noverlap"])


def _bins(c):
    return c["nfft"] if c["dtype"] == "c64" else c["nfft"] // 2 + 1


def _log(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def draw(rng):
    largest = _flops(listed()[4]), work(listed()[4])["bytes"]
    while True:
        kind = rng.choice(["modes"] * 7 + ["grad"] * 2 + ["coeffs"])
        nfft = rng.choice([256, 384, 512, 720] * 3 + [64, 96, 100, 125, 128, 180, 200, 240, 300, 320, 360, 480, 625])
        noverlap = rng.choice([nfft // 2] * 3 + [nfft // 4 * 3, nfft // 4, 0, rng.randrange(nfft * 3 // 4)])
        dtype, precision = rng.choice([("f32", "bf16x3")] * 5 + [("f32", "fp32")] * 3 +
                                      [("f64", "fp64"), ("bf16", "bf16x3"), ("bf16", "bf16"), ("c64", "bf16x3"),
                                       ("c64", "fp32")])
        if kind != "modes":
            dtype, precision = "f32", rng.choice(["bf16x3", "bf16x3", "fp32"])
        nb = rng.randint(4, 60)
        nt = noverlap + nb * (nfft - noverlap) + rng.randrange(nfft - noverlap)
        npoints = _log(rng, 1000, 270000)
        if rng.random() < 0.6:
            npoints = npoints // 32 * 32
        nvars = rng.choice([1, 1, 2, 3])
        c = _case("", kind, npoints, nvars, nt, nfft, noverlap, dtype, precision,
                  2 if kind != "modes" else rng.choice([1, 3, 5, 5, 10, nb]))
        c["nmodes"] = min(c["nmodes"], nb)
        del c["name"]
        if nt > 12000 or nb != _blocks(c):
            continue
        # FP64 and FP32 arithmetic run far below the tensor rate, and the longest records come in
        # the block lengths listed: smaller records otherwise
        cost = _flops(c) * {"fp64": 200, "fp32": 8}.get(precision, 1)
        if cost > largest[0] or work(c)["bytes"] > largest[1] * (
                0.5 if kind != "modes" else 1 if nfft in (256, 384, 512, 720) else 0.3):
            continue
        return c


def _flops(c):
    M, nb, nf, N = c["npoints"] * c["nvars"], _blocks(c), _bins(c), c["nfft"]
    fft = (5.0 if c["dtype"] == "c64" else 2.5) * N * math.log2(N) * nb * M
    gram = 4.0 * nf * nb * (nb + 1) * M
    if c["kind"] == "modes":
        return fft + gram + 8.0 * nf * nb * c["nmodes"] * M
    if c["kind"] == "grad":
        return 2 * fft + gram + 8.0 * nf * nb * nb * M
    K = 2 * c["nmodes"] * len(_tones(c))
    return 4.0 * K * c["nt"] * M + 2.0 * K * K * M


def work(c):
    M, nb, nf = c["npoints"] * c["nvars"], _blocks(c), _bins(c)
    x = c["nt"] * M * BYTES[c["dtype"]]
    cplx = 16 if c["precision"] == "fp64" else 8
    if c["kind"] == "modes":
        return {"bytes": x + nf * c["nmodes"] * M * cplx, "flops": _flops(c)}
    if c["kind"] == "grad":
        return {"bytes": 2 * x, "flops": _flops(c)}
    # the record and the modes in, the coefficients out; modes and coefficients in, the record out
    nsel = len(_tones(c))
    return {"bytes": 2 * (x + nsel * c["nmodes"] * (M * cplx + c["nt"] * 16)), "flops": _flops(c)}


def _tones(c):
    """The bins of the coherent patterns: 16 over the lower nine tenths of the spectrum."""
    return sorted({max(1, int(c["nfft"] * 0.45 * (j + 1) / 16)) for j in range(16)})


def _red(e):
    """AR(1) in time: e_t + phi e_(t-1) + phi^2 e_(t-2) + ..., 128 terms."""
    for s in range(7):
        if e.shape[0] > 1 << s:
            e[1 << s:] = torch.add(e[1 << s:], e[:-(1 << s)], alpha=0.9 ** (1 << s))
    return e


def _record(c, seed):
    """X[nt][M] on the GPU and the quadrature weights W[M]."""
    dev, nt, M = torch.device("cuda"), c["nt"], c["npoints"] * c["nvars"]
    g = torch.Generator(device=dev)
    g.manual_seed(seed)
    cols = 2 * M if c["dtype"] == "c64" else M
    ft = torch.float64 if c["dtype"] == "f64" else torch.float32
    tones, n = _tones(c), 96
    t = torch.arange(nt, device=dev, dtype=torch.float64)[:, None]
    k = torch.tensor([b for b in tones for _ in range(2)], device=dev, dtype=torch.float64)[None]
    # two patterns a tone, the second a little off the bin, so that they are not coherent
    k = k + 0.37 * (torch.arange(2 * len(tones), device=dev) % 2)[None]
    amp = torch.tensor([a for j in range(len(tones)) for a in (0.5 / (1 + j / 8), 0.3 / (1 + j / 8))], device=dev,
                       dtype=torch.float64)[None]
    T = amp * torch.sin(2 * math.pi * k * t / c["nfft"] +
                        6.28 * torch.rand(1, 2 * len(tones), generator=g, device=dev, dtype=torch.float64))
    broad = _red(torch.randn(nt, n, generator=g, device=dev, dtype=torch.float64)) * \
        0.3 / torch.arange(1, n + 1, device=dev, dtype=torch.float64).sqrt()
    T = torch.cat([T, broad], 1).to(ft)
    n = T.shape[1]
    x = (torch.arange(cols, device=dev, dtype=ft) / cols)[None]
    centre = torch.rand(n, 1, generator=g, device=dev, dtype=ft)
    wave = 20 + 200 * torch.rand(n, 1, generator=g, device=dev, dtype=ft)
    S = torch.exp(-((x - centre) / 0.15) ** 2) * torch.cos(6.28 * wave * (x - centre))
    mean = 5 * torch.randn(1, cols, generator=g, device=dev, dtype=ft)
    X = torch.empty(nt, cols, device=dev, dtype=DTYPES[c["dtype"]] if c["dtype"] != "c64" else ft)
    w = max(1, (1 << 28) // nt)                      # columns at a time
    for a in range(0, cols, w):
        b = min(cols, a + w)
        e = torch.randn(nt, b - a, generator=g, device=dev, dtype=ft).mul_(0.03)
        X[:, a:b] = e.addmm_(T, S[:, a:b]).add_(mean[:, a:b])
    if c["dtype"] == "c64":
        X = torch.view_as_complex(X.view(nt, M, 2))
    W = 0.1 + np.random.default_rng(seed).random(M)
    return X, W


def prepare(c, seed):
    X, W = _record(c, seed)
    sp = SPOD(c["npoints"], c["nvars"], c["nt"], c["nfft"], c["noverlap"], dtype=X.dtype, precision=c["precision"],
              weights=W)
    s = dict(case=c, X=X, plan=sp)
    if c["kind"] == "grad":
        X.requires_grad_()
    if c["kind"] == "coeffs":
        sp.fit(X)
        s["phi"] = sp.modes(X, c["nmodes"])
    return s


def _working(c, v):
    """Eigenvalues and coefficients come in FP64 whatever the plan computes in; a program
    keeps them in the type it works in, beside its modes."""
    if c["precision"] == "fp64":
        return v
    return v.to(torch.complex64 if v.is_complex() else torch.float32)


def run(s):
    c, X, sp = s["case"], s["X"], s["plan"]
    if c["kind"] == "modes":
        sp.fit(X)
        lam = torch.empty(sp.nf, sp.nb, dtype=torch.float64, device=X.device)
        _lib.spod_get_eigs(sp.handle, lam, None, on_device=True)
        return {"lam": _working(c, lam), "phi": sp.modes(X, c["nmodes"])}
    if c["kind"] == "grad":
        lam = spod_eigs(X, sp)
        loss = lam[_tones(c), :c["nmodes"]].sum()
        (dX,) = torch.autograd.grad(loss, X)
        return {"lam": _working(c, lam.detach()), "grad": dX}
    stream, sel = torch.cuda.current_stream(X.device), _tones(c)  # the modes of the coherent bins
    A = torch.empty(len(sel), c["nmodes"], c["nt"], dtype=torch.complex128, device=X.device)
    _lib.spod_coeffs(sp.handle, X, s["phi"], c["nmodes"], c["nmodes"], sel, A, stream)
    Xr = torch.empty_like(X)
    _lib.spod_reconstruct(sp.handle, s["phi"], c["nmodes"], c["nmodes"], sel, A, Xr, stream)
    return {"coeffs": _working(c, A), "record": Xr}


# ---------------------------------------------------------------- the same in FP64 torch
def _window(c, dev):
    n = torch.arange(c["nfft"], device=dev, dtype=torch.float64)
    w = 0.54 - 0.46 * torch.cos(2 * math.pi * n / (c["nfft"] - 1))
    return w / w.sum()


def _spectra(c, x, w):
    """Qhat [nf][nb][columns] of FP64 columns x[nt][columns] with their mean removed."""
    q = x.unfold(0, c["nfft"], c["nfft"] - c["noverlap"]) * w          # [nb][columns][nfft]
    return (torch.fft.fft(q) if x.is_complex() else torch.fft.rfft(q)).permute(2, 0, 1)


def _columns(c, X):
    """Chunks of columns whose spectra take about 1 GB."""
    w = max(64, (1 << 30) // (16 * _blocks(c) * c["nfft"]))
    for a in range(0, X.shape[1], w):
        x = X[:, a:a + w]
        x = x.to(torch.complex128 if x.is_complex() else torch.float64)
        yield a, x - x.mean(0, keepdim=True)


def _decompose(c, X, W):
    nb, w = _blocks(c), _window(c, X.device)
    G = torch.zeros(_bins(c), nb, nb, dtype=torch.complex128, device=X.device)
    for a, x in _columns(c, X):
        q = _spectra(c, x, w) * W[a:a + x.shape[1]].sqrt()
        G += q.conj() @ q.transpose(1, 2)
    lam, psi = np.linalg.eigh((G / nb).cpu().numpy())
    lam, psi = lam[:, ::-1].copy(), psi[:, :, ::-1].copy()
    top = np.take_along_axis(psi, np.abs(psi).argmax(1)[:, None, :], 1)
    psi = psi * (np.abs(top) / top)                  # largest entry real and positive
    return torch.from_numpy(lam).to(X.device), torch.from_numpy(psi).to(X.device)


def _modes(c, X, lam, psi, n):
    w, M = _window(c, X.device), X.shape[1]
    B = (psi[:, :, :n] / (_blocks(c) * lam[:, None, :n]).sqrt()).transpose(1, 2)
    phi = torch.empty(_bins(c), n, M, dtype=torch.complex128, device=X.device)
    for a, x in _columns(c, X):
        phi[:, :, a:a + x.shape[1]] = B @ _spectra(c, x, w)
    return phi


def _gradient(c, X, W, psi):
    w = _window(c, X.device)
    k, P = _tones(c), psi[_tones(c), :, :c["nmodes"]].transpose(1, 2).contiguous()
    out = torch.empty(X.shape, dtype=torch.float64, device=X.device)
    for a in range(0, X.shape[1], 2048):
        with torch.enable_grad():
            x = X[:, a:a + 2048].double().requires_grad_()
            q = _spectra(c, x - x.mean(0, keepdim=True), w)[k]
            loss = ((P @ q).abs().square() * W[a:a + 2048]).sum() / _blocks(c)
            (out[:, a:a + 2048],) = torch.autograd.grad(loss, x)
    return out


def _expansion(c, X, W, phi):
    P = torch.cat([torch.cat([p.real, p.imag]) for p in phi[_tones(c)]])      # [K][M]
    mu = X.double().mean(0)
    B = torch.cat([(P * W) @ (X[t:t + 256].double() - mu).T for t in range(0, X.shape[0], 256)], 1)
    C = torch.linalg.solve((P * W) @ P.T, B)                                     # [K][nt]
    n = c["nmodes"]
    A = torch.stack([torch.complex(0.5 * v[:n], -0.5 * v[n:]) for v in C.split(2 * n)])
    rec = torch.cat([mu + C[:, t:t + 256].T @ P for t in range(0, X.shape[0], 256)])
    return {"coeffs": A, "record": rec}


@torch.no_grad()
def exact(c, seed):
    X, W = _record(c, seed)
    W = torch.from_numpy(W).to(X.device)
    lam, psi = _decompose(c, X, W)
    if c["kind"] == "grad":
        return {"lam": lam, "grad": _gradient(c, X, W, psi)}
    phi = _modes(c, X, lam, psi, c["nmodes"])
    return {"lam": lam, "phi": phi} if c["kind"] == "modes" else _expansion(c, X, W, phi)
