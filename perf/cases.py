"""The work that users of this framework have it do, as measurable cases.

Sizes are those of the repository's workloads (64^3 with 16 shells, the 256^3
particle workload, the 512^3 grid, 50 modal functions, mocks on 96^3 / 128^3 /
160^3 with 24 shells, 512 mocks in a covariance, 8^3 sub-cubes) and, between
them, odd and ragged ones.  Fields follow the repository's synthetic model:
a Gaussian field with P(k) = A k^n_s plus its local quadratic term, Kaiser
distortion along z.  ``exact`` is plain FP64 torch.
"""
import math
import random

import torch

from paper_1708_05303_gb300 import bsp

BOX = 1000.0
F64 = torch.float64


# ---------------------------------------------------------------- the cases
def listed():
    return [
        # the smallest call: one small grid, where launches and latency are the time
        dict(name="bispec_32_f16", kind="bispec", n=32, shells=8, start=1.0, width=2.0, ells="0,2,4", prec="split_f16",
             shot=False, full=False, sigma=0.3),
        # the small workload: 64^3, 16 shells of width 2 k_f, the field not rescaled
        dict(name="bispec_64_fp32", kind="bispec", n=64, shells=16, start=1.0, width=2.0, ells="0,2,4", prec="fp32",
             shot=False, full=False, sigma=0.0),
        # a ragged survey grid: n^3 is no multiple of the point blocks, an odd shell width, two multipoles
        dict(name="bispec_150_f16", kind="bispec", n=150, shells=21, start=1.5, width=1.75, ells="0,2", prec="split_f16",
             shot=False, full=False, sigma=0.3),
        # every Legendre leg, so that other conventions can be read off, in the other split type
        dict(name="full_tensor_128_bf16", kind="bispec", n=128, shells=24, start=1.0, width=1.0, ells="0,2,4",
             prec="split_bf16", shot=False, full=True, sigma=0.3),
        # a particle catalogue's multipoles with Poisson shot noise subtracted (256^3, 32 shells)
        dict(name="shot_256_fp32", kind="bispec", n=256, shells=32, start=1.0, width=2.0, ells="0,2,4", prec="fp32",
             shot=True, full=False, sigma=0.3),
        # the headline grid and k-range (512^3 up to 129 k_f) with half its shells, so that several states fit the card
        dict(name="bispec_512_f16", kind="bispec", n=512, shells=32, start=1.0, width=4.0, ells="0,2,4", prec="split_f16",
             shot=False, full=False, sigma=0.3),
        # the modal estimator with its 50 functions up to 0.3 h/Mpc
        dict(name="modal_256_f16", kind="modal", n=256, modes=50, ells="0,2,4", prec="split_f16"),
        # mock catalogues on uneven grids from host memory, for a covariance
        dict(name="batch_12_fp32", kind="batch", mocks=12, shells=24, ells="0,2,4", prec="fp32"),
        # the covariance of 512 mocks' multipoles (3 x 1654 bins)
        dict(name="covariance_512", kind="cov", mocks=512, dim=4962),
        # a catalogue of 4 Mi particles onto a 256^3 interlaced grid
        dict(name="density_256", kind="density", n=256, particles=4 * 2 ** 20),
        # the skew spectrum: one transform each way and shell sums
        dict(name="skew_256", kind="skew", n=256, shells=32, start=1.0, width=2.0, ells="0,2,4"),
        # the integrated bispectrum: 512 sub-cubes of the 512^3 field
        dict(name="integrated_512", kind="ib", n=512, m=8, shells=64, start=1.0, width=2.0, ells="0,2,4"),
    ]


def _good_sizes(lo, hi):
    out = []
    for n in range(lo, hi + 1, 2):
        m = n
        for q in (2, 3, 5):
            while m % q == 0:
                m //= q
        if m == 1:
            out.append(n)
    return out


def _log_pick(rng, values):
    """One of the ascending values, spread over their logarithm."""
    t = math.exp(rng.uniform(math.log(values[0]), math.log(values[-1])))
    return min(values, key=lambda v: abs(math.log(v / t)))


def draw(rng):
    kind = rng.choice(["bispec", "bispec", "bispec", "shot", "modal", "batch", "cov", "density", "skew", "ib"])
    ells = rng.choice(["0", "0,2", "0,2,4", "0,2,4"])
    if kind in ("bispec", "shot"):
        n = _log_pick(rng, _good_sizes(24, 360 if kind == "bispec" else 256))
        shells = rng.randint(4, 40 if n <= 256 else 24) if kind == "bispec" else rng.randint(4, 32)
        start = rng.choice([1.0, 1.5, 2.0])
        top = rng.uniform(0.2, 0.45) * n
        width = max(1.0, round((top - start) / shells, 2))
        shells = max(3, min(shells, int((0.8 * n - start) / width)))
        full = kind == "bispec" and rng.random() < 0.2 and shells <= 24
        prec = "fp32" if kind == "shot" else rng.choice(["split_f16", "split_f16", "fp32", "split_bf16"])
        return dict(kind="bispec", n=n, shells=shells, start=start, width=width, ells=ells, prec=prec, shot=kind == "shot",
                    full=full, sigma=0.3)
    if kind == "modal":
        prec = rng.choice(["split_f16", "split_f16", "fp32"])
        return dict(kind="modal", n=_log_pick(rng, _good_sizes(32, 120 if prec == "fp32" else 240)), modes=rng.randint(5, 50),
                    ells=ells, prec=prec)
    if kind == "batch":
        return dict(kind="batch", mocks=rng.randint(2, 24), shells=rng.randint(6, 24), ells=ells,
                    prec=rng.choice(["fp32", "split_f16"]))
    if kind == "cov":
        return dict(kind="cov", mocks=int(math.exp(rng.uniform(math.log(20), math.log(1000)))),
                    dim=int(math.exp(rng.uniform(math.log(50), math.log(5000)))))
    if kind == "density":
        return dict(kind="density", n=_log_pick(rng, _good_sizes(32, 512)),
                    particles=int(math.exp(rng.uniform(math.log(2e4), math.log(8e6)))))
    if kind == "skew":
        n = _log_pick(rng, [v for v in _good_sizes(32, 512) if v % 4 == 0])
        shells = rng.randint(8, 64)
        return dict(kind="skew", n=n, shells=shells, start=1.0, width=round(max(0.5, rng.uniform(0.25, 0.5) * n / shells), 2),
                    ells=ells)
    m, s = rng.choice([(2, 32), (2, 60), (4, 24), (4, 48), (4, 64), (4, 90), (8, 16), (8, 32), (8, 48), (8, 64)])
    shells = rng.randint(8, 64)
    return dict(kind="ib", n=m * s, m=m, shells=shells, start=1.0, width=round(rng.uniform(0.3, 0.5) * m * s / shells, 2), ells=ells)


# ------------------------------------------------------------------- inputs
def _ells(case):
    return tuple(int(v) for v in case["ells"].split(","))


def _edges(case):
    return [case["start"] + case["width"] * i for i in range(case["shells"] + 1)]


def _generator(seed):
    return torch.Generator(device="cuda").manual_seed(int(seed) * 7919 + 17)


def _freqs(n):
    j = torch.arange(n, device="cuda")
    return torch.where(j < n // 2, j, j - n)


def _n2(n):
    """|n|^2 and f_z^2 over the half spectrum (integers)."""
    f = _freqs(n)
    fz = torch.arange(n // 2 + 1, device="cuda")
    return f[:, None, None] ** 2 + f[None, :, None] ** 2 + fz[None, None, :] ** 2, (fz ** 2)[None, None, :]


def _gaussian(n, gen, n_s, sigma, amp=2.0e4):
    V, kf = BOX ** 3, 2 * math.pi / BOX
    n2, _ = _n2(n)
    k = kf * n2.to(F64).sqrt()
    P = torch.where(n2 > 0, amp * k.clamp_min(kf).pow(n_s), torch.zeros((), dtype=F64, device="cuda"))
    w = torch.randn((n, n, n), generator=gen, dtype=F64, device="cuda")
    g = torch.fft.irfftn((P * V).sqrt() * torch.fft.rfftn(w) / math.sqrt(n ** 3) * (n ** 3 / V), s=(n, n, n))
    return g * (sigma / g.std()) if sigma else g


def _field(n, seed, n_s=-1.5, f=0.7, sigma=0.3):
    """complex64 half spectrum of the quadratic Kaiser field."""
    g = _gaussian(n, _generator(seed), n_s, sigma)
    d = g + 0.5 * (g * g - (g * g).mean())
    dk = torch.fft.rfftn(d) * (BOX ** 3 / n ** 3)
    n2, fz2 = _n2(n)
    dk = dk * (1.0 + f * fz2.to(F64) / n2.clamp_min(1).to(F64))
    return dk.to(torch.complex64).contiguous()


def _cell_counts(n, gen, particles):
    lam = torch.exp(_gaussian(n, gen, -1.5, 0.3))
    return torch.poisson(lam * (particles / lam.sum()), generator=gen)


def _catalogue(case, seed):
    """float32 positions of a lognormal Poisson sample, in the order of the cells."""
    n, gen = case["n"], _generator(seed)
    cell = torch.repeat_interleave(torch.arange(n ** 3, device="cuda"), _cell_counts(n, gen, case["particles"]).long().flatten())
    pos = torch.stack([cell // (n * n), cell // n % n, cell % n], dim=1).to(F64)
    pos = pos + torch.rand(pos.shape, generator=gen, dtype=F64, device="cuda")
    pos = (pos * (BOX / n)).float()
    return torch.where(pos >= BOX, torch.zeros_like(pos), pos).contiguous()


def _sampled(n, seed):
    """A Poisson-sampled field's half spectrum (counts per cell) and its number density."""
    c = _cell_counts(n, _generator(seed), n ** 3 / 4)
    dk = torch.fft.rfftn(c / c.mean() - 1.0) * (BOX ** 3 / n ** 3)
    return dk.to(torch.complex64).contiguous(), float(c.sum()) / BOX ** 3


def _mock_models(case, seed):
    """(size index, seed, n_s, f) of each mock."""
    r = random.Random(int(seed) * 104729 + 1)
    return [(m % 3, int(seed) * 1009 + m, r.uniform(-2.0, -1.0), r.uniform(0.5, 0.9)) for m in range(case["mocks"])]


_SIZES = (96, 128, 160)


def _mock_rows(case, seed):
    """Rows as mocks give them: multipoles of very different size with common and own scatter."""
    gen = _generator(seed)
    m, d = case["mocks"], case["dim"]
    scale = torch.exp(3.0 * torch.randn(d, generator=gen, dtype=F64, device="cuda")) * 1e8
    own = torch.randn((m, d), generator=gen, dtype=F64, device="cuda")
    common = torch.randn((m, 8), generator=gen, dtype=F64, device="cuda") @ torch.randn((8, d), generator=gen, dtype=F64, device="cuda")
    return (scale * (2.0 + 0.3 * own + 0.2 * common)).contiguous()


def _modal_radial(case):
    kf = 2 * math.pi / BOX
    return bsp.bsp_modal_radial_powerlaw(case["n"], BOX, case["modes"], kf, _modal_kmax(case), 2.0e4, -1.5)


def _modal_kmax(case):
    return min(0.3, 0.9 * math.pi * case["n"] / BOX)


def prepare(case, seed):
    kind = case["kind"]
    if kind == "bispec":
        est = bsp.Bispectrum(case["n"], BOX, _edges(case), _ells(case), prec=case["prec"], shot_noise=case["shot"],
                             full_tensor=case["full"])
        if case["shot"]:
            dk, nbar = _sampled(case["n"], seed)
        else:
            dk, nbar = _field(case["n"], seed, sigma=case["sigma"]), 0.0
        return kind, est, dk, nbar
    if kind == "modal":
        return kind, bsp.Modal(case["n"], BOX, _modal_radial(case), _ells(case), prec=case["prec"]), _field(case["n"], seed)
    if kind == "batch":
        batch = bsp.Batch(_SIZES, BOX, [1.0 + i for i in range(case["shells"] + 1)], _ells(case), prec=case["prec"])
        models = _mock_models(case, seed)
        host = [_field(_SIZES[i], s, n_s, f).cpu().pin_memory() for i, s, n_s, f in models]
        return kind, batch, host, [m[0] for m in models]
    if kind == "cov":
        return kind, _mock_rows(case, seed)
    if kind == "density":
        return kind, case["n"], _catalogue(case, seed)
    est = bsp.Spectra(case["n"], BOX, _edges(case), _ells(case))
    return kind, est, _field(case["n"], seed), case.get("m", 0)


def run(state):
    kind = state[0]
    if kind == "bispec":
        return state[1].compute(state[2], state[3])
    if kind == "modal":
        return state[1].compute(state[2])
    if kind == "batch":
        return state[1].run(state[2], state[3])
    if kind == "cov":
        return bsp.Batch.covariance(state[1])
    if kind == "density":
        return bsp.density_from_particles(state[2], state[1], BOX)
    if kind == "skew":
        return state[1].skew(state[2])
    return state[1].integrated(state[2], state[3])


# ------------------------------------------------------- what a pass cannot do without
def _fft_flops(n, fields):
    return 2.5 * n ** 3 * math.log2(n ** 3) * fields


def _bin_count(case):
    """Bins (a >= b >= c) that can hold a triangle, or with every leg their (a; b >= c)."""
    e = _edges(case) if "width" in case else [1.0 + i for i in range(case["shells"] + 1)]
    k = 0
    for a in range(case["shells"]):
        for b in range(a + 1):
            for c in range(b + 1):
                if e[a] < e[b + 1] + e[c + 1] or e[a + 1] + e[b + 1] + e[c + 1] > case.get("n", 1 << 30):
                    k += len({a, b, c}) if case.get("full") else 1
    return k


def work(case):
    kind, half = case["kind"], lambda n: 8 * n * n * (n // 2 + 1)
    if kind == "bispec":
        n, ne, nb = case["n"], len(_ells(case)), _bin_count(case)
        fields = case["shells"] * (ne + (1 if 0 not in _ells(case) else 0))
        if case["shot"]:   # the power fields and unit fields, and the sums over their pairs
            fields, ne = 3 * fields, 4 * ne
        return {"bytes": half(n) + 8 * nb * len(_ells(case)), "flops": _fft_flops(n, fields) + 2.0 * n ** 3 * nb * ne}
    if kind == "modal":
        n, p, ells = case["n"], case["modes"], _ells(case)
        trip = p * (p + 1) * (p + 2) // 6
        sums = sum({0: 1, 2: 3, 4: 6}[l] for l in ells) * trip
        return {"bytes": half(n) + 8 * trip * len(ells), "flops": _fft_flops(n, p * len(ells)) + 2.0 * n ** 3 * sums}
    if kind == "batch":
        ne, nb = len(_ells(case)), _bin_count(case)
        got = {"bytes": 0.0, "flops": 0.0}
        for m in range(case["mocks"]):
            n = _SIZES[m % 3]
            got["bytes"] += half(n) + 8 * nb * ne
            got["flops"] += _fft_flops(n, case["shells"] * ne) + 2.0 * n ** 3 * nb * ne
        return got
    if kind == "cov":
        m, d = case["mocks"], case["dim"]
        return {"bytes": 8 * (m * d + d * d + d), "flops": 1.0 * m * d * d}
    if kind == "density":
        n, p = case["n"], case["particles"]
        return {"bytes": 12 * p + half(n), "flops": 2 * _fft_flops(n, 1) + 16.0 * 6 * p}
    n = case["n"]
    out = 8 * case["shells"] * (len(_ells(case)) + 1)
    return {"bytes": half(n) + out, "flops": 2 * _fft_flops(n, 1) + 10.0 * n ** 3}


# --------------------------------------------------------------- FP64 values
def _weight(l, n2, fz2):
    mu2 = fz2.to(F64) / n2.clamp_min(1).to(F64)
    if l == 0:
        return torch.ones_like(mu2)
    return 2.5 * (3 * mu2 - 1) if l == 2 else 1.125 * ((35 * mu2 - 30) * mu2 + 3)


def _shells64(n, edges, scale=1):
    """Shell of each mode of the half spectrum (-1: none), |n|^2 scaled."""
    n2 = _n2(n)[0].to(F64) * scale
    sq = torch.tensor([e * e for e in edges], dtype=F64, device="cuda")
    s = torch.bucketize(n2, sq, right=True) - 1
    return torch.where((s >= 0) & (s < len(edges) - 1), s, torch.full_like(s, -1))


def _real(spec, n):
    return torch.fft.irfftn(spec, s=(n, n, n)).flatten() * n ** 3


def _hermitian(d, n):
    """The half spectrum with only the Hermitian part on the n_z = 0 and n/2 planes."""
    d = d.to(torch.complex128)
    neg = (-torch.arange(n, device="cuda")) % n
    for z in (0, n // 2):
        p = d[:, :, z]
        d[:, :, z] = 0.5 * (p + p[neg][:, neg].conj())
    return d


def _shell_fields(spec, n, edges, l, shell):
    n2, fz2 = _n2(n)
    w = _weight(l, n2, fz2) * spec
    del n2
    out = torch.empty((len(edges) - 1, n ** 3), dtype=F64, device="cuda")
    for a in range(len(edges) - 1):
        out[a] = _real(torch.where(shell == a, w, torch.zeros((), dtype=w.dtype, device="cuda")).to(torch.complex128), n)
    return out


def _triple(rows, X, Y, sorted_only, sym=False):
    """T[r][b][c] = sum_x rows_r X_b Y_c (+ X_c Y_b) for b >= c; rows: per multipole [shells][points]; with
    sorted_only just the rows r >= b."""
    ns, npts = X.shape
    T = torch.zeros((len(rows), rows[0].shape[0], ns, ns), dtype=F64, device="cuda")
    L, C = 4096, 256
    for x0 in range(0, npts, L * C):
        x1 = min(npts, x0 + L * C)
        cut = (x1 - x0) // L if (x1 - x0) % L == 0 else 1

        def part(v):
            return v[:, x0:x1].reshape(v.shape[0], cut, -1).transpose(0, 1)

        R, Xp, Yp = [part(r) for r in rows], part(X), part(Y)
        for b in range(ns):
            P = Xp[:, b:b + 1] * Yp[:, :b + 1]
            if sym:
                P = P + Yp[:, b:b + 1] * Xp[:, :b + 1]
            lo = b if sorted_only else 0
            for i, r in enumerate(R):
                T[i, lo:, b, :b + 1] += torch.bmm(r[:, lo:], P.transpose(1, 2)).sum(0)
    return T


def _bins64(n, edges, full):
    """The valid bins (a, b, c) and their counts, from FP64 unit fields."""
    unit = _shell_fields(1.0, n, edges, 0, _shells64(n, edges))
    N = torch.round(_triple([unit], unit, unit, True)[0] / n ** 3).cpu()
    del unit
    ns, got = len(edges) - 1, {}
    for a in range(ns):
        for b in range(a + 1):
            for c in range(b + 1):
                if N[a, b, c] >= 1:
                    for u, v, w in ((a, b, c), (b, a, c), (c, a, b)) if full else ((a, b, c),):
                        got[u, v, w] = float(N[a, b, c])
    abc = sorted(got)
    return torch.tensor(abc, device="cuda").reshape(-1, 3), torch.tensor([got[t] for t in abc], dtype=F64, device="cuda")


def _bispectrum64(dk, n, edges, ells, nbar=0.0, full=False, bins=None):
    V, n3 = BOX ** 3, n ** 3
    shell = _shells64(n, edges)
    abc, N = bins or _bins64(n, edges, full)
    pick = lambda T: T[:, abc[:, 0], abc[:, 1], abc[:, 2]]  # noqa: E731
    d = dk.to(torch.complex128)
    F0 = _shell_fields(d, n, edges, 0, shell)
    out = []
    for l in ells:
        out.append(pick(_triple([F0 if l == 0 else _shell_fields(d, n, edges, l, shell)], F0, F0, not full)) / V)
    B = torch.cat(out)
    if nbar:
        del F0
        p = _hermitian(dk, n)
        p = p.real ** 2 + p.imag ** 2
        unit, pw = _shell_fields(1.0, n, edges, 0, shell), _shell_fields(p, n, edges, 0, shell)
        for i, l in enumerate(ells):
            S = pw if l == 0 else _shell_fields(p, n, edges, l, shell)
            W = unit if l == 0 else _shell_fields(1.0, n, edges, l, shell)
            T_s, T_w = pick(_triple([S], unit, unit, not full)), pick(_triple([W], unit, unit, not full))
            T_si = pick(_triple([W], pw, unit, not full, sym=True))
            B[i] -= ((T_s + T_si) / (V * nbar) - 2.0 * T_w / nbar ** 2)[0]
    return B / (n3 * N)


def _modal64(case, seed):
    n, ells, nf = case["n"], _ells(case), case["modes"]
    dk = _field(n, seed).to(torch.complex128)
    n2, fz2 = _n2(n)
    kf, kmin, kmax = 2 * math.pi / BOX, 2 * math.pi / BOX, _modal_kmax(case)
    k = kf * n2.to(F64).sqrt()
    t = 2.0 * (k - kmin) / (kmax - kmin) - 1.0
    live = (n2 > 0) & (k >= kmin) & (k <= kmax)
    den = torch.where(live, (k * 2.0e4 * k.clamp_min(kf).pow(-1.5)).sqrt(), torch.ones((), dtype=F64, device="cuda"))
    M = {}
    for l in set(ells) | {0} | ({2} if 4 in ells else set()):
        w = torch.where(live, _weight(l, n2, fz2) / den, torch.zeros((), dtype=F64, device="cuda")) * dk
        M[l] = torch.empty((nf, n ** 3), dtype=F64, device="cuda")
        p0, p1 = torch.ones_like(t), t.clone()
        for j in range(nf):
            M[l][j] = _real(p0 * w, n)
            p0, p1 = p1, ((2 * j + 3) * t * p1 - (j + 1) * p0) / (j + 2)
    del n2, k, t, live, den, w, p0, p1
    trip = torch.combinations(torch.arange(nf, device="cuda"), 3, with_replacement=True)
    p, q, r = trip[:, 0], trip[:, 1], trip[:, 2]
    out = []
    for l in ells:
        T = _triple([M[l]], M[0], M[0], l == 0)[0]
        v = T[r, q, p]
        if l:
            v = v + T[p, r, q] + T[q, r, p]
        if l == 4:
            U = _triple([M[0]], M[2], M[2], False)[0]
            v = v + U[r, q, p] + U[p, r, q] + U[q, r, p]
        out.append(v / (n ** 3 * BOX ** 9))
    return torch.stack(out)


def _shell_sums64(prod, n, edges, ells, scale=1):
    """sum over the full grid's modes of w_l * prod per shell, and the mode counts, from the half spectrum."""
    n2, fz2 = _n2(n)
    s = _shells64(n, edges, scale)
    h = torch.full((n // 2 + 1,), 2.0, dtype=F64, device="cuda")
    h[0] = h[n // 2] = 1.0
    idx = torch.where(s < 0, torch.full_like(s, len(edges) - 1), s)
    h = h.expand(idx.shape)

    def total(v):
        return torch.zeros(len(edges), dtype=F64, device="cuda").scatter_add_(0, idx.flatten(), v.flatten())[:-1]

    return torch.stack([total(h * _weight(l, n2, fz2) * prod) for l in ells]), total(h)


def _skew64(case, seed):
    n, V = case["n"], BOX ** 3
    d = _hermitian(_field(n, seed), n)
    d[0, 0, 0] = 0
    Q = torch.fft.rfftn((torch.fft.irfftn(d, s=(n, n, n)) * (n ** 3 / V)) ** 2) * (V / n ** 3)
    P, N = _shell_sums64((Q.conj() * d).real, n, _edges(case), _ells(case))
    return torch.where(N > 0, P / (V * N), torch.zeros_like(P)), N


def _ib64(case, seed):
    n, m, V = case["n"], case["m"], BOX ** 3
    s, nc = n // m, m ** 3
    d = _field(n, seed).to(torch.complex128)
    d[0, 0, 0] = 0
    x = torch.fft.irfftn(d, s=(n, n, n)) * (n ** 3 / V)
    x = x.reshape(m, s, m, s, m, s).permute(0, 2, 4, 1, 3, 5).reshape(nc, s, s, s)
    prod = torch.zeros((s, s, s // 2 + 1), dtype=F64, device="cuda")
    for c in x:
        T = torch.fft.rfftn(c) / s ** 3
        prod += T[0, 0, 0].real * (T.real ** 2 + T.imag ** 2)
    Vs = V / nc
    P, N = _shell_sums64(prod * Vs, s, _edges(case), _ells(case), m * m)
    return torch.where(N > 0, P / (nc * N.clamp_min(1)), torch.zeros_like(P)), N


def _density64(case, seed):
    n, pos = case["n"], _catalogue(case, seed).to(F64)
    half = []
    for shift in (0.0, 0.5):
        u = (pos * (n / BOX) - shift) % n
        b = u.floor()
        t, b = u - b, b.long() % n
        g = torch.zeros(n ** 3, dtype=F64, device="cuda")
        for o in range(8):
            bit = [(o >> 2) & 1, (o >> 1) & 1, o & 1]
            w = torch.ones(pos.shape[0], dtype=F64, device="cuda")
            i = torch.zeros(pos.shape[0], dtype=torch.long, device="cuda")
            for a in range(3):
                w = w * (t[:, a] if bit[a] else 1.0 - t[:, a])
                i = i * n + (b[:, a] + bit[a]) % n
            g.index_add_(0, i, w)
        half.append(torch.fft.rfftn((g * (n ** 3 / pos.shape[0]) - 1.0).reshape(n, n, n)))
    f = _freqs(n).to(F64)
    fz = torch.arange(n // 2 + 1, device="cuda").to(F64)
    fz[n // 2] = -(n // 2)
    phase = torch.exp(-1j * math.pi * (f[:, None, None] + f[None, :, None] + fz[None, None, :]) / n)
    w = [torch.sinc(v / n) ** 2 for v in (f, fz)]
    win = w[0][:, None, None] * w[0][None, :, None] * w[1][None, None, :]
    return (half[0] + phase * half[1]) * (0.5 * BOX ** 3 / n ** 3) / win, pos.shape[0] / BOX ** 3


def exact(case, seed):
    kind = case["kind"]
    if kind == "bispec":
        n = case["n"]
        dk, nbar = _sampled(n, seed) if case["shot"] else (_field(n, seed, sigma=case["sigma"]), 0.0)
        return _bispectrum64(dk, n, _edges(case), _ells(case), nbar, case["full"])
    if kind == "modal":
        return _modal64(case, seed)
    if kind == "batch":
        edges = [1.0 + i for i in range(case["shells"] + 1)]
        bins = _bins64(_SIZES[0], edges, False)   # the same bins and counts on every grid: none of them wraps
        return torch.stack([_bispectrum64(_field(_SIZES[i], s, n_s, f), _SIZES[i], edges, _ells(case), bins=bins).flatten()
                            for i, s, n_s, f in _mock_models(case, seed)])
    if kind == "cov":
        x = _mock_rows(case, seed)
        mean = x.mean(0)
        return mean, (x - mean).T @ (x - mean) / (x.shape[0] - 1)
    if kind == "density":
        return _density64(case, seed)
    return _skew64(case, seed) if kind == "skew" else _ib64(case, seed)
