"""The calls whose speed is measured: what a user of the library has it do.

Every case is one call, or one driver step, through the public entry points
(``api.Context``, ``posterior.KDEPosterior``) on synthetic windows: analytic
A/E/T noise, one to four injected binaries per window and a batch of
candidates.  A case's dict fixes all shapes (windows, template lengths,
candidates per window); the seed draws the sources, the noise and the
candidates.

Fields of a case:
  kind     loglik | phase | grad | certified | waveform | snr | generation | ladder
  prec     "fp64" or "mixed"
  chan     "AE", or "AET" (T joins A and E in the windows above f*/2)
  n_win    windows; their centres are log-spaced over [f_lo, f_hi] Hz
  lo, hi   candidates per window, uniform in [lo, hi] (ladder, certified and
           generation: lo = hi; snr: sources per window)
  years    observation time
  N        template samples per window (0: by frequency band, 32 ... 1024; -1: the posterior
           configuration's 128 below 3.6 mHz and 256 above)
  wide     window bins: wide * N + extra (extra may be negative)
  spread   how the candidates lie: "box" around a source (a search's
           population near an optimum), "gauss" (proposals of a posterior,
           ten widths ~1/SNR wide), "prior" (a search's first population)
"""
import math

import numpy as np
import torch

from paper_2307_03763_gb300 import api, posterior
from paper_2307_03763_gb300 import workloads as wk

C = 299792458.0
AU = 1.495978707e11
YEAR = 31557600.0
ARM = 2.5e9
FSTAR = C / (2.0 * math.pi * ARM)
PI = math.pi


def _case(kind, name=None, prec="mixed", chan="AE", n_win=1, lo=1, hi=None, f_lo=1e-3, f_hi=None, years=2.0, N=0,
          wide=1, extra=0, spread="box"):
    c = {"kind": kind, "prec": prec, "chan": chan, "n_win": n_win, "lo": lo, "hi": lo if hi is None else hi,
         "f_lo": f_lo, "f_hi": f_lo if f_hi is None else f_hi, "years": years, "N": N, "wide": wide,
         "extra": extra, "spread": spread}
    if name:
        c["name"] = name
    return c


def listed():
    return [
        # a first look at one window: 1,000 candidates near a source; launch latency counts
        _case("loglik", "loglik_mixed_one_window", lo=1000, f_lo=1.5e-3, N=128),
        # the headline: a 10,000-proposal posterior round of 16 sources, chains certified equal to FP64's
        _case("certified", "posterior_round", n_win=16, lo=10000, f_lo=0.5e-3, f_hi=5e-3, N=-1,
              spread="gauss"),
        # a whole search band in one call: every template length, ragged populations
        _case("loglik", "loglik_mixed_band", n_win=512, lo=2000, hi=20000, f_lo=0.3e-3, f_hi=20e-3, years=1.0),
        # the band above f*/2, where T joins A and E
        _case("loglik", "loglik_mixed_aet", chan="AET", n_win=40, lo=2000, hi=20000, f_lo=9.8e-3, f_hi=20e-3,
              years=1.0),
        # one generation of the genetic search over a stretch of Alg. 1 windows: phase-maximised likelihood of
        # the populations, gradient at each window's best, selection and mutation
        _case("generation", "search_generation", n_win=1200, lo=1024, f_lo=1e-3, f_hi=8e-3, spread="prior"),
        # gradients of a whole population
        _case("grad", "grad_mixed_population", n_win=64, lo=4096, f_lo=2e-3, f_hi=6.5e-3, N=256, spread="prior"),
        # the 16 gradients around each window's optimum that a Fisher matrix or a Newton polish takes
        _case("grad", "grad_mixed_fisher", n_win=2048, lo=16, f_lo=0.4e-3, f_hi=12e-3, spread="gauss"),
        # the plain double-precision likelihood of a posterior round
        _case("loglik", "loglik_fp64_posterior", prec="fp64", n_win=16, lo=10000, f_lo=0.5e-3, f_hi=5e-3, N=-1,
              spread="gauss"),
        # double-precision gradients (autograd, Fisher matrices)
        _case("grad", "grad_fp64_population", prec="fp64", n_win=64, lo=512, f_lo=2e-3, f_hi=6.5e-3, N=256,
              spread="prior"),
        # templates of found signals, to be added to or subtracted from the data
        _case("waveform", "waveform_fp64", prec="fp64", lo=8192, f_lo=3e-3, f_hi=5e-3, N=256),
        # match metrics of recoveries against injections: 2 x 2 Gram matrices over 2N-bin windows
        _case("snr", "snr_pairs", prec="fp64", n_win=4096, lo=2, f_lo=0.5e-3, f_hi=6e-3, wide=2),
        # the annealed posterior of Alg. 4 (six temperatures, KDE proposals) of 16 sources, replayed
        _case("ladder", "posterior_ladder", n_win=16, lo=10000, f_lo=0.5e-3, f_hi=5e-3, N=-1,
              spread="gauss"),
    ]


def _log(rng, a, b):
    return math.exp(rng.uniform(math.log(a), math.log(b)))


def draw(rng):
    """One more call of the same ranges: any kind, any size up to the listed one, odd sizes as a rule."""
    kind = rng.choice(["loglik", "loglik", "loglik64", "aet", "phase", "grad", "grad64", "certified", "waveform",
                       "snr", "generation", "ladder"])
    n = lambda a, b: int(_log(rng, a, b))  # noqa: E731
    fa, fb = _log(rng, 0.3e-3, 2e-3), _log(rng, 2e-3, 12e-3)
    years = rng.choice([0.5, 1.0, 2.0])
    extra = rng.choice([0, 0, -7, 13, 100])
    spread = rng.choice(["box", "gauss", "prior"])
    if kind == "loglik":
        lo = n(1, 3000)
        return _case("loglik", n_win=n(1, 400), lo=lo, hi=lo + n(1, 4000), f_lo=fa, f_hi=fb, years=years,
                     extra=extra, spread=spread)
    if kind == "loglik64":
        lo = n(1, 4000)
        return _case("loglik", prec="fp64", chan=rng.choice(["AE", "AE", "AET"]), n_win=n(1, 12), lo=lo,
                     hi=lo + n(1, 2000), f_lo=fa, f_hi=_log(rng, 2e-3, 6e-3), years=years, extra=extra, spread=spread)
    if kind == "aet":
        lo = n(16, 4000)
        return _case("loglik", chan="AET", n_win=n(1, 32), lo=lo, hi=lo + n(1, 4000),
                     f_lo=_log(rng, 8e-3, 11e-3), f_hi=_log(rng, 11e-3, 18e-3), years=rng.choice([0.5, 1.0]),
                     extra=extra, spread=spread)
    if kind == "phase":
        return _case("phase", n_win=n(1, 400), lo=n(64, 1500), f_lo=fa, f_hi=_log(rng, 2e-3, 8e-3), years=years,
                     extra=extra, spread="prior")
    if kind == "grad":
        lo = n(1, 3000)
        return _case("grad", n_win=n(1, 64), lo=lo, hi=lo + n(1, 200), f_lo=fa, f_hi=_log(rng, 2e-3, 8e-3),
                     years=years, extra=extra, spread=spread)
    if kind == "grad64":
        lo = n(1, 300)
        return _case("grad", prec="fp64", n_win=n(1, 40), lo=lo, hi=lo + n(1, 100), f_lo=fa,
                     f_hi=_log(rng, 2e-3, 5e-3), years=years, extra=extra, spread=spread)
    if kind == "certified":
        return _case("certified", n_win=n(1, 16), lo=n(300, 10000), f_lo=fa, f_hi=_log(rng, 2e-3, 5e-3), years=years,
                     N=-1, extra=rng.choice([0, 13]), spread="gauss")
    if kind == "waveform":
        N = rng.choice([32, 64, 128, 256, 512, 1024])
        f = {32: 0.4e-3, 64: 1e-3, 128: 2e-3, 256: 4e-3, 512: 7e-3, 1024: 1.2e-2}[N]
        return _case("waveform", prec=rng.choice(["fp64", "fp64", "mixed"]), chan=rng.choice(["AE", "AE", "AET"]),
                     lo=n(1, 8192 * 256 // N), f_lo=f, f_hi=1.5 * f, N=N)
    if kind == "snr":
        lo = rng.choice([1, 2, 3, 5])
        return _case("snr", prec="fp64", n_win=n(1, 8192 // (lo * (lo + 1))), lo=lo, hi=lo + rng.choice([0, 1]),
                     f_lo=fa, f_hi=_log(rng, 2e-3, 6e-3), years=years, wide=rng.choice([1, 2]), extra=rng.choice([0, 13]))
    if kind == "generation":
        return _case("generation", n_win=n(1, 800), lo=n(64, 1500), f_lo=fa, f_hi=_log(rng, 2e-3, 6e-3),
                     years=years, spread="prior")
    return _case("ladder", n_win=n(1, 16), lo=n(500, 10000), f_lo=fa, f_hi=_log(rng, 2e-3, 5e-3), years=years,
                 N=-1, spread="gauss")


# ---------------------------------------------------------------------------
# layouts: a case's windows, from the case alone
# ---------------------------------------------------------------------------

def _shapes(c):
    """[(centre frequency, W, N, candidates)] of the case's windows."""
    n = c["n_win"]
    f = np.exp(np.linspace(math.log(c["f_lo"]), math.log(max(c["f_hi"], c["f_lo"])), n)) if n > 1 else [c["f_lo"]]
    rng = np.random.default_rng([n, c["lo"], c["hi"], int(c["f_lo"] * 1e9), int(c["f_hi"] * 1e9)])
    counts = rng.integers(c["lo"], c["hi"] + 1, n)
    out = []
    for fc, k in zip(f, counts):
        if c["N"] > 0:
            N = c["N"]
        elif c["N"] < 0:
            N = 128 if fc < 3.6e-3 else 256
        else:
            N = min(max(wk.n_for_band(float(fc), c["years"] * YEAR), 32), 1024)
        out.append((float(fc), c["wide"] * N + c["extra"], N, int(k)))
    return out


def _flops(c, N):
    """Per candidate: response samples, transforms, window sums; the reverse pass of a gradient."""
    ch = 3 if c["chan"] == "AET" else 2
    fwd = N * 560 + 5 * ch * N * math.log2(N) + 13 * ch * N
    return fwd + (N * 1150 + 5 * ch * N * math.log2(N) if c["kind"] == "grad" else 0)


def work(case):
    c = case
    ch = 3 if c["chan"] == "AET" else 2
    fl = by = 0.0
    for _, W, N, k in _shapes(c):
        kind = c["kind"]
        reps = 6 if kind == "ladder" else 1
        fl += reps * k * _flops(c, N)
        by += ch * 24 * W
        if kind == "snr":
            fl += k * (k + 1) / 2 * 16 * W
            by += 64 * k + 8 * k * k
        elif kind == "waveform":
            by += k * (64 + 16 * ch * N + 8)
        elif kind == "grad":
            by += k * (64 + 8 + 64)
        elif kind == "certified":
            by += k * (64 + 16 + 24 + 4)
        elif kind == "generation":
            fl += N * 1150
            by += k * (64 + 32 + 64)
        elif kind == "ladder":
            by += k * (64 + 8 + 4)
        else:
            by += k * (64 + 24 + (8 if kind == "phase" else 0))
    return {"bytes": by, "flops": fl}


# ---------------------------------------------------------------------------
# the model in plain torch, 64 bits: data for the inputs, and exact()
# ---------------------------------------------------------------------------

def _template(th, N, T):
    """Carrier bins and the A, E, T templates on bins q - N/2 ... q + N/2 - 1 of the rows th."""
    dev = th.device
    f0, fd, be, la, A, io, ps, ph = (x[:, None] for x in th.unbind(1))
    f0T = f0 * T
    q = torch.floor((f0T + ((0.5 * fd) * T) * T) + 0.5).detach()
    delta = f0T - q
    n = torch.arange(N, device=dev, dtype=torch.float64)
    t = n * (T / N)
    a = 2.0 * PI * t / YEAR
    ecc = ARM / (2.0 * math.sqrt(3.0) * AU)
    x = []
    for i in range(3):
        b = 2.0 * PI * i / 3.0
        x.append((AU * torch.cos(a) + 0.5 * AU * ecc * (torch.cos(2.0 * a - b) - 3.0 * math.cos(b)),
                  AU * torch.sin(a) + 0.5 * AU * ecc * (torch.sin(2.0 * a - b) - 3.0 * math.sin(b)),
                  -math.sqrt(3.0) * AU * ecc * torch.cos(a - b)))
    sb, cb, sl, cl = torch.sin(be), torch.cos(be), torch.sin(la), torch.cos(la)
    k = (-cb * cl, -cb * sl, -sb)
    u = (sb * cl, sb * sl, -cb)
    v = (sl, -cl)
    c2, s2, ci = torch.cos(2.0 * ps), torch.sin(2.0 * ps), torch.cos(io)
    Ap, Ax = A * (1.0 + ci * ci), -2.0 * A * ci
    rx = []
    for i in range(3):
        kap = (k[0] * x[i][0] + k[1] * x[i][1] + k[2] * x[i][2]) / C
        cyc = delta * (n / N) + 0.5 * fd * t * t - f0 * kap - fd * t * kap + 0.5 * fd * kap * kap
        rx.append(torch.polar(torch.ones_like(cyc), 2.0 * PI * (cyc - torch.round(cyc).detach()) + ph))
    f = f0 + fd * t
    h = f / (2.0 * FSTAR)
    z = {}
    for i, j in ((0, 1), (1, 2), (2, 0)):
        d = [x[j][m] - x[i][m] for m in range(3)]
        r = torch.sqrt(d[0] ** 2 + d[1] ** 2 + d[2] ** 2)
        d = [y / r for y in d]
        kn = k[0] * d[0] + k[1] * d[1] + k[2] * d[2]
        nu = u[0] * d[0] + u[1] * d[1] + u[2] * d[2]
        nv = v[0] * d[0] + v[1] * d[1]
        Fp, Fx = nu * nu - nv * nv, 2.0 * nu * nv
        G = torch.complex(Ap * (c2 * Fp - s2 * Fx), -Ax * (s2 * Fp + c2 * Fx))
        for (p, c), sg in (((i, j), -1.0), ((j, i), 1.0)):
            X = h * (1.0 + sg * kn)
            z[(p, c)] = torch.complex(torch.zeros_like(X), -h * torch.sinc(X / PI)) * torch.polar(
                torch.ones_like(X), -X) * G * rx[c]
    D = torch.polar(torch.ones_like(f), -f / FSTAR)
    om = 1.0 - D * D
    XYZ = [om * ((z[(p, c)] + D * z[(c, p)]) - (z[(r, c)] + D * z[(c, r)]))
           for c, p, r in ((0, 1, 2), (1, 2, 0), (2, 0, 1))]
    s = ((XYZ[2] - XYZ[0]) / math.sqrt(2.0), (XYZ[0] - 2.0 * XYZ[1] + XYZ[2]) / math.sqrt(6.0),
         (XYZ[0] + XYZ[1] + XYZ[2]) / math.sqrt(3.0))
    sc = T / (2.0 * N)
    return q[:, 0].to(torch.int64), [sc * torch.fft.fftshift(torch.fft.fft(y), dim=1) for y in s]


def _groups(wins, dev, chunk):
    """Candidate rows with their windows, in chunks of one template length: (N, rows, window values)."""
    W = torch.tensor([[w[0], w[1], w[3]] for w in wins], device=dev)
    for N in sorted({w[2] for w in wins}):
        sel = [i for i, w in enumerate(wins) if w[2] == N and w[5] > 0]
        if not sel:
            continue
        rows = torch.cat([torch.arange(wins[i][4], wins[i][4] + wins[i][5], device=dev) for i in sel])
        own = torch.repeat_interleave(torch.tensor(sel, device=dev),
                                      torch.tensor([wins[i][5] for i in sel], device=dev))
        step = max(1, chunk // N)
        for c in range(0, rows.numel(), step):
            yield N, rows[c:c + step], own[c:c + step], W[own[c:c + step]]


def _on_window(q, N, w):
    """Index of every template bin in the data arrays, and whether it is inside the window."""
    j = q[:, None] - N // 2 + torch.arange(N, device=q.device)[None, :] - w[:, 0:1]
    ok = (j >= 0) & (j < w[:, 1:2])
    return (w[:, 2:3] + j.clamp(min=0)).clamp(max=int((w[:, 1] + w[:, 2]).max()) - 1), ok


def _uses(k0, T, n_ch):
    return [True, True] + [k0 / T >= 0.5 * FSTAR] * (n_ch - 2)


def _loglik64(s, theta, grad=False, chunk=1 << 21):
    """logL, <d|h>, Im <d|h>, <h|h> (and with grad d logL/d theta) of every row."""
    T, wins, data, wts = s["T"], s["wins"], s["data"], s["weights"]
    dev = theta.device
    out = torch.zeros((4, theta.shape[0]), dtype=torch.float64, device=dev)
    g = torch.zeros_like(theta)
    dd = torch.zeros(len(wins), dtype=torch.float64, device=dev)
    use = torch.tensor([_uses(w[0], T, len(data)) for w in wins], device=dev)
    for i, w in enumerate(wins):
        for c in range(len(data)):
            if c < 2 or w[0] / T >= 0.5 * FSTAR:
                sl = slice(w[3], w[3] + w[1])
                dd[i] += (wts[c][sl] * (data[c][sl].real ** 2 + data[c][sl].imag ** 2)).sum()
    for N, rows, own, w in _groups(wins, dev, chunk // 4 if grad else chunk):
        th = theta[rows].clone().requires_grad_(grad)
        with torch.set_grad_enabled(grad):
            q, h = _template(th, N, T)
            idx, ok = _on_window(q, N, w)
            zdh, hh = 0.0, 0.0
            for c in range(len(data)):
                m = (ok & use[own, c][:, None]).to(torch.float64) * wts[c][idx]
                zdh = zdh + (m * (data[c][idx] * h[c].conj())).sum(1)
                hh = hh + (m * (h[c].real ** 2 + h[c].imag ** 2)).sum(1)
            zdh, hh = (4.0 / T) * zdh, (4.0 / T) * hh
            logL = zdh.real - 0.5 * hh - 0.5 * (4.0 / T) * dd[own]
            if grad:
                g[rows] = torch.autograd.grad(logL.sum(), th)[0]
        out[:, rows] = torch.stack([logL.detach(), zdh.real.detach(), zdh.imag.detach(), hh.detach()])
    return out, g


# ---------------------------------------------------------------------------
# inputs
# ---------------------------------------------------------------------------

def _psd(f, c):
    return wk.psd_T(f) if c == 2 else wk.psd_AE(f)


def _sources(gen, f, T, dev):
    """One random binary per frequency (amplitude 1), chirping by Eq. 8."""
    n = f.numel()
    r = torch.rand((n, 6), generator=gen, device=dev, dtype=torch.float64)
    m = (0.2 + 0.8 * r[:, 0]) * wk.G_MSUN_S
    fd = 96.0 / 5.0 * PI ** (8.0 / 3.0) * m ** (5.0 / 3.0) * f ** (11.0 / 3.0)
    return torch.stack([f - 0.5 * fd * T, fd, torch.asin(2 * r[:, 1] - 1), PI * (2 * r[:, 2] - 1),
                        torch.ones_like(f), torch.acos(2 * r[:, 3] - 1), PI * r[:, 4], 2 * PI * r[:, 5]], 1)


def prepare(case, seed):
    c = dict(case)
    dev = torch.device("cuda", torch.cuda.current_device())
    gen = torch.Generator(device=dev)
    gen.manual_seed(int(seed))
    T = c["years"] * YEAR
    ctx = api.Context(T)
    shapes = _shapes(c)
    s = {"case": c, "ctx": ctx, "T": T}
    rand = lambda *n: torch.rand(n, generator=gen, device=dev, dtype=torch.float64)  # noqa: E731
    normal = lambda *n: torch.randn(n, generator=gen, device=dev, dtype=torch.float64)  # noqa: E731
    if c["kind"] == "waveform":
        n = shapes[0][3]
        th = _sources(gen, c["f_lo"] * (c["f_hi"] / c["f_lo"]) ** rand(n), T, dev)
        th[:, 4] = 10.0 ** (-23.0 + 2.0 * rand(n))
        s.update(theta=th.contiguous(), N=shapes[0][2])
        return s
    # windows and their data: noise and one to four sources each
    wins, off, coff = [], 0, 0
    for fc, W, N, k in shapes:
        wins.append((int(round(fc * T)) - W // 2, W, N, off, coff, k))
        off += W
        coff += k
    s["wins"] = wins
    f = torch.cat([torch.arange(w[0], w[0] + w[1], device=dev, dtype=torch.float64) for w in wins]).clamp(min=1.0) / T
    fh = f.cpu().numpy()
    n_ch = 3 if c["chan"] == "AET" else 2
    psd = [torch.as_tensor(_psd(fh, ch), device=dev) for ch in range(n_ch)]
    s["weights"] = [1.0 / p for p in psd]
    s["data"] = [torch.sqrt(T * p / 4.0) * torch.complex(normal(off), normal(off)) for p in psd]
    nw = len(wins)
    w0 = torch.tensor([[w[0], w[1], w[3]] for w in wins], device=dev)
    fc = torch.tensor([(w[0] + 0.5 * w[1]) / T for w in wins], device=dev, dtype=torch.float64)
    Nw = torch.tensor([float(w[2]) for w in wins], device=dev, dtype=torch.float64)
    n_src = 1 if c["spread"] == "gauss" else 2
    snr = torch.exp(math.log(20.0) + math.log(10.0) * rand(n_src, nw))
    src = []
    for j in range(n_src):
        th = _sources(gen, fc + (0.3 * (rand(nw) - 0.5) * Nw) / T, T, dev)
        for N in sorted({w[2] for w in wins}):
            sel = torch.tensor([i for i, w in enumerate(wins) if w[2] == N], device=dev)
            q, h = _template(th[sel], N, T)
            idx, ok = _on_window(q, N, w0[sel])
            hh = sum(((4.0 / T) * ok * s["weights"][x][idx] * (h[x].real ** 2 + h[x].imag ** 2)).sum(1) for x in (0, 1))
            amp = snr[j, sel] / torch.sqrt(hh)
            th[sel, 4] = amp
            for x in range(n_ch):
                hx = torch.view_as_real(h[x] * amp[:, None])
                torch.view_as_real(s["data"][x]).index_add_(0, idx[ok], hx[ok])
        src.append(th)
    src = torch.stack(src)
    # candidates
    own = torch.repeat_interleave(torch.arange(nw, device=dev), torch.tensor([w[5] for w in wins], device=dev))
    n = own.numel()
    mid = src[torch.randint(n_src, (nw,), generator=gen, device=dev), torch.arange(nw, device=dev)]
    if c["kind"] == "snr":   # a recovery near an injection, then further sources of the window
        th = _sources(gen, fc[own] + (0.3 * (rand(n) - 0.5) * Nw[own]) / T, T, dev)
        th[:, 4] = mid[own, 4] * (0.5 + rand(n))
        s["theta"] = th.contiguous()
        return s
    lo, hi = torch.empty((nw, 8), dtype=torch.float64, device=dev), torch.empty((nw, 8), dtype=torch.float64, device=dev)
    lo[:] = torch.tensor([0, 0, -PI / 2, -PI, 1e-24, 0, 0, 0], device=dev)
    hi[:] = torch.tensor([0, 0, PI / 2, PI, 1e-20, PI, PI, 2 * PI], device=dev)
    fdm = 96.0 / 5.0 * PI ** (8.0 / 3.0) * wk.G_MSUN_S ** (5.0 / 3.0) * fc ** (11.0 / 3.0)
    hi[:, 1] = fdm
    lo[:, 0], hi[:, 0] = fc - 0.25 * Nw / T, fc + 0.25 * Nw / T
    lo[:, 4], hi[:, 4] = 0.1 * mid[:, 4], 10.0 * mid[:, 4]
    rho = snr[0]
    one = torch.ones_like(rho)
    width = torch.stack([0.3 / T / rho, 1.0 / T ** 2 / rho, 2.0 / rho, 2.0 / rho, mid[:, 4] / rho, 2.0 / rho,
                         2.0 / rho, 2.0 / rho], 1)
    width[:, 2:4] = torch.minimum(width[:, 2:4], 0.05 * one[:, None])
    width[:, 5:8] = torch.minimum(width[:, 5:8], 0.2 * one[:, None])
    width[:, 4] = torch.minimum(width[:, 4], 0.2 * mid[:, 4])
    if c["kind"] == "ladder":
        box = posterior.reduced_box(mid.cpu().numpy(), width.cpu().numpy(), lo.cpu().numpy(), hi.cpu().numpy())
        s["ladder"] = posterior.KDEPosterior(ctx, wins, s["data"][0], s["data"][1], s["weights"][0], s["weights"][1],
                                             box, n=wins[0][5], seed=int(seed) + 1, prec=c["prec"])
        return s
    if c["spread"] == "prior":
        th = lo[own] + (hi - lo)[own] * rand(n, 8)
    elif c["spread"] == "gauss":
        z = normal(n, 8)
        th = mid[own] + width[own] * z
        s["log_g"] = (-0.5 * (z * z).sum(1) - torch.log(width[own]).sum(1) - 4.0 * math.log(2.0 * PI)).reshape(nw, -1) \
            if c["kind"] == "certified" else None
    else:
        half = torch.stack([5.0 / T * one, 0.5 * mid[:, 1].abs() + 1e-20, 0.2 * one, 0.2 * one, 0.5 * mid[:, 4],
                            0.3 * one, 0.3 * one, 0.3 * one], 1)
        th = mid[own] + half[own] * (2.0 * rand(n, 8) - 1.0)
    th[:, 2] = th[:, 2].clamp(-PI / 2, PI / 2)
    s["theta"] = th.contiguous()
    if c["kind"] == "certified":
        s["log_u"] = torch.log(rand(nw, n // nw).clamp(min=1e-300))
        s["temperature"] = torch.ones(nw, dtype=torch.float64, device=dev)
    if c["kind"] == "generation":   # the buffers that the search keeps from one generation to the next
        z = lambda *k: torch.zeros(k, dtype=torch.float64, device=dev)  # noqa: E731
        s["box"] = torch.cat([lo, hi], 1).contiguous()
        s["best_in"] = mid.contiguous()
        s["best_wins"] = [(w[0], w[1], w[2], w[3], i, 1) for i, w in enumerate(wins)]
        s["out"] = (z(n), z(n), z(n), z(n))
        s["grad"], s["next"], s["best"] = z(nw, 8), z(n, 8), z(nw, 8)
        s["gen"] = torch.tensor([3, 0], dtype=torch.int64, device=dev)
        s["params"] = api.GAParams(3, 0, 0.9, 0.15, 0.02)
    return s


def run(s):
    c, ctx = s["case"], s["ctx"]
    kind, prec = c["kind"], c["prec"]
    if kind == "waveform":
        return (ctx.waveform_aet if c["chan"] == "AET" else ctx.waveform)(s["theta"], s["N"], prec)
    if kind == "ladder":
        k = s["ladder"].run(graph=True)
        return {"theta": k.theta, "log_g": k.log_g, "logL": k.logL, "chain": k.chain, "accepted": k.accepted,
                "cdf": k.cdf, "ext": k.ext}
    d, w, wins = s["data"], s["weights"], s["wins"]
    if kind == "snr":
        rho, gram, dh = ctx.snr_multi(wins, d[0], d[1], w[0], w[1], s["theta"])
        return {"rho": rho, "gram": gram, "dh": dh}
    if kind == "certified":
        return ctx.mh_certified(wins, d[0], d[1], w[0], w[1], s["theta"], s["log_g"], s["log_u"], s["temperature"])
    if kind == "generation":
        logL, dh, dh_im, hh = ctx.loglik_phase(wins, d[0], d[1], w[0], w[1], s["theta"], prec=prec, out=s["out"])
        ctx.loglik_grad(s["best_wins"], d[0], d[1], w[0], w[1], s["best_in"], prec=prec, out=(None, s["grad"]))
        ctx.ga_step(len(wins), c["lo"], s["theta"], dh, hh, s["box"], 7, s["gen"][0:1], s["gen"][1:2], s["params"],
                    s["grad"], out=s["next"], best=s["best"], dh_im=dh_im)
        return {"logL": logL, "dh": dh, "dh_im": dh_im, "hh": hh, "grad": s["grad"], "next": s["next"],
                "best": s["best"]}
    aet = len(d) == 3
    args = (wins, *d, *w, s["theta"])
    if kind == "phase":
        return ctx.loglik_phase(*args, prec=prec)
    if kind == "grad":
        return (ctx.loglik_grad_aet if aet else ctx.loglik_grad)(*args, prec=prec)
    return (ctx.loglik_aet if aet else ctx.loglik)(*args, prec=prec)


def exact(case, seed):
    kind = case["kind"]
    if kind == "ladder":   # its proposals are drawn by the sampler itself
        return None
    s = prepare(case, seed)
    if kind == "waveform":
        n_ch = 3 if case["chan"] == "AET" else 2
        parts = [_template(t, s["N"], s["T"]) for t in s["theta"].split(max(1, (1 << 21) // s["N"]))]
        return [torch.cat([p[1][ch] for p in parts]) for ch in range(n_ch)] + [torch.cat([p[0] for p in parts])]
    if kind == "snr":
        wins, wts, T = s["wins"], s["weights"], s["T"]
        dev = s["theta"].device
        kmax = max(w[5] for w in wins)
        out, _ = _loglik64(s, s["theta"])
        gram = torch.full((len(wins), kmax, kmax), float("nan"), dtype=torch.float64, device=dev)
        where = torch.full((len(wins), kmax), -1, device=dev)
        for i, w in enumerate(wins):
            where[i, :w[5]] = torch.arange(w[4], w[4] + w[5], device=dev)
        for N in sorted({w[2] for w in wins}):
            sel = torch.tensor([i for i, w in enumerate(wins) if w[2] == N], device=dev)
            wv = torch.tensor([[w[0], w[1], w[3]] for w in wins], device=dev)[sel]
            Wm = int(wv[:, 1].max())
            on = []   # every source's templates on its window's bins
            for a in range(kmax):
                q, h = _template(s["theta"][where[sel, a].clamp(min=0)], N, T)
                idx, ok = _on_window(q, N, wv)
                pos = (idx - wv[:, 2:3]).clamp(0, Wm)
                full = torch.zeros((2, sel.numel(), Wm + 1), dtype=torch.complex128, device=dev)
                for ch in (0, 1):
                    full[ch].scatter_(1, torch.where(ok, pos, Wm), h[ch] * ok)
                on.append(full[:, :, :Wm])
            at = (wv[:, 2:3] + torch.arange(Wm, device=dev)).clamp(max=wts[0].numel() - 1)
            inside = torch.arange(Wm, device=dev)[None, :] < wv[:, 1:2]
            for a in range(kmax):
                for b in range(kmax):
                    v = sum((inside * wts[ch][at] * (on[a][ch] * on[b][ch].conj()).real).sum(1) for ch in (0, 1))
                    have = (where[sel, a] >= 0) & (where[sel, b] >= 0)
                    gram[sel, a, b] = torch.where(have, (4.0 / T) * v, float("nan"))
        num = torch.stack([out[1][w[4]:w[4] + w[5]].sum() for w in wins])
        return {"rho": num / torch.sqrt(torch.nansum(gram, (1, 2))), "gram": gram, "dh": out[1]}
    if kind == "generation":
        out, _ = _loglik64(s, s["theta"])
        _, g = _loglik64(dict(s, wins=s["best_wins"]), s["best_in"], grad=True)
        return {"logL": out[0], "dh": out[1], "dh_im": out[2], "hh": out[3], "grad": g, "next": None, "best": None}
    out, g = _loglik64(s, s["theta"], grad=kind == "grad")
    if kind == "grad":
        return [out[0], g]
    if kind == "certified":
        return [None, None, out[0], out[1], out[3], None, None]
    return [out[0], out[1], out[2], out[3]] if kind == "phase" else [out[0], out[1], out[3]]
