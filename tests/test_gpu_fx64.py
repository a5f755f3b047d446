"""The FP64 path's fixed-point slow part and transform at the edges of its ranges.

Candidates on both sides of each range (series tiers at f_max/f* = 1/2 and
1.3, drift f0/1024, f0 <= 0) and every template length, against the model in
long double.  The tolerance is the rounding of phases in double: a handful of
roundings (8) of terms of the size of f0 k.x/c, fdot T^2/2 and phi0/2pi
cycles, times 2 pi, on top of 1e-14 for the response."""
import math

import numpy as np
import pytest
import torch

from oracle import gb
from paper_2307_03763_gb300 import api
from paper_2307_03763_gb300 import workloads as wk

from tests import _longdouble as ld

pytestmark = pytest.mark.gpu

FSTAR = gb.transfer_frequency()


def candidates(f0, fdot, n, seed):
    rng = np.random.default_rng(seed)
    th = np.empty((n, 8))
    th[:, 0] = f0
    th[:, 1] = fdot
    th[:, 2], th[:, 3], th[:, 5], th[:, 6], th[:, 7] = wk.random_angles(rng, n)
    th[:, 4] = np.exp(rng.uniform(math.log(1e-23), math.log(1e-21), n))
    th[0, 2], th[1 % n, 2] = math.pi / 2, -math.pi / 2
    return th


def tolerance(th, T):
    cycles = np.abs(th[:, 0]) * 510.0 + np.abs(0.5 * th[:, 1]) * T * T + np.abs(th[:, 7]) / (2 * math.pi) + 1.0
    return 8 * 2 * math.pi * 2.0 ** -53 * cycles + 1e-14


CASES = [(0.3e-3, 0.0, 32), (1e-3, 1e-18, 64), (0.4995 * FSTAR, 1e-15, 128), (0.5005 * FSTAR, 1e-15, 256),
         (1.299 * FSTAR, 2e-13, 512), (1.301 * FSTAR, 2e-13, 256), (2.0 * FSTAR, 0.0, 64), (3.0 * FSTAR, 0.0, 64),
         (15e-3, 1.2e-13, 1024), (20e-3, 9e-13, 1024), (5e-3, -3e-14, 128),
         (1e-3, 0.999e-3 / (1024 * wk.YEAR), 64), (1e-3, 1.001e-3 / (1024 * wk.YEAR), 64),
         (-2e-3, 1e-17, 64), (0.0, 0.0, 32)]


@pytest.mark.parametrize("f0,fdot,N", CASES)
def test_templates_at_range_edges(f0, fdot, N):
    T = wk.YEAR
    th = candidates(f0, fdot, 7, int(N))
    ctx = api.Context(T)
    out = ctx.waveform_aet(torch.as_tensor(th, device="cuda"), N)
    q, ref = ld.template_aet(th, N, T)
    assert np.array_equal(out[3].cpu().numpy(), q)
    tol = tolerance(th, T)
    norm = lambda x: np.sqrt((np.abs(x) ** 2).sum(1).astype(np.float64))  # noqa: E731
    for h, r in zip(out[:2], ref[:2]):
        assert np.all(norm(h.cpu().numpy() - r) <= tol * np.maximum(norm(r), 1e-300))
    # T is a small difference of terms of A's size in the plain form
    assert np.all(norm(out[2].cpu().numpy() - ref[2]) <= tol * np.maximum(norm(ref[0]) + norm(ref[1]), 1e-300))
    ctx.check()


@pytest.mark.parametrize("n", [1, 5, 16, 17, 127, 130])
def test_mixed_forms_in_one_call(n):
    """Fixed-point and plain-double candidates side by side, counts around a warp's set-up group."""
    T = 0.5 * wk.YEAR
    th = candidates(4e-3, 1e-15, n, n)
    th[::3, 0] = 1.4 * FSTAR       # plain double
    th[::3, 1] = 0.0
    N = 128
    wins = [(int(4e-3 * T) - 64, 128, N, 0, 0, n)]
    rng = np.random.default_rng(n)
    d = rng.standard_normal((2, 128, 2)) @ np.array([1, 1j])
    w = rng.uniform(0.5, 1.5, (2, 128)) * 1e41
    ctx = api.Context(T)
    dev = lambda x: torch.as_tensor(x, device="cuda")  # noqa: E731
    d = d * 1e-20
    args = [dev(np.ascontiguousarray(x)) for x in (d[0], d[1], w[0], w[1])]
    got = ctx.loglik(wins, *args, dev(th))
    ref = [np.asarray(x, dtype=np.float64) for x in ld.loglik(wins[0], d[0], d[1], w[0], w[1], th, T)]
    tol = tolerance(th, T)
    dd = -2.0 * float(ref[0][0]) if n > 0 else 0.0   # the first candidate lies outside the window: logL = -<d|d>/2
    for g, r in zip(got, ref):
        scale = np.abs(ref[2]) + np.sqrt(np.abs(ref[2]) * dd) + dd
        assert np.all(np.abs(g.cpu().numpy() - r) <= 2 * tol * scale)
    # the row list evaluates the same bits
    rows = torch.arange(n, dtype=torch.int32, device="cuda")
    lo, hi = torch.zeros(1, dtype=torch.int32, device="cuda"), torch.full((1,), n, dtype=torch.int32, device="cuda")
    again = ctx.loglik_rows(wins, *args, dev(th), rows, lo, hi)
    for a, b in zip(again, got):
        assert torch.equal(a, b)


@pytest.mark.parametrize("f0,fdot,N", [c for c in CASES if c[0] > 0 and c[2] <= 512])
@pytest.mark.parametrize("aet", [False, True])
def test_gradients_at_range_edges(f0, fdot, N, aet):
    """Against the oracle's autodiff to the repository's 1e-9 of the gradient's norm (natural units)."""
    T = 0.5 * wk.YEAR
    n = 5
    th = candidates(f0, fdot, n, N + 1)
    th[1, 0] *= 1.01               # outside the window: zero gradient
    qc = int(f0 * T + 0.5 * fdot * T * T)
    W = N + 9
    win = [(qc - W // 2, W, N, 0, 0, n)]
    rng = np.random.default_rng(N)
    d = [(rng.standard_normal(W) + 1j * rng.standard_normal(W)) * 1e-19 for _ in range(3)]
    w = [rng.uniform(0.5, 1.5, W) * 1e41 for _ in range(3)]
    dev = lambda x: torch.as_tensor(x, device="cuda")  # noqa: E731
    ctx = api.Context(T)
    if aet:
        logL, g = ctx.loglik_grad_aet(win, *[dev(x) for x in d], *[dev(x) for x in w], dev(th))
        ref_l, ref = gb.loglik_grad_aet(win, *d, *w, th, T)
    else:
        logL, g = ctx.loglik_grad(win, dev(d[0]), dev(d[1]), dev(w[0]), dev(w[1]), dev(th))
        ref_l, ref = gb.loglik_grad(win, d[0], d[1], w[0], w[1], th, T)
    scale = np.stack([np.full(n, 1 / T), np.full(n, 1 / T ** 2)] + [np.ones(n)] * 2 + [th[:, 4]] + [np.ones(n)] * 3, 1)
    g, ref = g.cpu().numpy() * scale, np.asarray(ref) * scale
    norm = np.linalg.norm(ref, axis=1)
    assert np.all(np.linalg.norm(g - ref, axis=1) <= 1e-9 * np.maximum(norm, 1e-300) + (norm == 0) * 1e-300)
    np.testing.assert_allclose(logL.cpu().numpy(), np.asarray(ref_l), rtol=1e-10)


def test_gradient_of_non_finite_data_is_nan():
    T, N, n = 0.5 * wk.YEAR, 64, 3
    th = candidates(2e-3, 1e-17, n, 3)
    win = [(int(2e-3 * T) - N // 2, N, N, 0, 0, n)]
    d = torch.full((N,), 1e-19 + 0j, dtype=torch.complex128, device="cuda")
    w = torch.full((N,), 1e41, dtype=torch.float64, device="cuda")
    bad = d.clone()
    bad[N // 2] = float("nan")
    _, g = api.Context(T).loglik_grad(win, bad, d, w, w, torch.as_tensor(th, device="cuda"))
    assert torch.isnan(g).all()


# the eps terms' coefficient pi fdot (L/c)/3 1024 is admitted up to 2^-27
FDOT_MAX = 2.0 ** -27 / (math.pi * 2.5e9 / 299792458.0 / 3.0 * 1024.0)


@pytest.mark.parametrize("f0", [16e-3, 20e-3, 24e-3])
@pytest.mark.parametrize("frac", [0.93, 0.999, 1.001, -0.93, -0.999])
def test_templates_at_the_chirp_limit(f0, frac):
    """Sky positions around those where the differences of the receivers' chirp terms are largest."""
    T, N, n = 0.5 * wk.YEAR, 1024, 60
    th = candidates(f0, frac * FDOT_MAX, n, int(1e4 * f0))
    rng = np.random.default_rng(n)
    th[2:, 2] = rng.uniform(-0.5, 0.5, n - 2)
    th[2:, 3] = np.where(np.arange(n - 2) % 2, 0.70, 3.84) + rng.uniform(-0.6, 0.6, n - 2)
    out = api.Context(T).waveform_aet(torch.as_tensor(th, device="cuda"), N)
    q, ref = ld.template_aet(th, N, T)
    assert np.array_equal(out[3].cpu().numpy(), q)
    norm = lambda x: np.sqrt((np.abs(x) ** 2).sum(1).astype(np.float64))  # noqa: E731
    for h, r in zip(out[:2], ref[:2]):
        assert np.all(norm(h.cpu().numpy() - r) <= tolerance(th, T) * norm(r))


@pytest.mark.parametrize("x", [0.05, 0.2199, 0.2201, 0.4999, 0.5001, 1.2999, 1.3001, 2.3499, 2.3501])
def test_plain_form_at_its_series_lengths(x):
    """Candidates outside the fixed-point ranges (a drift above f0/1024, or f above 1.3 f*) on both sides of
    each length of the link-transfer series."""
    T, N, n = wk.YEAR, 64, 9
    eta = 2.0 / 1024 if x < 1.3 else 0.0
    f0 = x * FSTAR / (1.0 + eta)           # x = f_max / f*
    th = candidates(f0, eta * f0 / T, n, int(1e4 * x))
    out = api.Context(T).waveform_aet(torch.as_tensor(th, device="cuda"), N)
    q, ref = ld.template_aet(th, N, T)
    assert np.array_equal(out[3].cpu().numpy(), q)
    norm = lambda y: np.sqrt((np.abs(y) ** 2).sum(1).astype(np.float64))  # noqa: E731
    for h, r in zip(out[:2], ref[:2]):
        assert np.all(norm(h.cpu().numpy() - r) <= tolerance(th, T) * norm(r))


@pytest.mark.parametrize("f0,fdot", [(15e-3, 1.2e-13), (23e-3, 2e-13)])
def test_gradients_beside_a_loud_bin(f0, fdot):
    """N = 1,024 against differences of fourth order of the long-double model,
    steps of 1e-4 rad of phase.  Samples carry 2^-49 of the channels' scale (8
    units of 2^-52), the response, the transforms and the sums a few units
    each: 32 units of 2^-52 of the gradient's norm in all."""
    T, N, n = wk.YEAR, 1024, 3
    th = candidates(f0, fdot, n, int(1e4 * f0))
    th[:, 2] = [0.3, -0.8, 1.1]
    q, h = ld.template_aet(th, N, T)
    rng = np.random.default_rng(N)
    win = (int(q[0]) - N // 2, N, N)
    d = [(rng.standard_normal(N) + 1j * rng.standard_normal(N)) * 1e-20 for _ in range(2)]
    for x in d:
        x[N // 2 + 3] = 1e3 * np.abs(x).max()
    w = [rng.uniform(0.5, 1.5, N) * 1e41 for _ in range(2)]
    dev = lambda x: torch.as_tensor(np.ascontiguousarray(x), device="cuda")  # noqa: E731
    _, g = api.Context(T).loglik_grad([win + (0, 0, n)], dev(d[0]), dev(d[1]), dev(w[0]), dev(w[1]), dev(th))
    j = q[:, None] - N // 2 + np.arange(N)[None, :] - win[0]
    ok, jc = (j >= 0) & (j < N), np.clip(j, 0, N - 1)

    def value(step):
        total = 0
        for x, wt, s in zip(d, w, ld.template_aet(th, N, T, step)[1]):
            x, wt = x.astype(np.clongdouble)[jc], wt.astype(np.longdouble)[jc] * ok
            total = total + (wt * ((x * s.conj()).real - (s.real ** 2 + s.imag ** 2) / 2)).sum(1)
        return total * (4 / np.longdouble(T))

    unit = 1 / np.concatenate([[2 * math.pi * T, math.pi * T * T], [2 * math.pi * f0 * 500] * 2, [1.0, 2.0, 4.0, 1.0]])
    unit = np.tile(unit.astype(np.longdouble), (n, 1))
    unit[:, 4] = th[:, 4]
    ref = np.empty((n, 8), np.longdouble)
    for k in range(8):
        e = np.zeros(8, np.longdouble)
        e[k] = 1e-4 * unit[:, k].min()
        ref[:, k] = (8 * (value(e) - value(-e)) - (value(2 * e) - value(-2 * e))) / (12 * e[k])
    err = np.abs((g.cpu().numpy() - ref) * unit).max(1) / np.sqrt(((ref * unit) ** 2).sum(1))
    assert err.max() < 32 * 2.0 ** -52, err
