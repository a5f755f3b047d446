"""The fixed-point slow part of the FP64 path, compiled for the host and held
against the response model in long double: rounding, and the index arithmetic
at the limits of the admitted ranges.  Every signed overflow is counted (the
products and sums of the headers must not wrap; the carrier phase, which does,
is unsigned)."""
import ctypes
import math
import os
import shutil
import subprocess

import numpy as np
import pytest

from tests import _longdouble as ld

HERE = os.path.dirname(os.path.abspath(__file__))
YEAR = 31557600.0
ARM_C = 2.5e9 / 299792458.0
# the eps terms' coefficient pi fdot (L/c)/3 1024 is admitted up to 2^-27
FDOT_MAX = 2.0 ** -27 / (math.pi * ARM_C / 3.0 * 1024.0)


@pytest.fixture(scope="module")
def host(tmp_path_factory):
    cxx = shutil.which("g++")
    if cxx is None:
        pytest.skip("no host compiler")
    tmp = tmp_path_factory.mktemp("fx64")
    obj, out = str(tmp / "fx64_host.o"), str(tmp / "fx64_host.so")
    subprocess.run([cxx, "-c", "-O2", "-std=c++20", "-fPIC", "-ffp-contract=off", "-fsanitize=signed-integer-overflow",
                    "-I", os.path.join(HERE, os.pardir, "paper_2307_03763_gb300", "csrc"),
                    os.path.join(HERE, "fx64_host.cpp"), "-o", obj], check=True)
    subprocess.run([cxx, "-shared", obj, "-o", out], check=True)
    return ctypes.CDLL(out)


def no_overflow(host):
    line = ctypes.c_int()
    n = host.host_overflows(ctypes.byref(line))
    assert n == 0, "%d signed overflows, the last at line %d" % (n, line.value)


def _ptr(a):
    return a.ctypes.data_as(ctypes.c_void_p)


def geometry(N, T):
    """Arm vectors n_01, n_12 and cos, sin of the orbital phase, (N, 8) doubles."""
    L = np.longdouble
    a = 2 * ld.PI * (np.arange(N).astype(L) * L(T) / L(N) / ld.YEAR)
    s, c = np.sin(a), np.cos(a)
    s2, c2, r3 = np.sin(2 * a), np.cos(2 * a), np.sqrt(L(3))
    g = ((4.5 - 1.5 * c2) / (4 * r3) + s2 / 8, -0.375 - c2 / 8 - 1.5 * s2 / (4 * r3), 0.75 * c - r3 / 4 * s,
         -s2 / 4, (c2 + 3) / 4, r3 / 2 * s, c, s)
    return np.ascontiguousarray(np.stack(g, 1).astype(np.float64))


def delta(th, T):
    f0T = th[:, 0] * float(T)
    return f0T - np.floor((f0T + ((0.5 * th[:, 1]) * float(T)) * float(T)) + 0.5)


def samples(host, th, N, T, arm_c=ARM_C):
    B, lg = len(th), N.bit_length() - 1
    th = np.ascontiguousarray(th)
    d, geo = np.ascontiguousarray(delta(th, T)), geometry(N, T)
    tier, out, sc = np.zeros(B, np.int32), np.zeros((B, N, 3, 2), np.int64), np.zeros((B, 3))
    host.host_samples(B, _ptr(th), _ptr(d), ctypes.c_double(T), ctypes.c_double(arm_c), lg, _ptr(geo), _ptr(tier),
                      _ptr(out), _ptr(sc))
    return tier, out, sc


def sky(f0, fdot, n, seed):
    """Candidates over the whole sky, the poles and the ecliptic among them."""
    rng = np.random.default_rng(seed)
    th = np.empty((n, 8))
    th[:, 0], th[:, 1], th[:, 4] = f0, fdot, 1e-22
    th[:, 2] = np.arcsin(rng.uniform(-1, 1, n))
    th[:, 3] = rng.uniform(-math.pi, math.pi, n)
    th[:, 5] = np.arccos(rng.uniform(-1, 1, n))
    th[:, 6], th[:, 7] = rng.uniform(0, math.pi, n), rng.uniform(0, 2 * math.pi, n)
    th[0, 2], th[1, 2], th[2, 2] = math.pi / 2, -math.pi / 2, 0.0
    return th


def template_errors(host, th, N, T):
    """|template - model| of A and E, relative to the model's norm."""
    tier, out, sc = samples(host, th, N, T)
    _, ref = ld.template_aet(th, N, T)
    err = []
    for ch in range(2):
        s = out[:, :, ch, 0].astype(np.longdouble) + 1j * out[:, :, ch, 1].astype(np.longdouble)
        h = np.fft.fftshift(np.fft.fft(s, axis=1), axes=1) * sc[:, ch, None].astype(np.longdouble)
        err.append(np.sqrt((np.abs(h - ref[ch]) ** 2).sum(1) / (np.abs(ref[ch]) ** 2).sum(1)).astype(np.float64))
    return tier, np.maximum(*err)


# Samples carry 2^-52 of the channels' scale; 2^-44 leaves room for sky
# positions at which A or E is weak.  A wrapped term is seen at 1e-9.
TOL = 2.0 ** -44


@pytest.mark.parametrize("f0,years,frac", [(f0, years, frac) for f0, years in ((16e-3, 0.5), (20e-3, 0.5), (24e-3, 0.5),
                                                                            (24e-3, 0.9))
                                           for frac in (0.9, 0.95, 1 - 2.0 ** -33, -0.92, -(1 - 2.0 ** -40))])
def test_chirp_at_its_limit(host, f0, years, frac):
    """fdot up to the limit of the eps terms, over the sky: no receiver's term, and no difference of two, may wrap."""
    T = years * YEAR
    th = sky(f0, frac * FDOT_MAX, 1500, int(f0 * 1e6))
    tier, err = template_errors(host, th, 64, T)
    inside = abs(frac * FDOT_MAX * T / f0) <= 2.0 ** -10
    assert (tier == -1).all() or inside
    assert err[tier >= 0].size == 0 or err[tier >= 0].max() < TOL, err[tier >= 0].max()
    no_overflow(host)


@pytest.mark.parametrize("f0,fdot,N", [(0.3e-3, 0.0, 32), (1e-3, 1e-18, 64), (9.5e-3, 1e-15, 128),
                                       (9.6e-3, 1e-15, 256), (24.8e-3, 2e-13, 512), (15e-3, 1.2e-13, 1024),
                                       (5e-3, -3e-14, 128)])
def test_samples_against_long_double(host, f0, fdot, N):
    th = sky(f0, fdot, 40, N)
    tier, err = template_errors(host, th, N, YEAR)
    assert (tier >= 0).all() and err.max() < TOL, err.max()
    no_overflow(host)


@pytest.mark.parametrize("sign", [1, -1])
def test_long_arms_at_the_chirp_limit(host, sign):
    """Arms of almost 300 s, where k.rho counts beside the guiding centre's K: nothing may wrap."""
    arm = 299.0
    fdot = sign * 0.9999 * 2.0 ** -27 / (math.pi * arm / 3.0 * 1024.0)
    tier, _, _ = samples(host, sky(6.5e-4, fdot, 1500, 5), 64, 0.8 * YEAR, arm)
    assert (tier >= 0).all()
    no_overflow(host)


@pytest.mark.parametrize("f0,fdot,N,years", [(24e-3, 0.97 * FDOT_MAX, 64, 0.5), (24e-3, -0.99 * FDOT_MAX, 64, 0.5),
                                             (20e-3, 0.95 * FDOT_MAX, 128, 0.5), (4e-3, 1e-15, 256, 1.0),
                                             (0.5e-3, 0.0, 32, 2.0)])
def test_gradients_against_long_double(host, f0, fdot, N, years):
    """Against differences of the model of fourth order, steps of 3e-4 rad of
    phase (3e-4^4/30, and 2^-63/3e-4 of rounding: 1e-11 leaves room for both)."""
    T, n, rng = years * YEAR, 60, np.random.default_rng(N)
    th, lg = sky(f0, fdot, n, N + 1), N.bit_length() - 1
    g = rng.uniform(-1, 1, (n, N, 3, 2))
    cot = np.rint(g * np.array([1, 3 ** -0.5, (2 / 3) ** 0.5])[:, None] * 2.0 ** 60).astype(np.int64)
    d, geo = np.ascontiguousarray(delta(th, T)), geometry(N, T)
    tier, grad = np.zeros(n, np.int32), np.zeros((n, 8))
    host.host_gradients(n, _ptr(th), _ptr(d), ctypes.c_double(T), ctypes.c_double(ARM_C), lg, _ptr(geo), _ptr(cot),
                        _ptr(tier), _ptr(grad))
    assert (tier >= 0).all()
    no_overflow(host)
    w = g[..., 0] + 1j * g[..., 1]   # conj(c_n)

    def value(step):
        total = np.zeros(n, np.longdouble)
        for ch, h in enumerate(ld.template_aet(th, N, T, step)[1]):
            s = np.fft.ifft(np.fft.ifftshift(h, axes=1), axis=1) * (2 * N / np.longdouble(T))
            total += (w[:, :, ch] * s).real.sum(1)
        return 2 * total / N

    ang = 2 * math.pi * max(f0 * 500.0, 1.0)
    unit = 1 / np.array([2 * math.pi * T, math.pi * T * T, ang, ang, 1e22, 2.0, 4.0, 1.0])   # about a radian each
    ref = np.empty((n, 8))
    for j in range(8):
        e = np.zeros(8, np.longdouble)
        e[j] = 3e-4 * unit[j]
        ref[:, j] = ((8 * (value(e) - value(-e)) - (value(2 * e) - value(-2 * e))) / (12 * e[j])).astype(np.float64)
    scale = np.linalg.norm(ref * unit, axis=1)
    err = (np.abs(grad - ref) * unit).max(1) / scale
    assert err.max() < 1e-11, err.max()


@pytest.mark.parametrize("N", [32, 64, 128, 256, 512, 1024])
@pytest.mark.parametrize("kind", ["white", "dominant", "equal", "edge", "tones", "huge", "tiny"])
def test_residual_transform_against_long_double(host, N, kind):
    """The adjoint transform, to the error of one in double: its output carries
    about log2 N roundings of 2^-53 (numpy's own: 2e-16 at N = 1,024); 2^-51.
    equal reaches the bound that the integers are scaled by."""
    rng = np.random.default_rng(N)
    B, lg = 8, N.bit_length() - 1
    x = rng.normal(size=(B, N)) + 1j * rng.normal(size=(B, N))
    if kind == "dominant":      # a loud source's bin
        x[np.arange(B), rng.integers(0, N, B)] = 1e3 * np.exp(2j * math.pi * rng.uniform(size=B))
    elif kind == "equal":
        x = np.exp(0.5j * math.pi * rng.integers(0, 4, (B, 1))) * np.ones((B, N)) * (1 - 2.0 ** -50)
    elif kind == "edge":        # a window that ends within the template
        x[:, N // 5:] = 0.0
    elif kind == "tones":
        x = np.exp(2j * math.pi * rng.integers(0, N, (B, 1)) * np.arange(N) / N)
    elif kind in ("huge", "tiny"):
        x = x * (1e300 if kind == "huge" else 1e-280)
    r = np.ascontiguousarray(np.stack([x.real, x.imag], -1))
    out, power = np.zeros((B, N, 2), np.int64), np.zeros(B, np.int32)
    host.host_transform(B, lg, _ptr(r), _ptr(out), _ptr(power))
    no_overflow(host)
    got = out[..., 0].astype(np.longdouble) + 1j * out[..., 1].astype(np.longdouble)
    ref = np.fft.fft(x.astype(np.clongdouble) * np.ldexp(np.longdouble(1), power)[:, None], axis=1)
    err = np.sqrt((np.abs(got - ref) ** 2).sum(1) / (np.abs(ref) ** 2).sum(1))
    assert err.max() < 2.0 ** -51, err.max()


def test_residuals_out_of_range(host):
    """Sums beyond a double's range, and none: finite integers without overflow."""
    for x in (np.full((1, 64, 2), 1.5e308), np.zeros((1, 64, 2)), np.full((1, 64, 2), 5e-324)):
        out, power = np.zeros((1, 64, 2), np.int64), np.zeros(1, np.int32)
        host.host_transform(1, 6, _ptr(x), _ptr(out), _ptr(power))
        no_overflow(host)
        assert abs(out).max() < 2 ** 62 + 2 ** 20
