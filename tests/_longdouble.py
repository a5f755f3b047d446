"""The response model in numpy's long double (64 or 113 bits of mantissa), as a
reference for results that are more exact than plain double arithmetic: the
oracle's expressions (oracle/gb.py), with the carrier bin and delta rounded as
reading R7 fixes them."""
import numpy as np

L = np.longdouble
PI = L("3.14159265358979323846264338327950288")
C, AU, ARM, YEAR = L(299792458), L(1.495978707e11), L(2.5e9), L(31557600)


def template_aet(theta, N, T, step=None):
    """q (int64) and the A, E, T templates on bins q - N/2 ... q + N/2 - 1, clongdouble.
    step (8 long doubles): the parameters' offset from theta, whose carrier bin and delta's rounding are kept."""
    th = np.asarray(theta, dtype=np.float64)
    f0T = th[:, 0] * float(T)
    q = np.floor((f0T + ((0.5 * th[:, 1]) * float(T)) * float(T)) + 0.5)
    step = np.zeros(8, L) if step is None else step
    delta = (f0T - q).astype(L)[:, None] + step[0] * L(T)
    T = L(T)
    n = np.arange(N).astype(L)
    t = n * T / L(N)
    a = 2 * PI * t / YEAR
    s3, ecc = np.sqrt(L(3)), ARM / (2 * np.sqrt(L(3)) * AU)
    x = []
    for i in range(3):
        b = 2 * PI * i / 3
        x.append((AU * np.cos(a) + AU * ecc / 2 * (np.cos(2 * a - b) - 3 * np.cos(b)),
                  AU * np.sin(a) + AU * ecc / 2 * (np.sin(2 * a - b) - 3 * np.sin(b)), -s3 * AU * ecc * np.cos(a - b)))
    f0, fd, be, la, A, io, ps, ph = (th[:, j].astype(L)[:, None] + step[j] for j in range(8))
    sb, cb, sl, cl = np.sin(be), np.cos(be), np.sin(la), np.cos(la)
    k, u, v = (-cb * cl, -cb * sl, -sb), (sb * cl, sb * sl, -cb), (sl, -cl)
    c2, s2, ci = np.cos(2 * ps), np.sin(2 * ps), np.cos(io)
    Ap, Ax = A * (1 + ci * ci), -2 * A * ci
    rx = []
    for i in range(3):
        kap = (k[0] * x[i][0] + k[1] * x[i][1] + k[2] * x[i][2]) / C
        cyc = delta * n / L(N) + fd * t * t / 2 - f0 * kap - fd * t * kap + fd * kap * kap / 2
        p = 2 * PI * (cyc - np.rint(cyc)) + ph
        rx.append(np.cos(p) + 1j * np.sin(p))
    f, fstar = f0 + fd * t, C / (2 * PI * ARM)
    h, z = f / (2 * fstar), {}
    for i, j in ((0, 1), (1, 2), (2, 0)):
        d = [x[j][m] - x[i][m] for m in range(3)]
        r = np.sqrt(sum(y * y for y in d))
        d = [y / r for y in d]
        kn, nu, nv = (sum(p * y for p, y in zip(w, d)) for w in (k, u, v))
        Fp, Fx = nu * nu - nv * nv, 2 * nu * nv
        G = Ap * (c2 * Fp - s2 * Fx) - 1j * Ax * (s2 * Fp + c2 * Fx)
        for (p, c), sg in (((i, j), -1), ((j, i), 1)):
            X = h * (1 + sg * kn)
            V = np.where(X != 0, np.sin(X) / np.where(X != 0, X, 1), 1) * (np.cos(X) - 1j * np.sin(X))
            z[(p, c)] = -1j * h * V * G * rx[c]
    D = np.cos(f / fstar) - 1j * np.sin(f / fstar)
    X, Y, Z = ((1 - D * D) * ((z[(p, c)] + D * z[(c, p)]) - (z[(r, c)] + D * z[(c, r)]))
               for c, p, r in ((0, 1, 2), (1, 2, 0), (2, 0, 1)))
    s = ((Z - X) / np.sqrt(L(2)), (X - 2 * Y + Z) / np.sqrt(L(6)), (X + Y + Z) / s3)
    return q.astype(np.int64), [T / (2 * L(N)) * np.fft.fftshift(np.fft.fft(y), axes=1) for y in s]


def loglik(win, dA, dE, wA, wE, theta, T):
    """logL, <d|h>, <h|h> of one window's candidates (A and E)."""
    k0, W, N = win[:3]
    q, h = template_aet(theta, N, T)
    j = q[:, None] - N // 2 + np.arange(N)[None, :] - k0
    ok, jc = (j >= 0) & (j < W), np.clip(j, 0, W - 1)
    dh = hh = dd = L(0)
    for d, w, s in ((dA, wA, h[0]), (dE, wE, h[1])):
        d, w = d.astype(np.clongdouble), w.astype(L)
        dh = dh + np.where(ok, w[jc] * (d[jc] * s.conj()).real, 0).sum(1)
        hh = hh + np.where(ok, w[jc] * (s.real ** 2 + s.imag ** 2), 0).sum(1)
        dd = dd + (w * (d.real ** 2 + d.imag ** 2)).sum()
    dh, hh, dd = (4 / L(T) * v for v in (dh, hh, dd))
    return dh - hh / 2 - dd / 2, dh, hh
