// fp64_common.cuh -- device code shared by the FP64 likelihood and gradient:
// candidates, their set-up, the template in fixed point (fx64.cuh) or plain
// double, and its transform.  Every definition sits in an anonymous namespace.
#pragma once
#include <cmath>

#include "fx64.cuh"
#include "gb_internal.cuh"

namespace gb {
namespace {

struct C64 {
    double x, y;
};
__device__ __forceinline__ C64 cadd(C64 a, C64 b) { return {a.x + b.x, a.y + b.y}; }
__device__ __forceinline__ C64 csub(C64 a, C64 b) { return {a.x - b.x, a.y - b.y}; }
__device__ __forceinline__ C64 cmul(C64 a, C64 b) { return {a.x * b.x - a.y * b.y, a.x * b.y + a.y * b.x}; }
__device__ __forceinline__ C64 cscale(C64 a, double s) { return {a.x * s, a.y * s}; }

// Per-candidate constants.
struct Cand64 {
    double k[3];          // propagation direction
    double u[3], v[3];    // polarisation basis (psi = 0)
    double gpr, gxr, gpi, gxi;   // n.H.n = (gpr Fp + gxr Fx) + i (gpi Fp + gxi Fx), Fp = (n.u)^2 - (n.v)^2, Fx = 2 (n.u)(n.v)
    double f0, fd, delta, phi0c, A;   // phi0c = phi0 / (2 pi)
    double D0r, D0i;      // exp(-i f0 / f*)
    double eps;           // fdot / f*
    int J;                // degree of the link-transfer series (0: direct evaluation)
};

// One candidate: its carrier bin and either form's constants.  sA, sE, sT: a
// channel's bin value per unit of its transform.
struct CandT {
    long long q;
    int bad;
    int tier;             // of the fixed-point form; -1: plain double
    double sA, sE, sT;
    union {
        CandFx f;
        Cand64 d;
    };
};

struct Geo64 {
    double T, T_over_N, inv_fstar, scale;   // scale = T / (2N)
    double arm_c;                           // L/c, s
    int N, logN, krho_q30;                  // (L/c)/(3 1024 s) in Q30
};

// Set-up of one candidate.  The carrier bin uses explicit round-to-nearest
// operations so that q is bit-identical to any IEEE evaluation of
// ((f0*T) + ((0.5*fdot)*T)*T) + 0.5.  `t`: the sines and cosines setup_fx
// wants.
__device__ void setup64(const double* th, double T, double inv_fstar, double delta, Cand64& c);
__device__ __forceinline__ double carrier64(const double* th, double T, CandT& c) {
    bool bad = false;
    for (int i = 0; i < 8; ++i) bad |= !isfinite(th[i]);
    c.bad = bad;
    const double f0T = __dmul_rn(th[0], T);
    const double xm = __dadd_rn(f0T, __dmul_rn(__dmul_rn(__dmul_rn(0.5, th[1]), T), T));
    const double qd = floor(__dadd_rn(xm, 0.5));
    c.q = bad ? 0 : (long long)qd;
    return __dadd_rn(f0T, -qd);
}
__device__ __forceinline__ void setup_t(const double* th, const Geo64& g, double delta, const FxTrig& t, CandT& c) {
    if (c.bad) {
        c.tier = -1;
        return;
    }
    setup_fx(th, g.T, g.arm_c, delta, g.logN, t, c.f);
    c.tier = c.f.tier;
    if (c.tier >= 0) {
        c.sA = c.f.sA;
        c.sE = c.f.sE;
        c.sT = c.f.sT;
    } else {
        setup64(th, g.T, g.inv_fstar, delta, c.d);
        c.sA = c.sE = c.sT = g.scale;
    }
}
// one lane, one candidate (t, ii: its sines and cosines, sin iota)
__device__ void setup_lane(const double* th, const Geo64& g, CandT& c, FxTrig& t, double& ii) {
    const double delta = carrier64(th, g.T, c);
    sincos(th[2], &t.sb, &t.cb);
    sincos(th[3], &t.sl, &t.cl);
    sincos(2.0 * th[6], &t.s2, &t.c2);
    sincos(th[5], &ii, &t.ci);
    sincos(kPi * th[0] * g.arm_c, &t.sa, &t.ca);
    setup_t(th, g, delta, t, c);
}
__device__ __forceinline__ void setup_lane(const double* th, const Geo64& g, CandT& c) {
    FxTrig t;
    double ii;
    setup_lane(th, g, c, t, ii);
}
// Up to six candidates by a whole warp: each one's five sines and cosines on
// five lanes (the double sincos is a long dependent chain), the rest on one
// lane per candidate.
constexpr int kSetupWarp = 6;
__device__ void setup_warp(const double* th, int cnt, const Geo64& g, CandT* c, int lane) {
    const int mine = lane / 5 < cnt ? lane / 5 : cnt - 1, kind = lane % 5;
    const double* t0 = th + 8 * mine;
    const double x = kind == 0 ? t0[2] : kind == 1 ? t0[3] : kind == 2 ? 2.0 * t0[6] : kind == 3 ? t0[5] : kPi * t0[0] * g.arm_c;
    double sn, cs;
    sincos(x, &sn, &cs);
    const int src = 5 * (lane < cnt ? lane : 0);
    FxTrig t;
    t.sb = __shfl_sync(0xffffffffu, sn, src);
    t.cb = __shfl_sync(0xffffffffu, cs, src);
    t.sl = __shfl_sync(0xffffffffu, sn, src + 1);
    t.cl = __shfl_sync(0xffffffffu, cs, src + 1);
    t.s2 = __shfl_sync(0xffffffffu, sn, src + 2);
    t.c2 = __shfl_sync(0xffffffffu, cs, src + 2);
    t.ci = __shfl_sync(0xffffffffu, cs, src + 3);
    t.sa = __shfl_sync(0xffffffffu, sn, src + 4);
    t.ca = __shfl_sync(0xffffffffu, cs, src + 4);
    if (lane < cnt) {
        const double* tl = th + 8 * lane;
        const double delta = carrier64(tl, g.T, c[lane]);
        setup_t(tl, g, delta, t, c[lane]);
    }
}

// 1/k!, k < 35: the link-transfer series
__constant__ double kInvFact64[35] = {
    1.00000000000000000e+00, 1.00000000000000000e+00, 5.00000000000000000e-01, 1.66666666666666657e-01,
    4.16666666666666644e-02, 8.33333333333333322e-03, 1.38888888888888894e-03, 1.98412698412698413e-04,
    2.48015873015873016e-05, 2.75573192239858925e-06, 2.75573192239858883e-07, 2.50521083854417202e-08,
    2.08767569878681002e-09, 1.60590438368216133e-10, 1.14707455977297245e-11, 7.64716373181981641e-13,
    4.77947733238738525e-14, 2.81145725434552060e-15, 1.56192069685862253e-16, 8.22063524662432950e-18,
    4.11031762331216484e-19, 1.95729410633912626e-20, 8.89679139245057408e-22, 3.86817017063068413e-23,
    1.61173757109611839e-24, 6.44695028438447359e-26, 2.47959626322479759e-27, 9.18368986379554601e-29,
    3.27988923706983776e-30, 1.13099628864477159e-31, 3.76998762881590539e-33, 1.21612504155351789e-34,
    3.80039075485474342e-36, 1.15163356207719509e-37, 3.38715753552116180e-39};

// Set-up of the plain double form (one lane, one candidate).
__device__ void setup64(const double* th, double T, double inv_fstar, double delta, Cand64& c) {
    const double f0 = th[0], fd = th[1], beta = th[2], lam = th[3];
    const double A = th[4], iota = th[5], psi = th[6], phi0 = th[7];
    c.delta = delta;
    c.f0 = f0;
    c.fd = fd;
    c.phi0c = phi0 * 0.15915494309189535;   // 1 / (2 pi)
    c.A = A;
    double sb, cb, sl, cl, s2, c2;
    sincos(beta, &sb, &cb);
    sincos(lam, &sl, &cl);
    sincos(2.0 * psi, &s2, &c2);
    const double ci = cos(iota);
    c.k[0] = -(cb * cl);
    c.k[1] = -(cb * sl);
    c.k[2] = -sb;
    c.u[0] = sb * cl;
    c.u[1] = sb * sl;
    c.u[2] = -cb;
    c.v[0] = sl;
    c.v[1] = -cl;
    c.v[2] = 0.0;
    // H = A+ E+(psi) - i Ax Ex(psi) with E+ = u u - v v and Ex = u v + v u rotated
    // by 2 psi: n.H.n = A+ (c2 Fp - s2 Fx) - i Ax (s2 Fp + c2 Fx)
    const double Ap = A * (1.0 + ci * ci);
    const double Ax = -2.0 * A * ci;
    c.gpr = Ap * c2;
    c.gxr = -(Ap * s2);
    c.gpi = -(Ax * s2);
    c.gxi = -(Ax * c2);
    // link-transfer series: first omitted term below 1e-17 for the largest
    // argument X = f (1 + |k.n|)/(2 f*) <= f_max / f*
    const double xmax = fmax(fabs(f0), fabs(f0 + fd * T)) * inv_fstar;
    c.J = xmax <= 0.22 ? 6 : xmax <= 0.5 ? 8 : xmax <= 1.3 ? 12 : xmax <= 2.35 ? 16 : 0;
    double sD, cD;
    sincos(f0 * inv_fstar, &sD, &cD);
    c.D0r = cD;
    c.D0i = -sD;
    c.eps = fd * inv_fstar;
}

// n.H.n for a unit arm vector n
__device__ __forceinline__ C64 nHn(const Cand64& c, double nx, double ny, double nz) {
    const double nu = c.u[0] * nx + c.u[1] * ny + c.u[2] * nz;
    const double nv = c.v[0] * nx + c.v[1] * ny;
    const double Fp = (nu - nv) * (nu + nv), Fx = 2.0 * nu * nv;
    return {c.gpr * Fp + c.gxr * Fx, c.gpi * Fp + c.gxi * Fx};
}

// sinc(X) exp(-iX): J+1 terms of the series of (1 - e^{-2iX})/(2iX) split into
// real and imaginary parts (Horner in y = -4X^2), or evaluated directly.  J is
// a run-time number: one length for all (16) took 20% longer at 4 mHz (160,000
// likelihoods of drifting candidates, N = 256: 49.8 -> 41.1 ms), an unrolled
// copy per length takes registers from the kernels' fixed-point form.
template <bool SERIES>
__device__ __forceinline__ C64 transfer64(double X, int J) {
    if constexpr (!SERIES) {
        double sX, cX;
        sincos(X, &sX, &cX);
        const double sinc = (X != 0.0) ? sX / X : 1.0;
        return {sinc * cX, -(sinc * sX)};
    } else {
        const double y = -4.0 * X * X;
        double re = kInvFact64[2 * J + 1], im = kInvFact64[2 * J + 2];
#pragma unroll 2
        for (int j = J - 1; j >= 0; --j) {
            re = fma(re, y, kInvFact64[2 * j + 1]);
            im = fma(im, y, kInvFact64[2 * j + 2]);
        }
        return {re, -2.0 * X * im};
    }
}

// -i a sinc(X) exp(-iX) G exp(i Psi)
template <bool SERIES>
__device__ __forceinline__ C64 link64(double a, double X, C64 G, C64 rx, int J) {
    const C64 t = transfer64<SERIES>(X, J);
    const C64 tr = {a * t.x, a * t.y};
    const C64 z = cmul(cmul(tr, G), rx);
    return {z.y, -z.x};                                    // times -i
}

// Slow part of one candidate into buf{A,E} at bit-reversed positions, then
// an in-place radix-2 FFT -> natural-order DFT S_k, k = 0..N-1.  The receiver
// phases reach ~1e6 rad; taken in cycles and reduced modulo one first, their
// sines come from a short argument.
// bufT (may be null): also T = (X + Y + Z)/sqrt3
// NT threads share the candidate (NT = 32: one warp, `lane` its lane; NT > 32:
// the whole CTA, `lane` the thread index); each sample and each butterfly is
// computed by the same code whichever thread takes it, so the bits do not
// depend on NT (here and in the fixed-point form).
template <bool SERIES, int NT>
__device__ __noinline__ void template64(const Cand64& c, const Geo64& g, const OrbitTables64& tab, const C64* tw,
                           C64* bufA, C64* bufE, C64* bufT, int lane) {
    const int N = g.N;
    const double inv_c = 1.0 / kC;
    const double u_step = 1.0 / (double)N;   // t/T = n/N exactly
    for (int n = lane; n < N; n += NT) {
        const double t = (double)n * g.T_over_N;
        C64 rx[3];
        for (int j = 0; j < 3; ++j) {
            const double kap = (c.k[0] * tab.x[(j * 3 + 0) * N + n] + c.k[1] * tab.x[(j * 3 + 1) * N + n] +
                                c.k[2] * tab.x[(j * 3 + 2) * N + n]) * inv_c;
            // receiver phase in cycles, reduced modulo one before the sine and cosine
            double cyc = c.delta * ((double)n * u_step) + 0.5 * c.fd * (t * t) - c.f0 * kap - c.fd * t * kap +
                         0.5 * c.fd * (kap * kap) + c.phi0c;
            cyc -= rint(cyc);
            double s, co;
            sincospi(2.0 * cyc, &s, &co);
            rx[j] = {co, s};
        }
        const double f = c.f0 + c.fd * t;
        const double a = f * (0.5 * g.inv_fstar);
        C64 z01, z10, z12, z21, z20, z02;
        {
            const double nx = tab.arm[0 * N + n], ny = tab.arm[1 * N + n], nz = tab.arm[2 * N + n];
            const double kn = c.k[0] * nx + c.k[1] * ny + c.k[2] * nz;
            const C64 G = nHn(c, nx, ny, nz);
            z01 = link64<SERIES>(a, a * (1.0 - kn), G, rx[1], c.J);
            z10 = link64<SERIES>(a, a * (1.0 + kn), G, rx[0], c.J);
        }
        {
            const double nx = tab.arm[3 * N + n], ny = tab.arm[4 * N + n], nz = tab.arm[5 * N + n];
            const double kn = c.k[0] * nx + c.k[1] * ny + c.k[2] * nz;
            const C64 G = nHn(c, nx, ny, nz);
            z12 = link64<SERIES>(a, a * (1.0 - kn), G, rx[2], c.J);
            z21 = link64<SERIES>(a, a * (1.0 + kn), G, rx[1], c.J);
        }
        {
            const double nx = tab.arm[6 * N + n], ny = tab.arm[7 * N + n], nz = tab.arm[8 * N + n];
            const double kn = c.k[0] * nx + c.k[1] * ny + c.k[2] * nz;
            const C64 G = nHn(c, nx, ny, nz);
            z20 = link64<SERIES>(a, a * (1.0 - kn), G, rx[0], c.J);
            z02 = link64<SERIES>(a, a * (1.0 + kn), G, rx[2], c.J);
        }
        // D = exp(-i f/f*) = exp(-i f0/f*) exp(-i th), th = fdot t / f*: a short
        // series while |th| <= 1/64 (terms to th^7, first omitted below 1e-19)
        C64 D;
        const double th = c.eps * t;
        if (fabs(th) <= 0.015625) {
            const double t2 = th * th;
            const double cs = fma(fma(fma(t2, -1.0 / 720.0, 1.0 / 24.0), t2, -0.5), t2, 1.0);
            const double sn = th * fma(fma(fma(t2, -1.0 / 5040.0, 1.0 / 120.0), t2, -1.0 / 6.0), t2, 1.0);
            D = cmul({c.D0r, c.D0i}, {cs, -sn});
        } else {
            double sD, cD;
            sincos(f * g.inv_fstar, &sD, &cD);
            D = {cD, -sD};
        }
        const C64 D2 = cmul(D, D);
        const C64 omd = {1.0 - D2.x, -D2.y};
        const C64 X = cmul(omd, csub(cadd(z10, cmul(D, z01)), cadd(z20, cmul(D, z02))));
        const C64 Y = cmul(omd, csub(cadd(z21, cmul(D, z12)), cadd(z01, cmul(D, z10))));
        const C64 Z = cmul(omd, csub(cadd(z02, cmul(D, z20)), cadd(z12, cmul(D, z21))));
        const double r2 = 0.70710678118654752, r6 = 0.40824829046386302;   // 1/sqrt(2), 1/sqrt(6)
        const C64 sA = {(Z.x - X.x) * r2, (Z.y - X.y) * r2};
        const C64 sE = {(X.x - 2.0 * Y.x + Z.x) * r6, (X.y - 2.0 * Y.y + Z.y) * r6};
        const int br = (int)(__brev((unsigned)n) >> (32 - g.logN));
        bufA[sw(br)] = sA;
        bufE[sw(br)] = sE;
        if (bufT) {
            const double r3 = 0.57735026918962576;   // 1/sqrt(3)
            bufT[sw(br)] = {(X.x + Y.x + Z.x) * r3, (X.y + Y.y + Z.y) * r3};
        }
    }
    sync_nt<NT>();
    // radix-2 decimation in time, bit-reversed input, natural-order output
    for (int s = 0; s < g.logN; ++s) {
        const int h = 1 << s;
        const int tstride = kTwiddles >> s;
        for (int b = lane; b < N / 2; b += NT) {
            const int j = b & (h - 1);
            const int e0 = ((b >> s) << (s + 1)) + j, i0 = sw(e0), i1 = sw(e0 + h);
            const C64 w = tw[j * tstride];
            const C64 ua = bufA[i0], va = cmul(w, bufA[i1]);
            bufA[i0] = cadd(ua, va);
            bufA[i1] = csub(ua, va);
            const C64 ue = bufE[i0], ve = cmul(w, bufE[i1]);
            bufE[i0] = cadd(ue, ve);
            bufE[i1] = csub(ue, ve);
            if (bufT) {
                const C64 ut = bufT[i0], vt = cmul(w, bufT[i1]);
                bufT[i0] = cadd(ut, vt);
                bufT[i1] = csub(ut, vt);
            }
        }
        sync_nt<NT>();
    }
}

// The plain double form, scaled to bin values in place.
template <int NT>
__device__ void template_plain(const CandT& c, const Geo64& g, const OrbitTables64& tab, const C64* tw, C64* bufA,
                               C64* bufE, C64* bufT, int lane) {
    if (c.d.J) template64<true, NT>(c.d, g, tab, tw, bufA, bufE, bufT, lane);
    else template64<false, NT>(c.d, g, tab, tw, bufA, bufE, bufT, lane);
    for (int i = lane; i < g.N; i += NT) {
        bufA[i] = cscale(bufA[i], g.scale);
        bufE[i] = cscale(bufE[i], g.scale);
        if (bufT) bufT[i] = cscale(bufT[i], g.scale);
    }
    sync_nt<NT>();
}

// Samples of one candidate into buf{A,E,T} at bit-reversed positions.
template <int TIER, bool T3>
__device__ __noinline__ void samples_fx(const CandFx& c, const int4* __restrict__ geo, const FxTw* tw, int krho_q30,
                                        int lg, Z64* bufA, Z64* bufE, Z64* bufT, int lane, int nt) {
    const int N = 1 << lg, sh = fx_shift(lg);
    for (int n = lane; n < N; n += nt) {
        const int4 a = __ldg(geo + n), b = __ldg(geo + N + n), e = __ldg(geo + 2 * N + n), f = __ldg(geo + 3 * N + n);
        const GeoFx g{{a.x, a.y}, {a.z, a.w}, {b.x, b.y}, {b.z, b.w}, {e.x, e.y}, {e.z, e.w}, {f.x, f.y}, {f.z, f.w}};
        fx o[6];
        sample_fx<TIER, T3>(c, g, tw, krho_q30, n, lg, sh, o);
        const int br = sw((int)(__brev((unsigned)n) >> (32 - lg)));
        bufA[br] = {o[0], o[1]};
        bufE[br] = {o[2], o[3]};
        if (T3) bufT[br] = {o[4], o[5]};
    }
}

// Tables of the fixed-point form
struct FxTab {
    const int4* geo;      // [4][N] of this size: (n01.x, n01.y), (n01.z, n12.x), (n12.y, n12.z), (cos a, sin a)
    const FxTw* tw;       // shared-memory copy of the twiddles
    const C64* tw64;      // double twiddles (global), for the plain form
};

// Template of one candidate: bin values of the channels in natural DFT order
// at sw(index).  buf: the channels' buffers, stride elements apart.
template <int NT>
__device__ __forceinline__ void template_any(const CandT& c, const Geo64& g, const OrbitTables64& tab, const FxTab& ft,
                                             C64* buf, int stride, bool t3, int lane) {
    if (c.tier < 0) {
        template_plain<NT>(c, g, tab, ft.tw64, buf, buf + stride, t3 ? buf + 2 * stride : nullptr, lane);
        return;
    }
    Z64* z = (Z64*)buf;
    if (c.tier == 0) {
        if (t3) samples_fx<0, true>(c.f, ft.geo, ft.tw, g.krho_q30, g.logN, z, z + stride, z + 2 * stride, lane, NT);
        else samples_fx<0, false>(c.f, ft.geo, ft.tw, g.krho_q30, g.logN, z, z + stride, nullptr, lane, NT);
    } else {
        if (t3) samples_fx<1, true>(c.f, ft.geo, ft.tw, g.krho_q30, g.logN, z, z + stride, z + 2 * stride, lane, NT);
        else samples_fx<1, false>(c.f, ft.geo, ft.tw, g.krho_q30, g.logN, z, z + stride, nullptr, lane, NT);
    }
    sync_nt<NT>();
    const double sc[3] = {c.sA, c.sE, c.sT};
    fft_fx<NT>(z, stride, t3 ? 3 : 2, g.logN, ft.tw, sc, lane);
}

__device__ __forceinline__ double warp_sum(double v) {
    for (int o = 16; o > 0; o >>= 1) v += __shfl_xor_sync(0xffffffffu, v, o);
    return v;
}

// the CTA's copy of the fixed-point twiddles
__device__ __forceinline__ void load_twiddles(const FxTw* __restrict__ g, FxTw* tw) {
    const int4* src = (const int4*)g;
    for (int i = threadIdx.x; i < kTwiddles; i += blockDim.x) ((int4*)tw)[i] = __ldg(src + i);
}

__device__ __forceinline__ Geo64 geometry64(int N, double T, double fstar, double arm_c, int krho_q30) {
    Geo64 g;
    g.N = N;
    g.logN = 31 - __clz(N);
    g.T = T;
    g.T_over_N = T / (double)N;
    g.inv_fstar = 1.0 / fstar;
    g.scale = T / (2.0 * (double)N);
    g.arm_c = arm_c;
    g.krho_q30 = krho_q30;
    return g;
}

}  // namespace
}  // namespace gb
