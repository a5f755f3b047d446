// fp64.cu -- double-precision path: template by the fast/slow decomposition,
// warp FFT in shared memory, window inner products, log-likelihood (Eq. 2).
//
// Mapping: one CTA per tile (window, <= 32*WARPS candidates).  Each warp owns
// up to 32 consecutive candidates: their per-candidate setup (sky basis,
// polarisation tensor, carrier bin) is computed lane-parallel, one candidate
// per lane, into shared memory; then the warp evaluates them one after the
// other with the N samples strided across the 32 lanes, an in-place FFT in the
// warp's shared-memory buffer, and the window inner products with a warp
// reduction.
//
// The slow part and the FFT run in 64-bit fixed point (fx64.cuh), which has
// more fractional bits than a double and runs on GB300's integer pipe, while
// the FP64 pipe (one warp instruction per 64 clocks and scheduler) is left
// with the set-up, the conversion of the bins and the inner products.
// Candidates outside the fixed-point ranges (f0 <= 0, f above 1.3 f*, a drift
// of more than f0/1024 over the observation, ...) take the plain double form.
//
// Measured on GB300, 16 windows x 10,000 candidates (N = 128, 256): 23.4 ms with
// every step in double (FP64 pipe 87% busy), 3.9 ms in this form; templates of
// 8,192 candidates at N = 256: 2.07 -> 0.38 ms.  Per 32 samples the kernel
// issues 3,140 warp instructions, half of them on the multiply pipe (74% busy
// on a full SM, FP64 pipe 55%), so integer products bound it.  Error of the
// templates against the model in long double, at 0.3-23 mHz: 4e-16 ... 5e-15 of
// their norm, where the double form had 5e-15 ... 3e-14 (arm vectors from
// differences of positions of 1 AU, phases rounded at several cycles).
#include <cmath>

#include "fx64.cuh"
#include "gb_internal.cuh"

namespace gb {
namespace {

constexpr int kWarps64 = 4;
// Candidates a warp sets up at a time, one per lane: the set-up is FP64 work
// whose cost does not depend on the lanes in use (8 in place of 16: 4.33 -> 4.58
// ms for the 160,000 candidates below), while 32 would cost a resident CTA.
constexpr int kCap64 = 16;
// Resident CTAs per SM the kernels are compiled for (168 registers; 2 or 4
// CTAs: 3 and 5% slower).
constexpr int kMinCtas64 = 3;

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
// one lane, one candidate
__device__ void setup_lane(const double* th, const Geo64& g, CandT& c) {
    const double delta = carrier64(th, g.T, c);
    FxTrig t;
    double ii;
    sincos(th[2], &t.sb, &t.cb);
    sincos(th[3], &t.sl, &t.cl);
    sincos(2.0 * th[6], &t.s2, &t.c2);
    sincos(th[5], &ii, &t.ci);
    sincos(kPi * th[0] * g.arm_c, &t.sa, &t.ca);
    setup_t(th, g, delta, t, c);
}
// one candidate by a whole warp: the five sines and cosines on five lanes (the
// double sincos is a long dependent chain), the rest on lane 0
__device__ void setup_warp(const double* th, const Geo64& g, CandT& c, int lane) {
    const double x = lane == 0 ? th[2] : lane == 1 ? th[3] : lane == 2 ? 2.0 * th[6] : lane == 3 ? th[5] : kPi * th[0] * g.arm_c;
    double sn, cs;
    sincos(x, &sn, &cs);
    FxTrig t;
    t.sb = __shfl_sync(0xffffffffu, sn, 0);
    t.cb = __shfl_sync(0xffffffffu, cs, 0);
    t.sl = __shfl_sync(0xffffffffu, sn, 1);
    t.cl = __shfl_sync(0xffffffffu, cs, 1);
    t.s2 = __shfl_sync(0xffffffffu, sn, 2);
    t.c2 = __shfl_sync(0xffffffffu, cs, 2);
    t.ci = __shfl_sync(0xffffffffu, cs, 3);
    t.sa = __shfl_sync(0xffffffffu, sn, 4);
    t.ca = __shfl_sync(0xffffffffu, cs, 4);
    if (lane == 0) {
        const double delta = carrier64(th, g.T, c);
        setup_t(th, g, delta, t, c);
    }
}

// Index of element e in a transform buffer: the low three bits XORed with the
// higher groups of three, so that eight lanes whose indices differ in any
// three neighbouring bits (every stage of the transform, the bit-reversed
// stores and the reads in order) meet eight different 16-byte bank groups.
__device__ __forceinline__ int sw(int e) { return e ^ ((e >> 3) & 7) ^ ((e >> 6) & 7) ^ ((e >> 9) & 1); }

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
    c.J = xmax <= 2.35 ? 16 : 0;
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
// real and imaginary parts (Horner in y = -4X^2); J = 0: direct evaluation
template <int J>
__device__ __forceinline__ C64 transfer64(double X) {
    if constexpr (J == 0) {
        double sX, cX;
        sincos(X, &sX, &cX);
        const double sinc = (X != 0.0) ? sX / X : 1.0;
        return {sinc * cX, -(sinc * sX)};
    } else {
        const double y = -4.0 * X * X;
        double re = kInvFact64[2 * J + 1], im = kInvFact64[2 * J + 2];
#pragma unroll
        for (int j = J - 1; j >= 0; --j) {
            re = fma(re, y, kInvFact64[2 * j + 1]);
            im = fma(im, y, kInvFact64[2 * j + 2]);
        }
        return {re, -2.0 * X * im};
    }
}

// -i a sinc(X) exp(-iX) G exp(i Psi)
template <int J>
__device__ __forceinline__ C64 link64(double a, double X, C64 G, C64 rx) {
    const C64 t = transfer64<J>(X);
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
template <int NT>
__device__ __forceinline__ void sync_nt() {
    if (NT == 32) __syncwarp();
    else __syncthreads();
}

template <int J, int NT>
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
            z01 = link64<J>(a, a * (1.0 - kn), G, rx[1]);
            z10 = link64<J>(a, a * (1.0 + kn), G, rx[0]);
        }
        {
            const double nx = tab.arm[3 * N + n], ny = tab.arm[4 * N + n], nz = tab.arm[5 * N + n];
            const double kn = c.k[0] * nx + c.k[1] * ny + c.k[2] * nz;
            const C64 G = nHn(c, nx, ny, nz);
            z12 = link64<J>(a, a * (1.0 - kn), G, rx[2]);
            z21 = link64<J>(a, a * (1.0 + kn), G, rx[1]);
        }
        {
            const double nx = tab.arm[6 * N + n], ny = tab.arm[7 * N + n], nz = tab.arm[8 * N + n];
            const double kn = c.k[0] * nx + c.k[1] * ny + c.k[2] * nz;
            const C64 G = nHn(c, nx, ny, nz);
            z20 = link64<J>(a, a * (1.0 - kn), G, rx[0]);
            z02 = link64<J>(a, a * (1.0 + kn), G, rx[2]);
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
    if (c.d.J == 16) template64<16, NT>(c.d, g, tab, tw, bufA, bufE, bufT, lane);
    else template64<0, NT>(c.d, g, tab, tw, bufA, bufE, bufT, lane);
    for (int i = lane; i < g.N; i += NT) {
        bufA[i] = cscale(bufA[i], g.scale);
        bufE[i] = cscale(bufE[i], g.scale);
        if (bufT) bufT[i] = cscale(bufT[i], g.scale);
    }
    sync_nt<NT>();
}

// a fixed-point complex value, or, after the last stage, the bits of two doubles
struct alignas(16) Z64 {
    fx x, y;
};
__device__ __forceinline__ Z64 zadd(Z64 a, Z64 b) { return {a.x + b.x, a.y + b.y}; }
__device__ __forceinline__ Z64 zsub(Z64 a, Z64 b) { return {a.x - b.x, a.y - b.y}; }
__device__ __forceinline__ Z64 zmi(Z64 a) { return {a.y, -a.x}; }   // times -i
__device__ __forceinline__ Z64 zmul(Z64 a, const FxTw& w) {   // times co - i si
    const Bx r = bal(a.x), i = bal(a.y), mr = bal(-a.x);
    Dot re = mul(r, w.co), im = mul(mr, w.si);
    re.add(i, w.si);
    im.add(i, w.co);
    return {re.get<2>(), im.get<2>()};
}
__device__ __forceinline__ Z64 zout(Z64 a, double s, bool last) {
    if (!last) return a;
    return {__double_as_longlong((double)a.x * s), __double_as_longlong((double)a.y * s)};
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

// In-place FFT of nch buffers (stride elements apart): bit-reversed input,
// natural order output as doubles times sc[ch].  Radix-2 decimation in time,
// two stages at a time (three twiddle products per four elements; the first
// two stages have none), the odd stage last.  Bound by the integer products
// of the twiddles.
template <int NT>
__device__ void fft_fx(Z64* buf, int stride, int nch, int lg, const FxTw* tw, const double* sc, int lane) {
    const int N = 1 << lg;
    for (int q = lane; q < N / 4; q += NT) {
        const int i0 = sw(4 * q), i1 = sw(4 * q + 1), i2 = sw(4 * q + 2), i3 = sw(4 * q + 3);
        for (int ch = 0; ch < nch; ++ch) {
            Z64* p = buf + (size_t)ch * stride;
            const Z64 x0 = p[i0], x1 = p[i1], x2 = p[i2], x3 = p[i3];
            const Z64 a = zadd(x0, x1), b = zsub(x0, x1), c = zadd(x2, x3), d = zmi(zsub(x2, x3));
            p[i0] = zadd(a, c);
            p[i1] = zadd(b, d);
            p[i2] = zsub(a, c);
            p[i3] = zsub(b, d);
        }
    }
    sync_nt<NT>();
    int s = 2;
    for (; s + 2 <= lg; s += 2) {
        const bool last = s + 2 == lg;
        const int h = 1 << s;
        for (int q = lane; q < N / 4; q += NT) {
            const int j = q & (h - 1), e = ((q >> s) << (s + 2)) + j;
            const int i0 = sw(e), i1 = sw(e + h), i2 = sw(e + 2 * h), i3 = sw(e + 3 * h);
            // exp(-2 pi i m j / 4h), m = 2, 1, 3; entry k >= 512 is minus entry k - 512
            const FxTw w1 = tw[j << (9 - s)], w2 = tw[j << (8 - s)];
            const int k3 = (3 * j) << (8 - s);
            const FxTw w3 = tw[k3 & 511];
            for (int ch = 0; ch < nch; ++ch) {
                Z64* p = buf + (size_t)ch * stride;
                const Z64 x0 = p[i0], x1 = zmul(p[i1], w1), x2 = zmul(p[i2], w2);
                Z64 x3 = zmul(p[i3], w3);
                if (k3 & 512) x3 = {-x3.x, -x3.y};
                const Z64 a = zadd(x0, x1), b = zsub(x0, x1), c = zadd(x2, x3), d = zmi(zsub(x2, x3));
                p[i0] = zout(zadd(a, c), sc[ch], last);
                p[i1] = zout(zadd(b, d), sc[ch], last);
                p[i2] = zout(zsub(a, c), sc[ch], last);
                p[i3] = zout(zsub(b, d), sc[ch], last);
            }
        }
        sync_nt<NT>();
    }
    if (s < lg) {
        const int h = 1 << s;
        for (int q = lane; q < N / 2; q += NT) {
            const int i0 = sw(q), i1 = sw(q + h);
            const FxTw w = tw[q << (9 - s)];
            for (int ch = 0; ch < nch; ++ch) {
                Z64* p = buf + (size_t)ch * stride;
                const Z64 a = p[i0], b = zmul(p[i1], w);
                p[i0] = zout(zadd(a, b), sc[ch], true);
                p[i1] = zout(zsub(a, b), sc[ch], true);
            }
        }
        sync_nt<NT>();
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

// <d|d> of window `win` over the whole block, in a fixed order (deterministic);
// every thread returns the same value.  `red` holds kWarps64 doubles.
__device__ __forceinline__ double window_dd64(const gb_window_t& win, bool useT, const C64* __restrict__ dA,
                                              const C64* __restrict__ dE, const double* __restrict__ wA,
                                              const double* __restrict__ wE, const C64* __restrict__ dT,
                                              const double* __restrict__ wT, double T, double* red) {
    const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
    double acc = 0.0;
    for (int i = threadIdx.x; i < win.W; i += blockDim.x) {
        const C64 a = dA[win.data_off + i], e = dE[win.data_off + i];
        acc += wA[win.data_off + i] * (a.x * a.x + a.y * a.y) + wE[win.data_off + i] * (e.x * e.x + e.y * e.y);
        if (useT) {
            const C64 t = dT[win.data_off + i];
            acc += wT[win.data_off + i] * (t.x * t.x + t.y * t.y);
        }
    }
    acc = warp_sum(acc);
    if (lane == 0) red[warp] = acc;
    __syncthreads();
    double dd = 0.0;
    for (int w = 0; w < kWarps64; ++w) dd += red[w];
    return dd * (4.0 / T);
}

// Window inner products of one computed template (one warp, in a fixed
// order) and Eq. 2; lane 0 writes output row `row`.
__device__ __forceinline__ void ip64(const CandT& c, int64_t row, const Geo64& g, const C64* bufA, const C64* bufE,
                                     const C64* bufT, const gb_window_t& win, double dd, const C64* __restrict__ dA,
                                     const C64* __restrict__ dE, const double* __restrict__ wA,
                                     const double* __restrict__ wE, const C64* __restrict__ dT,
                                     const double* __restrict__ wT, double* __restrict__ logL,
                                     double* __restrict__ dh_out, double* __restrict__ hh_out,
                                     double* __restrict__ dhi_out, int lane) {
    const double T = g.T;
    const int64_t half = win.N / 2;
    double sdh = 0.0, shh = 0.0, sdhi = 0.0;
    for (int m = lane; m < win.N; m += 32) {
        const int64_t kk = c.q - half + m - win.k0;
        if (kk >= 0 && kk < win.W) {
            const int idx = sw((m + (int)half) & (win.N - 1));
            const C64 hA = bufA[idx], hE = bufE[idx];
            const C64 a = dA[win.data_off + kk], e = dE[win.data_off + kk];
            const double wa = wA[win.data_off + kk], we = wE[win.data_off + kk];
            sdh += wa * (a.x * hA.x + a.y * hA.y) + we * (e.x * hE.x + e.y * hE.y);
            shh += wa * (hA.x * hA.x + hA.y * hA.y) + we * (hE.x * hE.x + hE.y * hE.y);
            if (dhi_out) sdhi += wa * (a.y * hA.x - a.x * hA.y) + we * (e.y * hE.x - e.x * hE.y);
            if (bufT) {
                const C64 hT = bufT[idx], t = dT[win.data_off + kk];
                const double wt = wT[win.data_off + kk];
                sdh += wt * (t.x * hT.x + t.y * hT.y);
                shh += wt * (hT.x * hT.x + hT.y * hT.y);
                if (dhi_out) sdhi += wt * (t.y * hT.x - t.x * hT.y);
            }
        }
    }
    sdh = warp_sum(sdh) * (4.0 / T);
    shh = warp_sum(shh) * (4.0 / T);
    if (dhi_out) sdhi = warp_sum(sdhi) * (4.0 / T);
    if (lane == 0) {
        logL[row] = sdh - 0.5 * shh - 0.5 * dd;
        if (dh_out) dh_out[row] = sdh;
        if (hh_out) hh_out[row] = shh;
        if (dhi_out) dhi_out[row] = sdhi;
    }
}

// NaN outputs of a candidate with a non-finite parameter (one thread)
__device__ __forceinline__ void bad64(int64_t row, double* logL, double* dh_out, double* hh_out, double* dhi_out,
                                      int* status) {
    logL[row] = nan("");
    if (dh_out) dh_out[row] = nan("");
    if (hh_out) hh_out[row] = nan("");
    if (dhi_out) dhi_out[row] = nan("");
    atomicOr(status, kStatusNonFinite);
}

// the CTA's copy of the fixed-point twiddles
__device__ __forceinline__ void load_twiddles(const FxTw* __restrict__ g, FxTw* tw) {
    const int4* src = (const int4*)g;
    for (int i = threadIdx.x; i < kTwiddles; i += blockDim.x) ((int4*)tw)[i] = __ldg(src + i);
}

// One candidate (one warp): template, window inner products and Eq. 2; lane 0
// writes output row `row`.
__device__ __forceinline__ void eval64(const CandT& c, int64_t row, const Geo64& g, const OrbitTables64& tab,
                                       const FxTab& ft, C64* buf, int stride, bool t3, const gb_window_t& win,
                                       double dd, const C64* __restrict__ dA, const C64* __restrict__ dE,
                                       const double* __restrict__ wA, const double* __restrict__ wE,
                                       const C64* __restrict__ dT, const double* __restrict__ wT,
                                       double* __restrict__ logL, double* __restrict__ dh_out,
                                       double* __restrict__ hh_out, double* __restrict__ dhi_out, int* status,
                                       int lane) {
    if (c.bad) {
        if (lane == 0) bad64(row, logL, dh_out, hh_out, dhi_out, status);
        return;
    }
    template_any<32>(c, g, tab, ft, buf, stride, t3, lane);
    ip64(c, row, g, buf, buf + stride, t3 ? buf + 2 * stride : nullptr, win, dd, dA, dE, wA, wE, dT, wT, logL, dh_out, hh_out, dhi_out, lane);
    __syncwarp();
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

// ROWS = false: one CTA per plan tile, the tile's candidates split over the
// warps.  ROWS = true: blockIdx.x is a window and its candidates are the rows
// listed in rows[cand_off + j], j in [row_lo[w], row_hi[w]) (device lists);
// the gridDim.y CTAs of a window take them one at a time (few rows, each
// spread over a CTA, for latency).
template <bool ROWS>
__global__ void __launch_bounds__(kWarps64 * 32, kMinCtas64) loglik64_kernel(
    const gb_window_t* __restrict__ wins, const Tile* __restrict__ tiles, TabSet64 tabs,
    const C64* __restrict__ tw_g, TabSetFx fxt, double T, double fstar, const C64* __restrict__ dA,
    const C64* __restrict__ dE, const double* __restrict__ wA, const double* __restrict__ wE,
    const double* __restrict__ theta, double* __restrict__ logL, double* __restrict__ dh_out,
    double* __restrict__ hh_out, double* __restrict__ dhi_out, const C64* __restrict__ dT,
    const double* __restrict__ wT, int* status, int n_max, const int32_t* __restrict__ rows,
    const int32_t* __restrict__ row_lo, const int32_t* __restrict__ row_hi, const int* __restrict__ gate) {
    if (ROWS && gate && *gate == 0) return;
    extern __shared__ __align__(16) unsigned char smem_raw[];
    FxTw* tw = (FxTw*)smem_raw;                                 // kTwiddles
    double* red = (double*)(tw + kTwiddles);                    // kWarps64
    CandT* cands = (CandT*)(red + kWarps64);                    // kWarps64 * kCap64
    C64* bufs = (C64*)(cands + kWarps64 * kCap64);              // kWarps64 * (2 or 3) * n_max
    const int nch = dT ? 3 : 2;

    const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
    Tile tile{};
    int lo = 0, hi = 0;
    if (ROWS) {
        tile.win = blockIdx.x;
    } else {
        tile = tiles[blockIdx.x];
    }
    const gb_window_t win = wins[tile.win];
    if (ROWS) {
        lo = max(row_lo[tile.win], 0);
        hi = min(row_hi[tile.win], win.n_cand);
        if (lo >= hi) return;                                   // nothing listed (block-uniform)
    }
    load_twiddles(fxt.tw, tw);

    // T enters windows whose lowest frequency is at least f*/2
    const bool useT = dT != nullptr && (double)win.k0 / T >= 0.5 * fstar;
    const double dd = window_dd64(win, useT, dA, dE, wA, wE, dT, wT, T, red);

    const Geo64 g = geometry64(win.N, T, fstar, fxt.arm_c, fxt.krho_q30);
    const OrbitTables64 tab = tabs.t[g.logN - 5];
    const FxTab ft{fxt.geo[g.logN - 5], tw, tw_g};
    C64* buf = bufs + (size_t)warp * nch * n_max;
    CandT* mycand = cands + warp * kCap64;

    if (!ROWS) {
        const int64_t tlen = tile.c_end - tile.c_begin;
        const int64_t grp = (tlen + kWarps64 - 1) / kWarps64;   // <= 32
        const int64_t c_lo = tile.c_begin + (int64_t)warp * grp;
        const int64_t c_hi = min(tile.c_end, c_lo + grp);
        for (int64_t c0 = c_lo; c0 < c_hi; c0 += kCap64) {
            const int cnt = (int)min((int64_t)kCap64, c_hi - c0);
            if (lane < cnt) setup_lane(theta + 8 * (c0 + lane), g, mycand[lane]);
            __syncwarp();
            for (int i = 0; i < cnt; ++i)
                eval64(mycand[i], c0 + i, g, tab, ft, buf, n_max, useT, win, dd, dA, dE, wA, wE, dT, wT, logL, dh_out,
                       hh_out, dhi_out, status, lane);
            __syncwarp();
        }
    } else {
        // one listed row at a time for the whole CTA (entries lo + y, lo + y
        // + Y, ... for CTA y of the window's Y): the template over all the
        // CTA's threads, the inner products in warp 0 in a warp's order
        for (int slot = lo + (int)blockIdx.y; slot < hi; slot += (int)gridDim.y) {
            const int64_t row = rows[win.cand_off + slot];
            if (row < win.cand_off || row >= win.cand_off + win.n_cand) continue;   // not this window's row
            if (warp == 0) setup_warp(theta + 8 * row, g, cands[0], lane);
            __syncthreads();
            if (cands[0].bad) {
                if (threadIdx.x == 0) bad64(row, logL, dh_out, hh_out, dhi_out, status);
            } else {
                template_any<kWarps64 * 32>(cands[0], g, tab, ft, bufs, n_max, false, threadIdx.x);
                if (warp == 0)
                    ip64(cands[0], row, g, bufs, bufs + n_max, nullptr, win, dd, dA, dE, wA, wE, nullptr, nullptr, logL, dh_out,
                         hh_out, dhi_out, lane);
            }
            __syncthreads();
        }
    }
}

__global__ void __launch_bounds__(kWarps64 * 32, kMinCtas64) waveform64_kernel(
    OrbitTables64 tab, const C64* __restrict__ tw_g, TabSetFx fxt, double T, double fstar, int N,
    const double* __restrict__ theta, int64_t B, int group, C64* __restrict__ hA, C64* __restrict__ hE,
    C64* __restrict__ hT, int64_t* __restrict__ q_out, int* status) {
    extern __shared__ __align__(16) unsigned char smem_raw[];
    FxTw* tw = (FxTw*)smem_raw;
    CandT* cands = (CandT*)(tw + kTwiddles);
    C64* bufs = (C64*)(cands + kWarps64 * kCap64);
    const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
    load_twiddles(fxt.tw, tw);
    __syncthreads();
    const Geo64 g = geometry64(N, T, fstar, fxt.arm_c, fxt.krho_q30);
    const FxTab ft{fxt.geo[g.logN - 5], tw, tw_g};
    C64* buf = bufs + (size_t)warp * (hT ? 3 : 2) * N;
    CandT* mycand = cands + warp * kCap64;
    const int64_t c_lo = ((int64_t)blockIdx.x * kWarps64 + warp) * group;
    const int64_t c_hi = min(B, c_lo + group);   // group <= kCap64
    if (c_lo >= c_hi) return;
    if (c_lo + lane < c_hi) setup_lane(theta + 8 * (c_lo + lane), g, mycand[lane]);
    __syncwarp();
    for (int64_t b = c_lo; b < c_hi; ++b) {
        const CandT& c = mycand[b - c_lo];
        C64* outA = hA + b * N;
        C64* outE = hE + b * N;
        if (c.bad) {
            for (int m = lane; m < N; m += 32) {
                outA[m] = outE[m] = C64{nan(""), nan("")};
                if (hT) hT[b * N + m] = C64{nan(""), nan("")};
            }
            if (lane == 0) {
                q_out[b] = 0;
                atomicOr(status, kStatusNonFinite);
            }
            continue;
        }
        template_any<32>(c, g, tab, ft, buf, N, hT != nullptr, lane);
        for (int m = lane; m < N; m += 32) {
            const int idx = sw((m + N / 2) & (N - 1));
            outA[m] = buf[idx];
            outE[m] = buf[N + idx];
            if (hT) hT[b * N + m] = buf[2 * N + idx];
        }
        if (lane == 0) q_out[b] = c.q;
        __syncwarp();
    }
}

// Window inner product <x|y> = (4/T) Re sum_k w_k x_k y_k* of two templates
// (or data, y) over the window's bins, block-wide in a fixed order.  A
// template is given by its buffers of bin values (natural order, at sw(index))
// and carrier bin; bins it does not reach count zero.  `red` holds kWarps64
// doubles.
struct WinTpl {
    const C64* A;
    const C64* E;
    long long q;
};
__device__ __forceinline__ C64 tpl_at(const WinTpl& t, int N, long long k) {
    const long long m = k - (t.q - N / 2);
    if (m < 0 || m >= N) return {0.0, 0.0};
    return t.A[sw((int)((m + N / 2) & (N - 1)))];
}
__device__ __forceinline__ C64 tpl_at_e(const WinTpl& t, int N, long long k) {
    const long long m = k - (t.q - N / 2);
    if (m < 0 || m >= N) return {0.0, 0.0};
    return t.E[sw((int)((m + N / 2) & (N - 1)))];
}
__device__ double block_sum64(double v, double* red) {
    const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
    v = warp_sum(v);
    __syncthreads();
    if (lane == 0) red[warp] = v;
    __syncthreads();
    double s = 0.0;
    for (int w = 0; w < kWarps64; ++w) s += red[w];
    return s;
}
// <x|y> with x a template and y a template (yt) or the data (yt == nullptr)
__device__ double win_inner(const WinTpl& x, const WinTpl* yt, const gb_window_t& win, const C64* __restrict__ dA,
                            const C64* __restrict__ dE, const double* __restrict__ wA, const double* __restrict__ wE,
                            double T, double* red) {
    double acc = 0.0;
    for (int i = threadIdx.x; i < win.W; i += blockDim.x) {
        const long long k = win.k0 + i;
        const C64 xa = tpl_at(x, win.N, k), xe = tpl_at_e(x, win.N, k);
        C64 ya, ye;
        if (yt) {
            ya = tpl_at(*yt, win.N, k);
            ye = tpl_at_e(*yt, win.N, k);
        } else {
            ya = dA[win.data_off + i];
            ye = dE[win.data_off + i];
        }
        acc += wA[win.data_off + i] * (xa.x * ya.x + xa.y * ya.y) + wE[win.data_off + i] * (xe.x * ye.x + xe.y * ye.y);
    }
    return block_sum64(acc, red) * (4.0 / T);
}

// Gram matrix G_ij = <s_i|s_j>, b_i = <d|s_i> and the multi-signal SNR
// rho = sum_i b_i / sqrt(sum_ij G_ij) (Eq. 11) of each window's sources (one
// CTA per window; the sources are the window's candidate rows).  Template i
// is held in buffer P while the templates j > i pass through buffer Q.
__global__ void __launch_bounds__(kWarps64 * 32, kMinCtas64) multi_gram_kernel(
    const gb_window_t* __restrict__ wins, TabSet64 tabs, const C64* __restrict__ tw_g, TabSetFx fxt, double T,
    double fstar,
    const C64* __restrict__ dA, const C64* __restrict__ dE, const double* __restrict__ wA,
    const double* __restrict__ wE, const double* __restrict__ theta, int kmax, double* __restrict__ gram,
    double* __restrict__ dh_out, double* __restrict__ rho_out, int* status, int n_max) {
    extern __shared__ __align__(16) unsigned char smem_raw[];
    FxTw* tw = (FxTw*)smem_raw;                 // kTwiddles
    double* red = (double*)(tw + kTwiddles);    // kWarps64
    CandT* cand = (CandT*)(red + kWarps64);     // 2
    C64* PA = (C64*)(cand + 2);                 // 4 buffers of n_max
    C64* QA = PA + 2 * n_max;
    const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
    const gb_window_t win = wins[blockIdx.x];
    const int K = win.n_cand;
    double* G = gram + (size_t)blockIdx.x * kmax * kmax;
    load_twiddles(fxt.tw, tw);
    const Geo64 g = geometry64(win.N, T, fstar, fxt.arm_c, fxt.krho_q30);
    const OrbitTables64 tab = tabs.t[g.logN - 5];
    const FxTab ft{fxt.geo[g.logN - 5], tw, tw_g};
    const bool data = dA != nullptr;
    double sum_b = 0.0, sum_g = 0.0;
    bool bad_any = false;
    for (int i = 0; i < K; ++i) {
        __syncthreads();
        if (warp == 0) setup_warp(theta + 8 * (win.cand_off + i), g, cand[0], lane);
        __syncthreads();
        const bool bad_i = cand[0].bad;
        if (!bad_i) template_any<kWarps64 * 32>(cand[0], g, tab, ft, PA, n_max, false, threadIdx.x);
        __syncthreads();
        const WinTpl P{PA, PA + n_max, cand[0].q};
        const double gii = bad_i ? nan("") : win_inner(P, &P, win, dA, dE, wA, wE, T, red);
        const double bi = bad_i || !data ? nan("") : win_inner(P, nullptr, win, dA, dE, wA, wE, T, red);
        if (threadIdx.x == 0) {
            G[i * kmax + i] = gii;
            if (dh_out) dh_out[win.cand_off + i] = bi;
            if (bad_i) atomicOr(status, kStatusNonFinite);
            sum_b += bi;
            sum_g += gii;
            bad_any |= bad_i;
        }
        for (int j = i + 1; j < K; ++j) {
            __syncthreads();
            if (warp == 0) setup_warp(theta + 8 * (win.cand_off + j), g, cand[1], lane);
            __syncthreads();
            const bool bad_j = cand[1].bad;
            if (!bad_j) template_any<kWarps64 * 32>(cand[1], g, tab, ft, QA, n_max, false, threadIdx.x);
            __syncthreads();
            const WinTpl Q{QA, QA + n_max, cand[1].q};
            const double gij = bad_i || bad_j ? nan("") : win_inner(P, &Q, win, dA, dE, wA, wE, T, red);
            if (threadIdx.x == 0) {
                G[i * kmax + j] = gij;
                G[j * kmax + i] = gij;
                sum_g += 2.0 * gij;
            }
        }
    }
    if (threadIdx.x == 0 && rho_out)
        rho_out[blockIdx.x] = (K == 0 || bad_any || !data) ? nan("") : sum_b / sqrt(sum_g);
}

}  // namespace

static size_t smem64_loglik(int n_max, int nch) {
    return sizeof(FxTw) * kTwiddles + sizeof(double) * kWarps64 + sizeof(CandT) * kWarps64 * kCap64 +
           sizeof(C64) * kWarps64 * nch * (size_t)n_max;
}

int launch_loglik_fp64(gb_ctx* ctx, const Plan& plan, const double* dA, const double* dE,
                       const double* wA, const double* wE, const double* theta, double* logL,
                       double* dh, double* hh, double* dh_im, const double* dT, const double* wT,
                       cudaStream_t s) {
    if (plan.n_tiles == 0) return GB_OK;
    const size_t smem = smem64_loglik(plan.n_max, dT ? 3 : 2);
    cudaError_t e = cudaFuncSetAttribute(loglik64_kernel<false>, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)smem);
    if (e != cudaSuccess) return cuda_error(ctx, e, "loglik64: smem attribute");
    loglik64_kernel<false><<<plan.n_tiles, kWarps64 * 32, smem, s>>>(
        plan.d_win, plan.d_tiles, tabset64(ctx), (const C64*)ctx->d_tw64, tabset_fx(ctx), ctx->obs.T_obs,
        transfer_frequency(ctx), (const C64*)dA, (const C64*)dE, wA, wE, theta, logL, dh, hh,
        dh_im, (const C64*)dT, wT, ctx->d_status, plan.n_max, nullptr, nullptr, nullptr, nullptr);
    ++ctx->launches;
    e = cudaGetLastError();
    if (e != cudaSuccess) return cuda_error(ctx, e, "loglik64 launch");
    return GB_OK;
}

int launch_loglik_rows64(gb_ctx* ctx, const gb_window_t* d_win, int n_win, int n_max, int ctas_per_win,
                         const double* dA, const double* dE, const double* wA, const double* wE, const double* theta,
                         const int32_t* rows, const int32_t* row_lo, const int32_t* row_hi, double* logL,
                         double* dh, double* hh, const int* gate, cudaStream_t s) {
    if (n_win == 0) return GB_OK;
    const size_t smem = smem64_loglik(n_max, 2);
    cudaError_t e = cudaFuncSetAttribute(loglik64_kernel<true>, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)smem);
    if (e != cudaSuccess) return cuda_error(ctx, e, "loglik64 rows: smem attribute");
    const dim3 grid((unsigned)n_win, (unsigned)(ctas_per_win < 1 ? 1 : ctas_per_win));
    loglik64_kernel<true><<<grid, kWarps64 * 32, smem, s>>>(
        d_win, nullptr, tabset64(ctx), (const C64*)ctx->d_tw64, tabset_fx(ctx), ctx->obs.T_obs, transfer_frequency(ctx),
        (const C64*)dA, (const C64*)dE, wA, wE, theta, logL, dh, hh, nullptr, nullptr, nullptr, ctx->d_status,
        n_max, rows, row_lo, row_hi, gate);
    ++ctx->launches;
    e = cudaGetLastError();
    if (e != cudaSuccess) return cuda_error(ctx, e, "loglik64 rows launch");
    return GB_OK;
}

int launch_waveform_fp64(gb_ctx* ctx, const double* theta, int64_t B, int N, double* hA, double* hE,
                         double* hT, int64_t* q, cudaStream_t s) {
    if (B == 0) return GB_OK;
    const size_t smem = sizeof(FxTw) * kTwiddles + sizeof(CandT) * kWarps64 * kCap64 +
                        sizeof(C64) * kWarps64 * (hT ? 3 : 2) * (size_t)N;
    cudaError_t e = cudaFuncSetAttribute(waveform64_kernel, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)smem);
    if (e != cudaSuccess) return cuda_error(ctx, e, "waveform64: smem attribute");
    int sms = 152;
    cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, ctx->device);
    int64_t group = (B + (int64_t)sms * kWarps64 * 2 - 1) / ((int64_t)sms * kWarps64 * 2);
    group = group < 1 ? 1 : group > kCap64 ? kCap64 : group;
    const int64_t blocks = (B + group * kWarps64 - 1) / (group * kWarps64);
    waveform64_kernel<<<(unsigned)blocks, kWarps64 * 32, smem, s>>>(
        tables64(ctx, N), (const C64*)ctx->d_tw64, tabset_fx(ctx), ctx->obs.T_obs, transfer_frequency(ctx), N,
        theta, B, (int)group, (C64*)hA, (C64*)hE, (C64*)hT, q, ctx->d_status);
    ++ctx->launches;
    e = cudaGetLastError();
    if (e != cudaSuccess) return cuda_error(ctx, e, "waveform64 launch");
    return GB_OK;
}

int launch_multi_gram(gb_ctx* ctx, const gb_window_t* d_win, int n_win, int n_max, const double* dA,
                      const double* dE, const double* wA, const double* wE, const double* theta, int kmax,
                      double* gram, double* dh, double* rho, cudaStream_t s) {
    if (n_win == 0) return GB_OK;
    const size_t smem = sizeof(FxTw) * kTwiddles + sizeof(double) * kWarps64 + sizeof(CandT) * 2 +
                        sizeof(C64) * 4 * (size_t)n_max;
    cudaError_t e = cudaFuncSetAttribute(multi_gram_kernel, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)smem);
    if (e != cudaSuccess) return cuda_error(ctx, e, "multi_gram: smem attribute");
    multi_gram_kernel<<<n_win, kWarps64 * 32, smem, s>>>(d_win, tabset64(ctx), (const C64*)ctx->d_tw64, tabset_fx(ctx), ctx->obs.T_obs,
                                                         transfer_frequency(ctx), (const C64*)dA, (const C64*)dE, wA,
                                                         wE, theta, kmax, gram, dh, rho, ctx->d_status, n_max);
    ++ctx->launches;
    e = cudaGetLastError();
    if (e != cudaSuccess) return cuda_error(ctx, e, "multi_gram launch");
    return GB_OK;
}

}  // namespace gb
