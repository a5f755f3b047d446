// fx64.cuh -- the slow part of a candidate in 64-bit fixed point, for the FP64
// path.
//
// GB300 issues one FP64 warp instruction per 64 clocks and scheduler (measured
// 64-75), a 32 x 32 -> 64-bit integer multiply-add (IMAD.WIDE) every 4 and an
// add every clock, and the two pipes overlap.  Every quantity of the slow part
// but the amplitude is bounded, so it is computed as 64-bit integers scaled by
// a power of two (Qk: value 2^-k per unit): a product is three IMAD.WIDE and a
// few adds, about 20 clocks, and keeps 58 to 62 fractional bits where a double
// keeps 53.
//
// The response is taken in its symmetric form.  With a = pi f L/c, b = a k.n of
// an arm n (emitter i, receiver j; n = (x_j - x_i)/L) and k.rho_i + k.rho_j =
// -k.rho_m (m the third spacecraft: the centroid is the guiding centre), the
// two links of an arm share one phase,
//   z_ij, z_ji = -i a sinc(a -+ b) (n.H.n) exp(-ia + i theta_m) exp(2 pi i P_c),
//   theta_m = pi f k.rho_m = (b_p - b_q)/3 (b_p, b_q the other two arms' b), sum theta = 0,
// and with Sh, Dh = (sinc(a + b) +- sinc(a - b))/2, p = Sh cos a, q = Dh sin a,
// H = (n.H.n) exp(i theta_m),
//   X = 4 a sin(2a) exp(i (2 pi P_c - 4a)) [H_0 (p_0 + i q_0) - H_2 (p_2 - i q_2)],
// Y and Z by rotation of the indices.  So one carrier phase per sample (its
// -4a folded into the phase polynomial), two small-angle phase factors (the
// third is the conjugate of their product) and six real sinc series replace
// three sines and cosines, six complex series and twelve complex products.
// The chirp breaks the symmetry by eps_j = pi fdot k.rho_j (2K + k.rho_j) rad
// at receiver j (below 1e-8): its mean over an arm's two receivers joins
// theta_m, its difference Delta gives dp = Sh sin a Delta/2, dq = Dh cos a
// Delta/2 to first order.
//
// Everything here also compiles for the host, where tests/test_fx64_host.py
// checks the rounding against long double and that no sum wraps.
#pragma once
#include <math.h>
#include <stdint.h>
#include <string.h>

#ifdef __CUDACC__
#define GB_FX __host__ __device__ __forceinline__
#define GB_FXN __host__ __device__
#else
#define GB_FX inline
#define GB_FXN
#endif

namespace gb {

typedef long long fx;   // a fixed-point value; the comment beside it gives its Q

// an operand split for multiplication: h 2^32 + l with l signed
struct Bx {
    int h, l;
};
GB_FX Bx bal(fx x) {
    return Bx{(int)(x >> 32) + (int)((uint32_t)x >> 31), (int)x};
}
GB_FX fx unbal(Bx b) { return ((fx)b.h << 32) + b.l; }
GB_FX fx wide(int a, int b) { return (fx)a * (fx)b; }
// sums of products: Qa x Qb -> Q(a + b - 64); the low x low parts (a quarter
// of a unit) are dropped
struct Dot {
    fx P, X;
    GB_FX void add(Bx a, Bx b) {
        P += wide(a.h, b.h);
        X += wide(a.h, b.l);
        X += wide(a.l, b.h);
    }
    GB_FX fx get() const { return P + (X >> 32); }
    GB_FX fx get(int s) const {
        const uint64_t t = (uint64_t)(P + (X >> 32));
        return (fx)(s ? (t << s) | ((uint32_t)X >> (32 - s)) : t);
    }
    // shifted left by S: Q(a + b - 64 + S), the lower bits from X
    template <int S>
    GB_FX fx get() const {
        const uint64_t t = (uint64_t)(P + (X >> 32));
        return (fx)((t << S) | ((uint32_t)X >> (32 - S)));
    }
};
GB_FX Dot mul(Bx a, Bx b) { return Dot{wide(a.h, b.h), wide(a.h, b.l) + wide(a.l, b.h)}; }
// product with an operand without low part (u = n/N in Q63, its high word)
GB_FX Dot mulu(Bx a, int u) { return Dot{wide(a.h, u), wide(a.l, u)}; }

// Horner step of 32-bit coefficients: c + r x (r, c in one Q, xh the high word
// of x in Q(64 - S))
template <int S>
GB_FX int step32(int r, int xh, int c) {
    return c + (int)(wide(r, xh) >> (32 - S));
}
// Horner step of 64-bit coefficients: c + r x (r, c in one Q, x in Q(64 - S))
template <int S>
GB_FX fx step64(fx r, Bx x, fx c) {
    const Dot d = mul(bal(r), x);
    return c + (S == 0 ? d.get() : d.get<S == 0 ? 1 : S>());
}

// Series of the response for the link arguments of a tier: x_max = f_max/f*
// <= 1/2 (TIER 0) or 1.3 (TIER 1).  Chebyshev interpolants in X^2 or z^2 over
// the tier's range, in powers of the argument; the terms below 2^-27 of the
// result in 32-bit arithmetic, the rest in Q62.  Interpolation error below
// 1e-17 (TIER 0) and 1e-18.

// The squares are kept in Q64 where they are below 1/2 (TIER 0), in Q62
// otherwise.

// sinc(X)/2 -> Q62, y = X^2
template <int TIER>
GB_FX fx half_sinc(Bx y) {
    if (TIER == 0) {
        fx r = -457508523479112ll + (wide(step32<0>(-7017712, y.h, 775660070), y.h) >> 19);
        r = step64<0>(r, y, 19215358409522656ll);
        r = step64<0>(r, y, -384307168202269651ll);
        return step64<0>(r, y, 2305843009213693908ll);
    }
    int s = step32<2>(12680, y.h, -3525731);
    s = step32<2>(s, y.h, 740591142);
    fx r = -57766228222ll + (wide(s, y.h) >> 31);
    r = step64<2>(r, y, 6354285188083ll);
    r = step64<2>(r, y, -457508533573999ll);
    r = step64<2>(r, y, 19215358410114092ll);
    r = step64<2>(r, y, -384307168202282324ll);
    return step64<2>(r, y, 2305843009213693952ll);
}

// x^2 of x in Q62 as the series take it
template <int TIER>
GB_FX Bx square(Bx x) {
    return bal(TIER == 0 ? mul(x, x).get<4>() : mul(x, x).get<2>());
}

// cos(z/3), sin(z/3) of z in Q62 -> Q62
template <int TIER>
GB_FX void cis_third(fx z, fx& co, fx& si) {
    const Bx zb = bal(z);
    const Bx w = square<TIER>(zb);
    if (TIER == 0) {
        fx r = 2372266470273632ll + (wide(step32<0>(2126806, w.h, -1072530573), w.h) >> 19);
        r = step64<0>(r, w, -256204778801518952ll);
        co = step64<0>(r, w, 4611686018427387894ll);
        r = 158151098022272ll + (wide(step32<0>(1260462, w.h, -817166207), w.h) >> 23);
        r = step64<0>(r, w, -28467197644613427ll);
        r = step64<0>(r, w, 1537228672809129301ll);
        si = mul(bal(r), zb).get<2>();
    } else {
        int s = step32<2>(1129, w.h, -1345124);
        s = step32<2>(s, w.h, 1089555069);
        fx r = -8786172112502ll + (wide(s, w.h) >> 26);
        r = step64<2>(r, w, 2372266470384452ll);
        r = step64<2>(r, w, -256204778801521550ll);
        co = step64<2>(r, w, 4611686018427387904ll);
        r = -418389146563ll + (wide(step32<2>(-650420, w.h, 645659751), w.h) >> 30);
        r = step64<2>(r, w, 158151098025140ll);
        r = step64<2>(r, w, -28467197644613452ll);
        r = step64<2>(r, w, 1537228672809129300ll);
        si = mul(bal(r), zb).get<2>();
    }
}

// Twiddle table entry: cos and sin of 2 pi k/1024 in Q62, k < 512
struct FxTw {
    Bx co, si;
};

// exp(2 pi i ph) for a phase in units of 2^-64 cycles -> Q62: the nearest
// multiple of 1/1024 from the table, the rest (at most 2^-11 cycles) by the
// Taylor series of sin and cos
GB_FX void cis_table(uint64_t ph, const FxTw* tw, fx& co, fx& si) {
    const uint64_t idx = (ph + (1ull << 53)) >> 54;
    const fx r = (fx)(ph - (idx << 54));
    const Bx rho = bal((fx)((uint64_t)r << 9));   // Q62 of the residual over 2^-11 cycles
    const Bx r2 = bal(mul(rho, rho).get<2>());
    const fx s = 14148475504056881ll + (wide(step32<2>(653, r2.h, -1387197337), r2.h) >> 26);
    const fx c = -21703489601094ll + (wide(17023473, r2.h) >> 30);
    const Bx cm = bal(mul(bal(c), r2).get<2>());
    const fx sn = mul(bal(s), rho).get<2>();
    const FxTw t = tw[idx & 511];
    Dot dc = mul(t.co, cm), ds = mul(t.co, bal(sn));
    dc.add(t.si, bal(-sn));
    ds.add(t.si, cm);
    co = unbal(t.co) + dc.get<2>();
    si = unbal(t.si) + ds.get<2>();
    if (idx & 512) {
        co = -co;
        si = -si;
    }
}

// Per-candidate constants
struct alignas(16) CandFx {
    Bx k0, k1, k2, u0, u1, u2, v0, v1;   // Q62
    Bx gpr, gxr, gpi, gxi;               // Q60, n.H.n = (gpr F+ + gxr nu nv) + i (...), unit amplitude
    Bx Kc, Ks;                           // Q62, K / 512 s
    Bx Fc, Fs;                           // Q57 cycles, f0 K
    Bx w2;                               // Q64, 512^2 fdot/2
    Bx c2;                               // Q62 cycles, fdot T^2/2 less its nearest integer c2i
    Bx a1;                               // Q70, a = a0 + a1 u
    Bx w1;                               // Q62, 512 fdot T
    fx a0;                               // Q62
    uint64_t C0, D1;                     // phase at u = 0 and its step per sample (without the chirp), 2^-64 cycles
    fx cc0, cs0;                         // C1(u), S1(u) coefficients: Q62
    fx cc1, cs1;                         // Q63
    fx cc2, cs2;                         // Q64
    int cc3, cc4, cc5, cs3, cs4, cs5;    // Q55
    int FD;                              // Q58, pi fdot (L/c)/3 1024 (of eps)
    int c2i;
    int tsh;                             // left shift of T, which is small at low frequency
    int tier;                            // 0, 1: series tier; -1: outside the fixed-point ranges
    double sA, sE, sT;                   // a channel's bin value per unit of its transform
};

// Sample constants: arm vectors n_01, n_12 and cos, sin of the orbital phase, Q62
struct GeoFx {
    Bx n0x, n0y, n0z, n1x, n1y, n1z, ca, sa;
};

// What a sample's response is made of, before the links are combined.
struct MidFx {
    int u;                     // n/N in Q31
    fx a, b[3];                // a and b = a k.n of the arms, Q62
    fx kn[3];                  // k.n, Q60
    fx nu[3], nv[3];           // n.u, n.v, Q62
    fx K;                      // K / 512 s, Q60
    uint64_t ph;               // carrier phase, 2^-64 cycles
    int ep[3];                 // eps of the receivers, Q56
    fx co[3], si[3];           // exp(i theta) of the arms, Q62
    Bx C1, S1;                 // amplitude polynomials, Q62
};

// krho_q30: (L/c)/(3 1024 s) in Q30
template <int TIER>
GB_FX void middle_fx(const CandFx& c, const GeoFx& g, int krho_q30, int n, int lg, MidFx& m) {
    const int u = m.u = n << (31 - lg);
    // projections of the arms; the third arm closes the triangle
    Dot d = mul(c.k0, g.n0x);
    d.add(c.k1, g.n0y);
    d.add(c.k2, g.n0z);
    const fx kn0 = d.get();   // Q60
    d = mul(c.k0, g.n1x);
    d.add(c.k1, g.n1y);
    d.add(c.k2, g.n1z);
    const fx kn1 = d.get();
    const fx kn2 = -kn0 - kn1;
    m.kn[0] = kn0;
    m.kn[1] = kn1;
    m.kn[2] = kn2;
    // a, b = a k.n in Q62
    const fx a = m.a = c.a0 + (mulu(c.a1, u).get() >> 7);
    const Bx ab = bal(a);
    fx* b = m.b;
    b[0] = mul(ab, bal(kn0)).get<4>();
    b[1] = mul(ab, bal(kn1)).get<4>();
    b[2] = -b[0] - b[1];
    // carrier phase, 2^-64 cycles: polynomial, Doppler f0 K, -fdot T u K + fdot K^2/2
    d = mul(c.Kc, g.ca);
    d.add(c.Ks, g.sa);
    const fx K = m.K = d.get();
    const Bx Kb = bal(K);
    uint64_t ph = c.C0 + c.D1 * (uint64_t)(unsigned)n;
    {
        const unsigned nn = (unsigned)(n * n);
        const uint64_t uu = (uint64_t)nn << (62 - 2 * lg);   // u^2 in Q62
        ph += (uint64_t)mul(c.c2, bal((fx)uu)).get<4>() + ((uint64_t)wide(c.c2i, (int)nn) << (64 - 2 * lg));
        d = mul(c.Fc, g.ca);
        d.add(c.Fs, g.sa);
        ph -= (uint64_t)d.get<9>();
        const fx t = (mulu(c.w1, u).get() >> 1) - mul(c.w2, Kb).get();   // Q60
        ph -= (uint64_t)mul(bal(t), Kb).get<8>();
    }
    m.ph = ph;
    // eps of the three receivers in Q56 (see the head of the file); k.rho_j in
    // units of (L/c)/3 s: the differences of the arms' k.n
    int ep0, ep1, ep2;
    {
        const int kr0 = (int)((kn2 - kn0) >> 31), kr1 = (int)((kn0 - kn1) >> 31), kr2 = (int)((kn1 - kn2) >> 31);   // Q29
        const int Kh = (int)(K >> 31);                                                                            // Q29
        const int s0 = Kh + (int)(wide(kr0, krho_q30) >> 30), s1 = Kh + (int)(wide(kr1, krho_q30) >> 30),
                  s2 = Kh + (int)(wide(kr2, krho_q30) >> 30);   // (2K + k.rho)/1024 s, Q29
        const int t0 = (int)(wide(kr0, s0) >> 29), t1 = (int)(wide(kr1, s1) >> 29), t2 = (int)(wide(kr2, s2) >> 29);
        ep0 = (int)(wide(t0, c.FD) >> 31);   // Q29 + Q58 - 31 = Q56
        ep1 = (int)(wide(t1, c.FD) >> 31);
        ep2 = (int)(wide(t2, c.FD) >> 31);
    }
    m.ep[0] = ep0;
    m.ep[1] = ep1;
    m.ep[2] = ep2;
    // arm phase factors; z = 3 theta + 3 (eps_i + eps_j)/2
    fx c0, s0, c1, s1, c2, s2;
    cis_third<TIER>(b[1] - b[2] + 96ll * (ep0 + ep1), c0, s0);   // Q56 -> Q62 and 3/2: x 96
    cis_third<TIER>(b[2] - b[0] + 96ll * (ep1 + ep2), c1, s1);
    {
        const Bx c0b = bal(c0), s0b = bal(s0), c1b = bal(c1), s1b = bal(s1);
        Dot dc = mul(c0b, c1b), ds = mul(s0b, c1b);
        dc.add(bal(-s0), s1b);
        ds.add(c0b, s1b);
        // conjugate of the product, turned by the sum of the three mean eps
        const int sg = ep0 + ep1 + ep2;   // Q56
        c2 = dc.get<2>();
        s2 = -ds.get<2>();
        const fx cr = wide((int)(s2 >> 32), sg) >> 24, sr = wide((int)(c2 >> 32), sg) >> 24;   // Q30 + Q56 -> Q62
        c2 -= cr;
        s2 += sr;
    }
    m.co[0] = c0;
    m.co[1] = c1;
    m.co[2] = c2;
    m.si[0] = s0;
    m.si[1] = s1;
    m.si[2] = s2;
    // amplitude polynomials C1 = a sin 2a cos a / (a0 sin 2a0), S1 = a sin 2a sin a / (a0 sin 2a0)
    {
        int r = c.cc4 + (int)(wide(c.cc5, u) >> 31);
        r = c.cc3 + (int)(wide(r, u) >> 31);
        fx q = c.cc2 + (wide(r, u) >> 22);
        q = c.cc1 + mulu(bal(q), u).get();   // Q64 -> Q63 -> Q62
        m.C1 = bal(c.cc0 + mulu(bal(q), u).get());
        r = c.cs4 + (int)(wide(c.cs5, u) >> 31);
        r = c.cs3 + (int)(wide(r, u) >> 31);
        q = c.cs2 + (wide(r, u) >> 22);
        q = c.cs1 + mulu(bal(q), u).get();
        m.S1 = bal(c.cs0 + mulu(bal(q), u).get());
    }
    // n.u, n.v in Q62
    fx *nu = m.nu, *nv = m.nv;
    d = mul(c.u0, g.n0x);
    d.add(c.u1, g.n0y);
    d.add(c.u2, g.n0z);
    nu[0] = d.get<2>();
    d = mul(c.u0, g.n1x);
    d.add(c.u1, g.n1y);
    d.add(c.u2, g.n1z);
    nu[1] = d.get<2>();
    nu[2] = -nu[0] - nu[1];
    d = mul(c.v0, g.n0x);
    d.add(c.v1, g.n0y);
    nv[0] = d.get<2>();
    d = mul(c.v0, g.n1x);
    d.add(c.v1, g.n1y);
    nv[1] = d.get<2>();
    nv[2] = -nv[0] - nv[1];
}

// polarisation response of arm k: G = n.H.n at unit amplitude, Q60, and
// F+ = (n.u)^2 - (n.v)^2, Fx/2 = (n.u)(n.v), Q60
struct PolFx {
    Bx Fp, Fx;
    fx Gr, Gi;
};
GB_FX PolFx pol_fx(const CandFx& c, const MidFx& m, int k) {
    PolFx p;
    p.Fp = bal(mul(bal(m.nu[k] - m.nv[k]), bal(m.nu[k] + m.nv[k])).get());
    p.Fx = bal(mul(bal(m.nu[k]), bal(m.nv[k])).get());
    Dot gr = mul(c.gpr, p.Fp), gi = mul(c.gpi, p.Fp);
    gr.add(c.gxr, p.Fx);
    gi.add(c.gxi, p.Fx);
    p.Gr = gr.get<4>();
    p.Gi = gi.get<4>();
    return p;
}

// Slow part of sample n of N = 2^lg: A, E (and T with T3) as integers, whose
// transforms times c.sA, c.sE, c.sT are the channels' bin values.
template <int TIER, bool T3>
GB_FX void sample_fx(const CandFx& c, const GeoFx& g, const FxTw* tw, int krho_q30, int n, int lg, int sh, fx (&o)[6]) {
    MidFx m;
    middle_fx<TIER>(c, g, krho_q30, n, lg, m);
    const Bx C1 = m.C1, S1 = m.S1;
    const fx a = m.a;
    const fx* b = m.b;
    Dot Ar{0, 0}, Ai{0, 0}, Er{0, 0}, Ei{0, 0}, Tr{0, 0}, Ti{0, 0};
#pragma unroll
    for (int k = 0; k < 3; ++k) {
        // polarisation response times the arm's phase factor: H in Q58
        const PolFx G = pol_fx(c, m, k);
        const Bx Gr = bal(G.Gr), Gi = bal(G.Gi);
        const Bx ck = bal(m.co[k]), sk = bal(m.si[k]);
        Dot hr = mul(Gr, ck), hi = mul(Gr, sk);
        hr.add(bal(-G.Gi), sk);
        hi.add(Gi, ck);
        const fx Hi_ = hi.get();   // Q58
        const Bx Hr = bal(hr.get()), Hi = bal(Hi_), mHi = bal(-Hi_);
        // links: Sh, Dh in Q62, p and q in Q60
        const Bx xm = bal(a - b[k]), xp = bal(a + b[k]);
        const fx sm = half_sinc<TIER>(square<TIER>(xm));
        const fx sp = half_sinc<TIER>(square<TIER>(xp));
        const Bx Sh = bal(sp + sm), Dh = bal(sp - sm);
        const fx p = mul(Sh, C1).get(), q = mul(Dh, S1).get();
        // dp = Sh S1 Delta/2, dq = Dh C1 Delta/2 in Q58, Delta = eps of the + receiver - eps of the - one
        const int dl = m.ep[k == 2 ? 0 : k + 1] - m.ep[k];   // Q56
        const int ss = (int)(wide(Sh.h, S1.h) >> 30), dc = (int)(wide(Dh.h, C1.h) >> 30);   // Q30
        const fx dp = (wide(ss, dl) >> 29) * 4, dq = (wide(dc, dl) >> 29) * 4;   // Q57 of value/2 = Q58; x 4: Q60
        // A sqrt2 = Z - X, E sqrt6 = X - 2Y + Z, T sqrt3 = X + Y + Z: coefficients of H_k
        fx ar, ai, er, ei;
        if (k == 0) {
            ar = -(p + dp);
            ai = -(q - dq);
            er = 3 * p - dp;
            ei = -(q + 3 * dq);
        } else if (k == 1) {
            ar = -(p - dp);
            ai = q + dq;
            er = -(3 * p + dp);
            ei = -(q - 3 * dq);
        } else {
            ar = 2 * p;
            ai = -2 * dq;
            er = 2 * dp;
            ei = 2 * q;
        }
        const Bx arb = bal(ar), aib = bal(ai), erb = bal(er), eib = bal(ei);
        Ar.add(Hr, arb);
        Ar.add(mHi, aib);
        Ai.add(Hi, arb);
        Ai.add(Hr, aib);
        Er.add(Hr, erb);
        Er.add(mHi, eib);
        Ei.add(Hi, erb);
        Ei.add(Hr, eib);
        if (T3) {
            const Bx trb = bal(2 * dp), tib = bal(2 * q);
            Tr.add(Hr, trb);
            Tr.add(mHi, tib);
            Ti.add(Hi, trb);
            Ti.add(Hr, tib);
        }
    }
    fx co, si;
    cis_table(m.ph, tw, co, si);
    const Bx cb = bal(co), sb = bal(si), msb = bal(-si);
    {
        const Bx r = bal(Ar.get()), i = bal(Ai.get());   // Q54
        Dot x = mul(r, cb), y = mul(r, sb);
        x.add(i, msb);
        y.add(i, cb);
        o[0] = x.get() >> sh;   // Q52
        o[1] = y.get() >> sh;
    }
    {
        const Bx r = bal(Er.get()), i = bal(Ei.get());
        Dot x = mul(r, cb), y = mul(r, sb);
        x.add(i, msb);
        y.add(i, cb);
        o[2] = x.get() >> sh;
        o[3] = y.get() >> sh;
    }
    if (T3) {
        const Bx r = bal(Tr.get(c.tsh)), i = bal(Ti.get(c.tsh));
        Dot x = mul(r, cb), y = mul(r, sb);
        x.add(i, msb);
        y.add(i, cb);
        o[4] = x.get() >> sh;
        o[5] = y.get() >> sh;
    }
}

// double -> fixed point with q fractional bits (|x| 2^q < 2^63)
GB_FX fx to_fx(double x, double scale) {
#ifdef __CUDA_ARCH__
    return __double2ll_rn(x * scale);
#else
    return (fx)llrint(x * scale);
#endif
}
GB_FX Bx to_bx(double x, double scale) { return bal(to_fx(x, scale)); }

// Samples are shifted right by this many bits so that the transform's sums
// stay inside 64 bits: with |n.H.n| <= 2 and |p| <= 1, |q| <= 0.1 the
// channels' moduli are below 12.8 in Q52, 2^55.7, and N 2^(55.7 - shift) < 2^63
GB_FX int fx_shift(int lg) { return lg > 7 ? lg - 7 : 0; }

struct FxTrig {
    double sb, cb, sl, cl, s2, c2, ci, sa, ca;   // of beta, lambda, 2 psi, iota, a0 = pi f0 L/c
};

// Taylor coefficients in v, a = a0 (1 + v), of
//   C1 = a sin 2a cos a/(a0 sin 2a0) = (1 + v) (sin 3a + sin a)/(2 sin 2a0),
//   S1 = a sin 2a sin a/(a0 sin 2a0) = (1 + v) (cos a - cos 3a)/(2 sin 2a0),
// from sin a0 and cos a0
GB_FX void amplitude_series(double a0, double s1, double c1, double (&Cv)[6], double (&Sv)[6]) {
    const double s3 = s1 * (3.0 - 4.0 * s1 * s1), c3 = c1 * (4.0 * c1 * c1 - 3.0);
    const double inv = 0.25 / (s1 * c1);
    double C[6], S[6];
    double ak = 1.0, p3 = 1.0;   // a0^k/k!, 3^k
    for (int k = 0; k < 6; ++k) {
        const int m = k & 3;
        const double ds3 = m == 0 ? s3 : m == 1 ? c3 : m == 2 ? -s3 : -c3, ds1 = m == 0 ? s1 : m == 1 ? c1 : m == 2 ? -s1 : -c1;
        const double dc3 = m == 0 ? c3 : m == 1 ? -s3 : m == 2 ? -c3 : s3, dc1 = m == 0 ? c1 : m == 1 ? -s1 : m == 2 ? -c1 : s1;
        C[k] = (p3 * ds3 + ds1) * ak * inv;
        S[k] = (dc1 - p3 * dc3) * ak * inv;
        ak *= a0 / (double)(k + 1);
        p3 *= 3.0;
    }
    C[0] = c1;
    S[0] = s1;
    for (int k = 0; k < 6; ++k) {
        Cv[k] = C[k] + (k > 0 ? C[k - 1] : 0.0);
        Sv[k] = S[k] + (k > 0 ? S[k - 1] : 0.0);
    }
}

// Candidate constants; c.tier = -1 when a parameter is outside the ranges.
// arm_c = L/c; the caller supplies the sines and cosines.
GB_FX void setup_fx(const double* th, double T, double arm_c, double delta, int lg, const FxTrig& t, CandFx& c) {
    const double f0 = th[0], fd = th[1], A = th[4], phi0 = th[7];
    const double pi = 3.14159265358979323846;
    const double N = (double)(1 << lg);
    const double a0 = pi * f0 * arm_c, a1 = pi * fd * T * arm_c, eta = fd * T / f0;
    const double xmax = 2.0 * fmax(fabs(a0), fabs(a0 + a1));
    const double r = 1.495978707e11 / 299792458.0;
    // f0 K reaches several cycles: its two products as double-word values
    const double rc = -r * t.cb, rc_e = fma(-r, t.cb, -rc);
    const double Kc = rc * t.cl, Ks = rc * t.sl;
    const double Fc = f0 * Kc, Fs = f0 * Ks;
    const double Fc_e = fma(f0, Kc, -Fc) + f0 * (fma(rc, t.cl, -Kc) + rc_e * t.cl);
    const double Fs_e = fma(f0, Ks, -Fs) + f0 * (fma(rc, t.sl, -Ks) + rc_e * t.sl);
    // fdot T^2/2 as a double-word value: it reaches hundreds of cycles
    const double fdT = fd * T, fdT_e = fma(fd, T, -fdT), c2h = 0.5 * (fdT * T),
                 c2l = 0.5 * (fma(fdT, T, -(fdT * T)) + fdT_e * T), c2r = rint(c2h);
    const double FD = pi * fd * (arm_c / 3.0) * 1024.0, w1 = 512.0 * fd * T, w2 = 131072.0 * fd;
    // The eps terms are 32-bit: with k.rho of up to sqrt3 (L/3c), |K| <= 500 s
    // and arm_c < 300 s, |k.rho (2K + k.rho)| stays below 1.99 units, so |eps|
    // below 1.99 2^29 (Q56) for FD 2^58 < 2^31 (rounded: hence not up to
    // 2^-27), and the difference of two below 3.3 2^29.
    const bool ok = f0 > 0.0 && xmax <= 1.3 && fabs(eta) <= 0x1p-10 && fabs(Fc) < 31.0 && fabs(Fs) < 31.0 &&
                    fabs(c2h) < 0x1p30 && fabs(FD) < 0x1.fffffp-28 && fabs(w1) < 0.9 && fabs(w2) < 0.2 && arm_c < 300.0 &&
                    fabs(delta) < 0x1p40 && fabs(phi0) < 0x1p30;
    c.tier = !ok ? -1 : xmax <= 0.5 ? 0 : 1;
    if (!ok) return;
    c.k0 = to_bx(-(t.cb * t.cl), 0x1p62);
    c.k1 = to_bx(-(t.cb * t.sl), 0x1p62);
    c.k2 = to_bx(-t.sb, 0x1p62);
    c.u0 = to_bx(t.sb * t.cl, 0x1p62);
    c.u1 = to_bx(t.sb * t.sl, 0x1p62);
    c.u2 = to_bx(-t.cb, 0x1p62);
    c.v0 = to_bx(t.sl, 0x1p62);
    c.v1 = to_bx(-t.cl, 0x1p62);
    const double Ap = 1.0 + t.ci * t.ci, Ax = -2.0 * t.ci;
    c.gpr = to_bx(Ap * t.c2, 0x1p60);
    c.gxr = to_bx(-2.0 * (Ap * t.s2), 0x1p60);
    c.gpi = to_bx(-(Ax * t.s2), 0x1p60);
    c.gxi = to_bx(-2.0 * (Ax * t.c2), 0x1p60);
    c.Kc = to_bx(Kc, 0x1p53);
    c.Ks = to_bx(Ks, 0x1p53);
    c.Fc = bal(to_fx(Fc, 0x1p57) + to_fx(Fc_e, 0x1p57));
    c.Fs = bal(to_fx(Fs, 0x1p57) + to_fx(Fs_e, 0x1p57));
    c.w1 = to_bx(w1, 0x1p62);
    c.w2 = to_bx(w2, 0x1p64);
    c.c2 = to_bx((c2h - c2r) + c2l, 0x1p62);
    c.c2i = (int)c2r;
    c.a0 = to_fx(a0, 0x1p62);
    c.a1 = to_bx(a1, 0x1p70);
    c.FD = (int)to_fx(FD, 0x1p58);
    double p0 = phi0 * 0.15915494309189535;
    p0 -= rint(p0);
    double d4 = -a0 * 0.63661977236758134;   // -4 a0 / (2 pi)
    d4 -= rint(d4);
    c.C0 = (uint64_t)to_fx(p0, 0x1p62) * 4u + (uint64_t)to_fx(d4, 0x1p62) * 4u;
    const double dr = delta - N * rint(delta / N);
    const double sc = ldexp(1.0, 62 - lg);
    c.D1 = (uint64_t)to_fx(dr, sc) * 4u + (uint64_t)to_fx(-a1 * 0.63661977236758134, 4.0 * sc);
    double Cv[6], Sv[6];
    amplitude_series(a0, t.sa, t.ca, Cv, Sv);
    double e = 1.0, Cu[6], Su[6];
    for (int k = 0; k < 6; ++k) {
        Cu[k] = Cv[k] * e;
        Su[k] = Sv[k] * e;
        e *= eta;
    }
    c.cc0 = to_fx(Cu[0], 0x1p62);
    c.cc1 = to_fx(Cu[1], 0x1p63);
    c.cc2 = to_fx(Cu[2], 0x1p64);
    c.cc3 = (int)to_fx(Cu[3], 0x1p55);
    c.cc4 = (int)to_fx(Cu[4], 0x1p55);
    c.cc5 = (int)to_fx(Cu[5], 0x1p55);
    c.cs0 = to_fx(Su[0], 0x1p62);
    c.cs1 = to_fx(Su[1], 0x1p63);
    c.cs2 = to_fx(Su[2], 0x1p64);
    c.cs3 = (int)to_fx(Su[3], 0x1p55);
    c.cs4 = (int)to_fx(Su[4], 0x1p55);
    c.cs5 = (int)to_fx(Su[5], 0x1p55);
    // |T| < 6 a^3 + 4 a 2^-20 (q < a^3/3, dp < a 2^-26): shifted up to A's range
    c.tsh = 0;
    for (double b = 6.0 * a0 * a0 * a0 * 1.01 + 0x1p-18 * a0; b < 3.0 && c.tsh < 24; b *= 2.0) ++c.tsh;
    const double amp = A * (8.0 * a0 * t.sa * t.ca) * (T / (2.0 * N)) * ldexp(1.0, fx_shift(lg) - 52);   // 4 a0 sin 2a0
    c.sA = amp * 0.70710678118654752;
    c.sE = amp * 0.40824829046386302;
    c.sT = amp * 0.57735026918962576 * ldexp(1.0, -c.tsh);
}

// Index of element e in a transform buffer: the low three bits XORed with the
// higher groups of three, so that eight lanes whose indices differ in any
// three neighbouring bits (every stage of the transform, the bit-reversed
// stores and the reads in order) meet eight different 16-byte bank groups.
GB_FX int sw(int e) { return e ^ ((e >> 3) & 7) ^ ((e >> 6) & 7) ^ ((e >> 9) & 1); }

// synchronisation of the NT threads that share a transform (one thread: none)
template <int NT>
GB_FX void sync_nt() {
#ifdef __CUDA_ARCH__
    if (NT == 32) __syncwarp();
    else __syncthreads();
#endif
}

GB_FX fx double_bits(double v) {
#ifdef __CUDA_ARCH__
    return __double_as_longlong(v);
#else
    fx b;
    memcpy(&b, &v, sizeof b);
    return b;
#endif
}

// a fixed-point complex value, or, after the last stage, the bits of two doubles
struct alignas(16) Z64 {
    fx x, y;
};
GB_FX Z64 zadd(Z64 a, Z64 b) { return {a.x + b.x, a.y + b.y}; }
GB_FX Z64 zsub(Z64 a, Z64 b) { return {a.x - b.x, a.y - b.y}; }
GB_FX Z64 zmi(Z64 a) { return {a.y, -a.x}; }   // times -i
GB_FX Z64 zmul(Z64 a, const FxTw& w) {   // times co - i si
    const Bx r = bal(a.x), i = bal(a.y), mr = bal(-a.x);
    Dot re = mul(r, w.co), im = mul(mr, w.si);
    re.add(i, w.si);
    im.add(i, w.co);
    return {re.get<2>(), im.get<2>()};
}
GB_FX Z64 zout(Z64 a, double s, bool last) {
    if (!last) return a;
    return {double_bits((double)a.x * s), double_bits((double)a.y * s)};
}

// In-place FFT of nch buffers (stride elements apart): bit-reversed input,
// natural order output, as doubles times sc[ch] or (RAW) as it is.  Radix-2 decimation in time,
// two stages at a time (three twiddle products per four elements; the first
// two stages have none), the odd stage last.  Bound by the integer products
// of the twiddles.
template <int NT, bool RAW = false>
GB_FXN void fft_fx(Z64* buf, int stride, int nch, int lg, const FxTw* tw, const double* sc, int lane) {
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
        const bool last = !RAW && s + 2 == lg;
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
                p[i0] = zout(zadd(a, b), sc[ch], !RAW);
                p[i1] = zout(zsub(a, b), sc[ch], !RAW);
            }
        }
        sync_nt<NT>();
    }
}

}  // namespace gb
