// fx64_grad.cuh -- reverse mode of fx64.cuh's sample, in the same arithmetic.
//
// With w_ch = conj(c_ch) exp(i Phi) (c_ch a channel's cotangent, Phi the
// carrier phase) and H_k = G_k exp(i theta_k), a sample's share of the
// gradient is Re sum_k G_k nu_k differentiated, where
//   nu_k = (p_k - i dq_k) P_k + (dp_k + i q_k) R_k,
//   P = (3 wE - wA, -3 wE - wA, 2 wA),  R = 2 wT + (-wA - wE, wA - wE, 2 wE),
// each turned by exp(i theta_k) (wE carries 1/sqrt3 and wT sqrt(2/3), so that
// all channels have A's normalisation).  So
//   tau_k = -Im(G_k nu_k)        dL/d theta_k, and Y = sum tau_k = dL/d Phi;
//   Re(G_k P_k), -Im(G_k R_k)    dL/dp_k, dL/dq_k;
//   sums of nu_k F+, nu_k Fx/2, nu_k (k.n)(n.u), nu_k (k.n)(n.v)
// give everything that comes through G (A, iota, psi, and beta and lambda's
// rotation of the polarisation basis), since F+ and Fx/2 change by
//   beta: -2 (k.n)(n.u), -(k.n)(n.v);
//   lambda: -4 sin b Fx/2 + 2 cos b (k.n)(n.v), sin b F+ - cos b (k.n)(n.u),
// and moments of Y with u, K, cos and sin of the orbital phase give all that
// comes through Phi.  p and q depend on a and b = a k.n through sinc and its
// derivative; d(k.n) = n.u d beta + cos b n.v d lambda.  The eps terms (1e-8
// rad at most) are differentiated in float.
//
// Cotangents are normalised per candidate, |Re|, |Im| <= 1 in Q60.
#pragma once
#include "fx64.cuh"

namespace gb {

// d sinc(X)/dy, y = X^2 -> Q62 (so d(sinc(X)/2)/dX = X times this)
template <int TIER>
GB_FX fx sinc_dy(Bx y) {
    if (TIER == 0) {
        fx r = 50834280834975ll + (wide(step32<0>(4321363, y.h, -564118257), y.h) >> 22);
        r = step64<0>(r, y, -2745051201405427ll);
        r = step64<0>(r, y, 76861433640455620ll);
        return step64<0>(r, y, -768614336404564648ll);
    }
    int s = step32<2>(25361, y.h, -6170044);
    s = step32<2>(s, y.h, 1110886789);
    fx r = -577662282807ll + (wide(s, y.h) >> 28);
    r = step64<2>(r, y, 50834281505203ll);
    r = step64<2>(r, y, -2745051201444233ll);
    r = step64<2>(r, y, 76861433640456413ll);
    return step64<2>(r, y, -768614336404564650ll);
}

// Scale 2^k that takes a residual to integers for its transform.  The sum of
// |re| + |im| over the bins (of the channel where it is largest) bounds the
// transform and everything on the way to it, and is brought below 2^62; the
// largest component times N would leave log2 N bits unused where one bin
// dominates.  The sum is taken from the components' high words, in units of
// 2^-19 of the largest component's power of two, each rounded up (FP64 sums:
// 2% of the gradient's time).  hi, top: high words of |component| and of the
// largest one; at most 2 x 1024 shares of 2^20 + 1 are added.
GB_FX unsigned residual_share(unsigned hi, unsigned top) {
    const unsigned d = (top >> 20) - (hi >> 20);
    return (((hi & 0xFFFFFu) | 0x100000u) >> (d < 30u ? d + 1u : 31u)) + 1u;
}
GB_FX int residual_shift(unsigned sum, unsigned top) {
    int b = 0;   // sum < 2^b
#ifdef __CUDA_ARCH__
    b = 32 - __clz((int)sum);
#else
    while (b < 32 && sum >> b) ++b;
#endif
    const int k = 62 - (b - 19 + (int)(top >> 20) - 1023);
    return k < 1000 ? k : 1000;
}

struct CandGFx {
    Bx a0, a3;                   // Q62, a0 and a0/3
    Bx eta;                      // Q70, fdot T/f0
    Bx w3;                       // Q64, 512 fdot/f0
    fx ec0, es0;                 // dC1/dv, dS1/dv (v = eta u): Q60
    fx ec1, es1;                 // Q61
    fx ec2, es2;                 // Q62
    int ec3, ec4, es3, es4;      // Q53
    float pfd, l3, rcb[2], rcl[2];   // pi fdot, L/3c, dK/dbeta and dK/dlambda/cos(beta) per cos a, sin a
};

enum {
    kGS1, kGS2, kGSk, kGSuk, kGSkk, kGSc, kGSs, kGQ0, kGQ0u, kGB, kGL, kGUPr, kGUPi, kGUQr, kGUQi, kGV1r, kGV1i,
    kGV2r, kGV2i, kGEf, kGEb, kGEl, kGSums
};

GB_FX float hi_f(fx x, float s) { return (float)(int)(x >> 32) * s; }

// One sample: gr, gi are the normalised conj(c) of A, E, T (Q60); adds to acc.
template <int TIER, bool T3>
GB_FX void adjoint_fx(const CandFx& c, const CandGFx& cg, const GeoFx& g, const FxTw* tw, int krho_q30, int n, int lg,
                      const fx (&gr)[3], const fx (&gi)[3], double (&acc)[kGSums]) {
    MidFx m;
    middle_fx<TIER>(c, g, krho_q30, n, lg, m);
    const int u = m.u;
    const Bx ab = bal(m.a);
    // cotangents on the carrier: Q60
    fx wr[3], wi[3];
    {
        fx co, si;
        cis_table(m.ph, tw, co, si);
        const Bx cb = bal(co), sb = bal(si), msb = bal(-si);
#pragma unroll
        for (int ch = 0; ch < (T3 ? 3 : 2); ++ch) {
            const Bx r = bal(gr[ch]), i = bal(gi[ch]);
            Dot x = mul(r, cb), y = mul(r, sb);
            x.add(i, msb);
            y.add(i, cb);
            wr[ch] = x.get<2>();
            wi[ch] = y.get<2>();
        }
    }
    // dC1/dv, dS1/dv in Q60
    Bx E1, F1;
    {
        int r = cg.ec3 + (int)(wide(cg.ec4, u) >> 31);
        fx q = cg.ec2 + (wide(r, u) >> 22);   // Q53 + 31 - 22 = Q62
        q = cg.ec1 + mulu(bal(q), u).get();
        E1 = bal(cg.ec0 + mulu(bal(q), u).get());
        r = cg.es3 + (int)(wide(cg.es4, u) >> 31);
        q = cg.es2 + (wide(r, u) >> 22);
        q = cg.es1 + mulu(bal(q), u).get();
        F1 = bal(cg.es0 + mulu(bal(q), u).get());
    }
    Dot UPr{0, 0}, UPi{0, 0}, UQr{0, 0}, UQi{0, 0}, V1r{0, 0}, V1i{0, 0}, V2r{0, 0}, V2i{0, 0}, Q0{0, 0};
    fx tau[3];                  // Q56
    Dot kk[3];                  // Q54: dL/d(k.n) / a but for theta's part
    float pk[3], xk[3];         // dL/d Delta_k, and dp, dq's share of dL/d(k.n)
#pragma unroll
    for (int k = 0; k < 3; ++k) {
        const PolFx G = pol_fx(c, m, k);
        const Bx Gr = bal(G.Gr), Gi = bal(G.Gi), mGi = bal(-G.Gi);   // Q60
        const Bx ck = bal(m.co[k]), sk = bal(m.si[k]), msk = bal(-m.si[k]);
        // P, R before the turn, then turned: Q60
        fx Pr, Pi, Rr, Ri;
        if (k == 0) {
            Pr = 3 * wr[1] - wr[0];
            Pi = 3 * wi[1] - wi[0];
            Rr = -wr[0] - wr[1];
            Ri = -wi[0] - wi[1];
        } else if (k == 1) {
            Pr = -3 * wr[1] - wr[0];
            Pi = -3 * wi[1] - wi[0];
            Rr = wr[0] - wr[1];
            Ri = wi[0] - wi[1];
        } else {
            Pr = 2 * wr[0];
            Pi = 2 * wi[0];
            Rr = 2 * wr[1];
            Ri = 2 * wi[1];
        }
        if (T3) {
            Rr += 2 * wr[2];
            Ri += 2 * wi[2];
        }
        Bx Prb, Pib, Rrb, Rib, mPi, mPr, mRi;
        {
            const Bx a = bal(Pr), b = bal(Pi), e = bal(Rr), f = bal(Ri);
            Dot x = mul(a, ck), y = mul(a, sk);
            x.add(b, msk);
            y.add(b, ck);
            const fx pr = x.get<2>(), pi = y.get<2>();
            Prb = bal(pr);
            Pib = bal(pi);
            mPr = bal(-pr);
            mPi = bal(-pi);
            x = mul(e, ck);
            y = mul(e, sk);
            x.add(f, msk);
            y.add(f, ck);
            const fx ri = y.get<2>();
            Rrb = bal(x.get<2>());
            Rib = bal(ri);
            mRi = bal(-ri);
        }
        // links and their derivatives: Sh, Dh, Sg = d Sh/da at fixed b, Dd = d Sh/db, Q62
        const Bx xm = bal(m.a - m.b[k]), xp = bal(m.a + m.b[k]);
        const Bx ym = square<TIER>(xm), yp = square<TIER>(xp);
        const fx sm = half_sinc<TIER>(ym), sp = half_sinc<TIER>(yp);
        const fx dm = mul(bal(sinc_dy<TIER>(ym)), xm).template get<2>(), dpl = mul(bal(sinc_dy<TIER>(yp)), xp).template get<2>();
        const Bx Sh = bal(sp + sm), Dh = bal(sp - sm);
        const fx Sg_ = dpl + dm, Dd_ = dpl - dm;
        const Bx Sg = bal(Sg_), Dd = bal(Dd_), kn = bal(m.kn[k]);
        const fx p = mul(Sh, m.C1).get(), q = mul(Dh, m.S1).get();   // Q60
        const int dl = m.ep[k == 2 ? 0 : k + 1] - m.ep[k];           // Q56
        const int ss = (int)(wide(Sh.h, m.S1.h) >> 30), dc = (int)(wide(Dh.h, m.C1.h) >> 30);
        const fx dp = (wide(ss, dl) >> 29) * 4, dq = (wide(dc, dl) >> 29) * 4;   // Q60
        // nu = (p - i dq) P + (dp + i q) R: Q60
        const Bx pb = bal(p), qb = bal(q), dpb = bal(dp), dqb = bal(dq);
        Dot x = mul(pb, Prb), y = mul(pb, Pib);
        x.add(dqb, Pib);
        y.add(dqb, mPr);
        x.add(dpb, Rrb);
        y.add(dpb, Rib);
        x.add(qb, mRi);
        y.add(qb, Rrb);
        const Bx nr = bal(x.get<4>()), ni = bal(y.get<4>());
        x = mul(Gr, ni);
        x.add(Gi, nr);
        tau[k] = -x.get();   // Q56
        // dL/dp, dL/dq in Q58
        x = mul(Gr, Prb);
        x.add(Gi, mPi);
        const Bx rp = bal(x.get<2>());
        y = mul(mGi, Rrb);
        y.add(Gr, mRi);
        const Bx rq = bal(y.get<2>());
        // sums through G: Q56
        UPr.add(nr, G.Fp);
        UPi.add(ni, G.Fp);
        UQr.add(nr, G.Fx);
        UQi.add(ni, G.Fx);
        const Bx knu = bal(mul(kn, bal(m.nu[k])).get<2>()), knv = bal(mul(kn, bal(m.nv[k])).get<2>());   // Q60
        V1r.add(nr, knu);
        V1i.add(ni, knu);
        V2r.add(nr, knv);
        V2i.add(ni, knv);
        // a0 d/da: p' = a0 (Sg + Dd kn) C1 + Sh E1, q' = a0 (Dd + Sg kn) S1 + Dh F1, Q60
        const Bx da = bal(Sg_ + mul(Dd, kn).get<4>()), db = bal(Dd_ + mul(Sg, kn).get<4>());   // Q62
        x = mul(bal(mul(da, m.C1).get<2>()), cg.a0);   // Q62 x Q62 -> Q60
        y = mul(Sh, E1);                                // Q62 x Q60 -> Q58
        Q0.add(rp, bal(x.get() + y.get<2>()));
        x = mul(bal(mul(db, m.S1).get<2>()), cg.a0);
        y = mul(Dh, F1);
        Q0.add(rq, bal(x.get() + y.get<2>()));
        // d/d(k.n) / a
        kk[k] = mul(rp, bal(mul(Dd, m.C1).get()));     // Q58 x Q60 -> Q54
        kk[k].add(rq, bal(mul(Sg, m.S1).get()));
        // the eps terms, float
        const float S = hi_f(sp + sm, 0x1p-30f), D = hi_f(sp - sm, 0x1p-30f), c1 = (float)m.C1.h * 0x1p-30f,
                    s1 = (float)m.S1.h * 0x1p-30f;
        const float gR = ((float)Gr.h * (float)Rrb.h - (float)Gi.h * (float)Rib.h) * 0x1p-56f;
        const float gP = ((float)Gr.h * (float)Pib.h + (float)Gi.h * (float)Prb.h) * 0x1p-56f;
        pk[k] = 0.5f * (gR * S * s1 + gP * D * c1);
        xk[k] = 0.5f * ((float)dl * 0x1p-56f) * hi_f(m.a, 0x1p-30f) *
                (gR * hi_f(Dd_, 0x1p-30f) * s1 + gP * hi_f(Sg_, 0x1p-30f) * c1);
    }
    // theta_k = (b_p - b_q)/3: its share of a0 d/da and of d/d(k.n)
    const fx t0 = tau[0] * 4, t1 = tau[1] * 4, t2 = tau[2] * 4;   // Q58
    Q0.add(bal(t0), bal(mul(cg.a3, bal(m.kn[1] - m.kn[2])).get<2>()));   // Q62 x Q60 -> Q60
    Q0.add(bal(t1), bal(mul(cg.a3, bal(m.kn[2] - m.kn[0])).get<2>()));
    Q0.add(bal(t2), bal(mul(cg.a3, bal(m.kn[0] - m.kn[1])).get<2>()));
    const Bx third = bal(384307168202282325ll);   // 1/3 in Q60
    kk[0].add(bal(t2 - t1), third);
    kk[1].add(bal(t0 - t2), third);
    kk[2].add(bal(t1 - t0), third);
    Dot B{0, 0}, Lm{0, 0};
#pragma unroll
    for (int k = 0; k < 3; ++k) {
        const Bx v = bal(kk[k].get<4>());   // Q58
        B.add(v, bal(m.nu[k]));
        Lm.add(v, bal(m.nv[k]));
    }
    const double q54 = 0x1p-54, q56 = 0x1p-56;
    acc[kGB] += (double)mul(bal(B.get()), ab).get() * q54;   // Q56 x Q62
    acc[kGL] += (double)mul(bal(Lm.get()), ab).get() * q54;
    const fx q0 = Q0.get();   // Q54
    acc[kGQ0] += (double)q0 * q54;
    acc[kGQ0u] += (double)mulu(bal(q0), u).get<1>() * q54;
    acc[kGUPr] += (double)UPr.get() * q56;
    acc[kGUPi] += (double)UPi.get() * q56;
    acc[kGUQr] += (double)UQr.get() * q56;
    acc[kGUQi] += (double)UQi.get() * q56;
    acc[kGV1r] += (double)V1r.get() * q56;
    acc[kGV1i] += (double)V1i.get() * q56;
    acc[kGV2r] += (double)V2r.get() * q56;
    acc[kGV2i] += (double)V2i.get() * q56;
    // moments of Y
    const fx Y = tau[0] + tau[1] + tau[2];
    const Bx Yb = bal(Y), Kb = bal(m.K);
    const fx Yu = mulu(Yb, u).get<1>();
    const Bx Yub = bal(Yu);
    const fx Yk = mul(Yb, Kb).get<4>();
    acc[kGS1] += (double)Yu * q56;
    acc[kGS2] += (double)mulu(Yub, u).get<1>() * q56;
    acc[kGSk] += (double)Yk * q56;
    acc[kGSuk] += (double)mul(Yub, Kb).get<4>() * q56;
    acc[kGSkk] += (double)mul(bal(Yk), Kb).get<4>() * q56;
    // (f - fdot K)/f0 = 1 + eta u - w3 K in Q60
    const fx psi = (1ll << 60) + (mulu(cg.eta, u).get() >> 9) - mul(cg.w3, Kb).get();
    const Bx Yp = bal(mul(Yb, bal(psi)).get<4>());
    acc[kGSc] += (double)mul(Yp, g.ca).get() * q54;
    acc[kGSs] += (double)mul(Yp, g.sa).get() * q54;
    // eps_j = pi fdot k.rho_j (2K + k.rho_j): dL/d eps_j from the arms' means and differences
    {
        const float f0 = hi_f(tau[0], 0x1p-24f), f1 = hi_f(tau[1], 0x1p-24f), f2 = hi_f(tau[2], 0x1p-24f);
        const float e[3] = {0.5f * (f0 + f2) - pk[0] + pk[2], 0.5f * (f0 + f1) + pk[0] - pk[1],
                            0.5f * (f1 + f2) + pk[1] - pk[2]};
        const float K = hi_f(m.K, 512.0f * 0x1p-28f), ca = (float)g.ca.h * 0x1p-30f, sa = (float)g.sa.h * 0x1p-30f;
        const float Kbt = cg.rcb[0] * ca + cg.rcb[1] * sa, Kl = cg.rcl[0] * ca + cg.rcl[1] * sa;
        float sf = 0.0f, sb = 0.0f, sl = 0.0f;
#pragma unroll
        for (int j = 0; j < 3; ++j) {
            const int p = j == 0 ? 2 : j - 1;   // k.rho_j = (L/3c) (kn_p - kn_j)
            const float kr = cg.l3 * hi_f(m.kn[p] - m.kn[j], 0x1p-28f);
            const float ku = cg.l3 * (hi_f(m.nu[p], 0x1p-30f) - hi_f(m.nu[j], 0x1p-30f));
            const float kv = cg.l3 * (hi_f(m.nv[p], 0x1p-30f) - hi_f(m.nv[j], 0x1p-30f));
            sf += e[j] * kr * (2.0f * K + kr);
            sb += 2.0f * e[j] * (ku * (K + kr) + kr * Kbt);
            sl += 2.0f * e[j] * (kv * (K + kr) + kr * Kl);
        }
        float xb = 0.0f, xl = 0.0f;
#pragma unroll
        for (int k = 0; k < 3; ++k) {
            xb += xk[k] * hi_f(m.nu[k], 0x1p-30f);
            xl += xk[k] * hi_f(m.nv[k], 0x1p-30f);
        }
        acc[kGEf] += (double)(3.14159265f * sf);
        acc[kGEb] += (double)(cg.pfd * sb + xb);
        acc[kGEl] += (double)(cg.pfd * sl + xl);
    }
}

// Extra constants of a candidate; false when outside the ranges
GB_FX bool setup_gfx(const double* th, double T, double arm_c, const FxTrig& t, CandGFx& c) {
    const double pi = 3.14159265358979323846;
    const double f0 = th[0], fd = th[1], a0 = pi * f0 * arm_c, eta = fd * T / f0, w3 = 512.0 * fd / f0;
    if (!(fabs(w3) < 0.4)) return false;
    c.a0 = to_bx(a0, 0x1p62);
    c.a3 = to_bx(a0 / 3.0, 0x1p62);
    c.eta = to_bx(eta, 0x1p70);
    c.w3 = to_bx(w3, 0x1p60 * 16.0);
    double Cu[6], Su[6];   // Taylor coefficients in v of C1, S1
    amplitude_series(a0, t.sa, t.ca, Cu, Su);
    double e = 1.0, Ec[5], Es[5];
    for (int k = 0; k < 5; ++k) {
        Ec[k] = (double)(k + 1) * Cu[k + 1] * e;
        Es[k] = (double)(k + 1) * Su[k + 1] * e;
        e *= eta;
    }
    c.ec0 = to_fx(Ec[0], 0x1p60);
    c.ec1 = to_fx(Ec[1], 0x1p61);
    c.ec2 = to_fx(Ec[2], 0x1p62);
    c.ec3 = (int)to_fx(Ec[3], 0x1p53);
    c.ec4 = (int)to_fx(Ec[4], 0x1p53);
    c.es0 = to_fx(Es[0], 0x1p60);
    c.es1 = to_fx(Es[1], 0x1p61);
    c.es2 = to_fx(Es[2], 0x1p62);
    c.es3 = (int)to_fx(Es[3], 0x1p53);
    c.es4 = (int)to_fx(Es[4], 0x1p53);
    const float r = (float)(1.495978707e11 / 299792458.0);
    c.pfd = (float)(pi * fd);
    c.l3 = (float)(arm_c / 3.0);
    c.rcb[0] = r * (float)(t.sb * t.cl);
    c.rcb[1] = r * (float)(t.sb * t.sl);
    c.rcl[0] = r * (float)t.sl;
    c.rcl[1] = -r * (float)t.cl;
    return true;
}

// What the sums of a candidate are contracted with at the end
struct FinGFx {
    double f0, a0, sb, cb, sl, cl, gp[2], gx[2], gpi[2], gxi[2], gpp[2], gxp[2];   // gx: of Fx/2
    double F;      // scale of everything but A's row, less the normalisation of the cotangents
    double FA;     // scale of A's row
};
GB_FX void setup_fin(const double* th, double arm_c, int lg, const FxTrig& t, double si, FinGFx& c) {
    const double pi = 3.14159265358979323846;
    c.f0 = th[0];
    c.a0 = pi * th[0] * arm_c;
    c.sb = t.sb;
    c.cb = t.cb;
    c.sl = t.sl;
    c.cl = t.cl;
    const double Ap = 1.0 + t.ci * t.ci, Ax = -2.0 * t.ci, dAp = -2.0 * t.ci * si, dAx = 2.0 * si;
    c.gp[0] = Ap * t.c2;
    c.gp[1] = -(Ax * t.s2);
    c.gx[0] = -2.0 * (Ap * t.s2);
    c.gx[1] = -2.0 * (Ax * t.c2);
    c.gpi[0] = dAp * t.c2;
    c.gpi[1] = -(dAx * t.s2);
    c.gxi[0] = -2.0 * (dAp * t.s2);
    c.gxi[1] = -2.0 * (dAx * t.c2);
    c.gpp[0] = -2.0 * Ap * t.s2;
    c.gpp[1] = -2.0 * Ax * t.c2;
    c.gxp[0] = -4.0 * Ap * t.c2;
    c.gxp[1] = 4.0 * Ax * t.s2;
    c.FA = 2.0 / (double)(1 << lg) * (8.0 * c.a0 * t.sa * t.ca) * 0.70710678118654752;
    c.F = c.FA * th[4];
}
// gradient from the sums; norm: the cotangents' value per unit (2^-60 of an integer)
GB_FX void finish_gfx(const FinGFx& c, double T, const double* s, double norm, double* grad) {
    const double pi = 3.14159265358979323846, r = 1.495978707e11 / 299792458.0;
    auto re = [](const double* a, double x, double y) { return a[0] * x - a[1] * y; };
    const double upr = s[kGUPr], upi = s[kGUPi], uqr = s[kGUQr], uqi = s[kGUQi], v1r = s[kGV1r], v1i = s[kGV1i],
                 v2r = s[kGV2r], v2i = s[kGV2i];
    const double Y = -(c.gp[0] * upi + c.gp[1] * upr + c.gx[0] * uqi + c.gx[1] * uqr);
    const double F = c.F * norm;
    grad[0] = F * ((s[kGQ0] - 4.0 * c.a0 * Y) / c.f0 + 2.0 * pi * (T * s[kGS1] - 512.0 * s[kGSk]));
    grad[1] = F * (T * (s[kGQ0u] - 4.0 * c.a0 * s[kGS1]) / c.f0 +
                   pi * (T * T * s[kGS2] - 1024.0 * T * s[kGSuk] + 262144.0 * s[kGSkk]) + s[kGEf]);
    grad[2] = F * (s[kGB] - 2.0 * re(c.gp, v1r, v1i) - re(c.gx, v2r, v2i) -
                   2.0 * pi * c.f0 * r * c.sb * (c.cl * s[kGSc] + c.sl * s[kGSs]) + s[kGEb]);
    grad[3] = F * (c.cb * s[kGL] - 4.0 * c.sb * re(c.gp, uqr, uqi) + 2.0 * c.cb * re(c.gp, v2r, v2i) +
                   c.sb * re(c.gx, upr, upi) - c.cb * re(c.gx, v1r, v1i) -
                   2.0 * pi * c.f0 * r * c.cb * (c.sl * s[kGSc] - c.cl * s[kGSs]) + c.cb * s[kGEl]);
    grad[4] = c.FA * norm * (re(c.gp, upr, upi) + re(c.gx, uqr, uqi));
    grad[5] = F * (re(c.gpi, upr, upi) + re(c.gxi, uqr, uqi));
    grad[6] = F * (re(c.gpp, upr, upi) + re(c.gxp, uqr, uqi));
    grad[7] = F * Y;
}

}  // namespace gb
