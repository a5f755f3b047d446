// grad64.cu -- gradient of the window log-likelihood, double precision.
//
// With h_k = (T/2N) S_m and r_m = w_k (d_k - h_k) on window bins (0 elsewhere),
//   d logL / d theta_i = (4/T) sum_k w_k Re[(d_k - h_k) conj(d h_k/d theta_i)]
//                      = (2/N) Re sum_n  conj(c_n) d s_n / d theta_i,
//   c_n = conj(sum_m conj(r_m) exp(-2 pi i m n / N))   (the adjoint of the DFT).
// Per candidate one warp (1) computes the template, (2) forms the residual r
// and logL, (3) runs the adjoint FFT to get c_n, and (4) sweeps the samples in
// reverse mode.  The template, the adjoint FFT and the sweep run in 64-bit
// fixed point (fx64.cuh, fx64_grad.cuh): the residual is scaled by a power of
// two per candidate, the cotangents again before the sweep, and every sample
// leaves 22 sums in double that are contracted with the candidate's constants
// at the end, one candidate per lane.
//
// Measured on GB300, 64 windows x 512 candidates at N = 256: 33.8 ms with every
// step in double (FP64 pipe 84% busy), 4.8 ms in this form (8,900 warp
// instructions per 32 samples, the multiply pipe 54-65% and the FP64 pipe 35%
// busy with eight warps per SM, the most that 255 registers leave).  Error of a
// gradient against 113-bit arithmetic, largest parameter over the norm, for
// data of a source and noise | of one loud bin: median 3e-16 | 3e-16 ... 1.6e-15,
// where the double form had 6e-16 ... 5e-15 | 1.3e-15 ... 8e-15 (0.4-23 mHz,
// N = 32-1024); beside a source, where the gradient all but vanishes, 2e-14
// against 3e-14.  The adjoint transform alone, N = 1024: 2e-16 (white residual)
// and 2e-17 (one loud bin) of its norm, in double 4e-16.
//
// Candidates outside the fixed-point ranges take the plain double form: each
// sample's forward values (the fast/slow response of
// Sec. II, in the same link form as the likelihood's), then the adjoints
// of the channel samples c_n propagated back through the TDI combination,
// the six links and the three receiver phases to the parameters.  The
// amplitude, inclination and polarisation enter only through the two complex
// polarisation coefficients alpha, gamma (n.H.n = alpha Fp + gamma Fx); their
// adjoints are summed over the samples and contracted with d alpha/d theta,
// d gamma/d theta once per candidate.
//
// Derivatives used (k = propagation direction, u, v the polarisation basis,
// kappa_j = k.x_j/c, f = f0 + fdot t, receiver phase 2 pi cyc_j):
//   d cyc_j/d f0 = t - kappa_j,  d cyc_j/d fdot = (t - kappa_j)^2 / 2,
//   d cyc_j/d beta = -(f - fdot kappa_j) u.x_j/c,
//   d cyc_j/d lambda = -(f - fdot kappa_j) cos(beta) v.x_j/c,  d cyc_j/d phi0 = 1/(2 pi),
//   dk/dbeta = u, dk/dlambda = cos(beta) v, du/dbeta = -k, du/dlambda = -sin(beta) v,
//   dv/dlambda = (cos lambda, sin lambda, 0),
//   d/dX [sinc(X) e^{-iX}] from the derivative of its series (or, evaluated
//   directly, (e^{-2iX} - sinc(X) e^{-iX}) / X).
#include "fp64_common.cuh"
#include "fx64_grad.cuh"

namespace gb {
namespace {

constexpr int kWarpsG = 2;
constexpr int kSumsG = kGSums + 4;   // sums a candidate leaves for its contraction: adjoint_fx's, <d|h>, <h|h>, norm
constexpr int kCapG = 16;   // candidates a warp sets up at a time
constexpr int K = 8;   // f0, fdot, beta, lambda, A, iota, psi, phi0

using C = C64;
// a conj(b)
__device__ __forceinline__ C cmulc(C a, C b) { return {a.x * b.x + a.y * b.y, a.y * b.x - a.x * b.y}; }
// Re(conj(a) b)
__device__ __forceinline__ double redot(C a, C b) { return a.x * b.x + a.y * b.y; }

// Series of the link transfer V(X) = sinc(X) e^{-iX} in y = -4 X^2:
//   Re V = sum_j y^j/(2j+1)!,          Im V = -2X sum_j y^j/(2j+2)!,
//   d Re V/dX = X sum_j y^j (-8(j+1))/(2j+3)!,   d Im V/dX = sum_j y^j (-2(2j+1))/(2j+2)!
// (each coefficient the double nearest its exact rational value)
struct Series4 {
    double re, im, dre, dim;
};
__constant__ Series4 kTransferSeries[17] = {
    {1.0, 0.5, -1.3333333333333333, -1.0},
    {0.16666666666666666, 0.041666666666666664, -0.13333333333333333, -0.25},
    {0.008333333333333333, 0.001388888888888889, -0.004761904761904762, -0.013888888888888888},
    {0.0001984126984126984, 2.48015873015873e-05, -8.818342151675486e-05, -0.00034722222222222224},
    {2.7557319223985893e-06, 2.755731922398589e-07, -1.0020843354176687e-06, -4.96031746031746e-06},
    {2.505210838544172e-08, 2.08767569878681e-09, -7.708341041674375e-09, -4.592886537330982e-08},
    {1.6059043836821613e-10, 1.1470745597729725e-11, -4.282411689819097e-11, -2.9823938554097286e-10},
    {7.647163731819816e-13, 4.779477332387385e-14, -1.7993326427811332e-13, -1.4338431997162156e-12},
    {2.8114572543455206e-15, 1.5619206968586225e-16, -5.918857377569517e-16, -5.310530369319317e-15},
    {8.22063524662433e-18, 4.110317623312165e-19, -1.565835285071301e-18, -1.5619206968586227e-17},
    {1.9572941063391263e-20, 8.896791392450574e-22, -3.403989750155002e-21, -3.7366523848292405e-20},
    {3.868170170630684e-23, 1.6117375710961184e-24, -6.189072273009094e-24, -7.413992827042144e-23},
    {6.446950284384474e-26, 2.4795962632247976e-27, -9.551037458347369e-27, -1.2397981316123987e-25},
    {9.183689863795546e-29, 3.279889237069838e-30, -1.2667158432821444e-29, -1.7711401880177124e-28},
    {1.1309962886447716e-31, 3.7699876288159054e-33, -1.4593500498642214e-32, -2.1865928247132253e-31},
    {1.216125041553518e-34, 3.8003907548547434e-36, -1.4740909594588097e-35, -2.356242268009941e-34},
    {1.151633562077195e-37, 3.387157535521162e-39, -1.3161526423739371e-38, -2.235523973443967e-37},
};

struct CandG {
    double k[3], u[3], v[3], w[3];   // w = dv/dlambda
    double cb, sb;
    C al, ga, al_i[3], ga_i[3];      // alpha, gamma and their derivatives wrt A, iota, psi
    double f0, fd, delta, phi0c;
    double D0r, D0i, eps;            // exp(-i f0/f*), fdot/f*
    int J;
};

// One candidate: its template's constants, and what the gradient adds to the
// fixed-point form, or the plain double form's constants.
struct CandGT {
    CandT t;
    union {
        struct {
            CandGFx g;
            FinGFx fin;
        };
        CandG d;
    };
};

__device__ void setup_grad(const double* th, double T, double inv_fstar, double delta, CandG& c) {
    const double f0 = th[0], fd = th[1], beta = th[2], lam = th[3];
    const double A = th[4], iota = th[5], psi = th[6], phi0 = th[7];
    c.delta = delta;
    c.f0 = f0;
    c.fd = fd;
    c.phi0c = phi0 * 0.15915494309189535;   // 1 / (2 pi)
    double sb, cb, sl, cl, s2, c2, si, ci;
    sincos(beta, &sb, &cb);
    sincos(lam, &sl, &cl);
    sincos(2.0 * psi, &s2, &c2);
    sincos(iota, &si, &ci);
    c.cb = cb;
    c.sb = sb;
    c.k[0] = -(cb * cl);
    c.k[1] = -(cb * sl);
    c.k[2] = -sb;
    c.u[0] = sb * cl;
    c.u[1] = sb * sl;
    c.u[2] = -cb;
    c.v[0] = sl;
    c.v[1] = -cl;
    c.v[2] = 0.0;
    c.w[0] = cl;
    c.w[1] = sl;
    c.w[2] = 0.0;
    const double Ap = A * (1.0 + ci * ci), Ax = -2.0 * A * ci;
    c.al = {Ap * c2, -(Ax * s2)};
    c.ga = {-(Ap * s2), -(Ax * c2)};
    // d/dA
    const double Ap1 = 1.0 + ci * ci, Ax1 = -2.0 * ci;
    c.al_i[0] = {Ap1 * c2, -(Ax1 * s2)};
    c.ga_i[0] = {-(Ap1 * s2), -(Ax1 * c2)};
    // d/diota: dA+ = -2 A cos(iota) sin(iota), dAx = 2 A sin(iota)
    const double dAp = -2.0 * A * ci * si, dAx = 2.0 * A * si;
    c.al_i[1] = {dAp * c2, -(dAx * s2)};
    c.ga_i[1] = {-(dAp * s2), -(dAx * c2)};
    // d/dpsi
    c.al_i[2] = {-2.0 * Ap * s2, -2.0 * Ax * c2};
    c.ga_i[2] = {-2.0 * Ap * c2, 2.0 * Ax * s2};
    // series degree of the link transfer: first omitted term (of the
    // transfer and of its derivative) below 1e-15 for the largest argument
    // X = f (1 + |k.n|)/(2 f*) <= f_max / f*
    const double xmax = fmax(fabs(f0), fabs(f0 + fd * T)) * inv_fstar;
    c.J = xmax <= 0.22 ? 6 : xmax <= 0.5 ? 8 : xmax <= 1.3 ? 12 : xmax <= 2.35 ? 16 : 0;
    double sD, cD;
    sincos(f0 * inv_fstar, &sD, &cD);
    c.D0r = cD;
    c.D0i = -sD;
    c.eps = fd * inv_fstar;
}

// V = sinc(X) e^{-iX} and, with DER, dV/dX
template <bool DER>
__device__ __forceinline__ void transfer(double X, int J, C& V, C& Vd) {
    if (J == 0) {
        double s, co;
        sincos(X, &s, &co);
        const double sinc = X != 0.0 ? s / X : 1.0;
        V = {sinc * co, -(sinc * s)};
        if (DER) {
            const C e2 = {co * co - s * s, -2.0 * s * co};
            Vd = X != 0.0 ? cscale(csub(e2, V), 1.0 / X) : C{0.0, -1.0};
        }
        return;
    }
    const double y = -4.0 * X * X;
    const Series4 cJ = kTransferSeries[J];
    double re = cJ.re, im = cJ.im, dim = cJ.dim, dre = kTransferSeries[J - 1].dre;
    for (int j = J - 1; j >= 0; --j) {
        const Series4 cj = kTransferSeries[j];
        re = fma(re, y, cj.re);
        im = fma(im, y, cj.im);
        if (DER) {
            dim = fma(dim, y, cj.dim);
            if (j > 0) dre = fma(dre, y, kTransferSeries[j - 1].dre);
        }
    }
    V = {re, -2.0 * X * im};
    if (DER) Vd = {X * dre, dim};
}

using Geo = Geo64;

// Forward values of one sample (Sec. II): receiver phasors, the six links
// z_ij = -i a V(a (1 -+ k.n)) (n.H.n) exp(2 pi i cyc), D = exp(-i f/f*) and
// the combinations P of X = (1 - D^2) P (Y, Z likewise).  Link order:
// 01, 10, 12, 21, 20, 02 (arm 0: 01, 10; arm 1: 12, 21; arm 2: 20, 02).
struct Fwd {
    double t, f, a, kap[3];
    C rx[3], z[6], D, omd, PX, PY, PZ;
};

__device__ __forceinline__ void arm_geometry(const CandG& c, const OrbitTables64& tab, int arm, int N, int n,
                                             double& kn, double& nu, double& nv, double& nw) {
    const double nx = tab.arm[(arm * 3 + 0) * N + n], ny = tab.arm[(arm * 3 + 1) * N + n],
                 nz = tab.arm[(arm * 3 + 2) * N + n];
    kn = c.k[0] * nx + c.k[1] * ny + c.k[2] * nz;
    nu = c.u[0] * nx + c.u[1] * ny + c.u[2] * nz;
    nv = c.v[0] * nx + c.v[1] * ny;
    nw = c.w[0] * nx + c.w[1] * ny;
}

// receiver of link l: 01 -> 1, 10 -> 0, 12 -> 2, 21 -> 1, 20 -> 0, 02 -> 2
__device__ __forceinline__ int link_rx(int l) { return l == 0 ? 1 : l == 1 ? 0 : l == 2 ? 2 : l == 3 ? 1 : l == 4 ? 0 : 2; }

__device__ void forward(const CandG& c, const Geo& g, const OrbitTables64& tab, int n, Fwd& fw) {
    const int N = g.N;
    const double inv_c = 1.0 / kC;
    fw.t = (double)n * g.T_over_N;
    const double t = fw.t;
#pragma unroll
    for (int j = 0; j < 3; ++j) {
        const double kap = (c.k[0] * tab.x[(j * 3 + 0) * N + n] + c.k[1] * tab.x[(j * 3 + 1) * N + n] +
                            c.k[2] * tab.x[(j * 3 + 2) * N + n]) * inv_c;
        fw.kap[j] = kap;
        double cyc = c.delta * ((double)n / (double)N) + 0.5 * c.fd * (t * t) - c.f0 * kap - c.fd * t * kap +
                     0.5 * c.fd * (kap * kap) + c.phi0c;
        cyc -= rint(cyc);
        double s, co;
        sincospi(2.0 * cyc, &s, &co);
        fw.rx[j] = {co, s};
    }
    fw.f = c.f0 + c.fd * t;
    fw.a = fw.f * (0.5 * g.inv_fstar);
#pragma unroll
    for (int arm = 0; arm < 3; ++arm) {
        double kn, nu, nv, nw;
        arm_geometry(c, tab, arm, N, n, kn, nu, nv, nw);
        const double Fp = (nu - nv) * (nu + nv), Fx = 2.0 * nu * nv;
        const C G = cadd(cscale(c.al, Fp), cscale(c.ga, Fx));
#pragma unroll
        for (int s = 0; s < 2; ++s) {
            const int l = 2 * arm + s;
            C V, Vd;
            transfer<false>(fw.a * (s == 0 ? 1.0 - kn : 1.0 + kn), c.J, V, Vd);
            const C q = cmul(cmul(cscale(V, fw.a), G), fw.rx[link_rx(l)]);
            fw.z[l] = {q.y, -q.x};   // times -i
        }
    }
    // D = exp(-i f/f*) = exp(-i f0/f*) exp(-i th), th = fdot t/f*: a short
    // series while |th| <= 1/64
    const double th = c.eps * t;
    if (fabs(th) <= 0.015625) {
        const double t2 = th * th;
        const double cs = fma(fma(fma(t2, -1.0 / 720.0, 1.0 / 24.0), t2, -0.5), t2, 1.0);
        const double sn = th * fma(fma(fma(t2, -1.0 / 5040.0, 1.0 / 120.0), t2, -1.0 / 6.0), t2, 1.0);
        fw.D = cmul({c.D0r, c.D0i}, {cs, -sn});
    } else {
        double sD, cD;
        sincos(fw.f * g.inv_fstar, &sD, &cD);
        fw.D = {cD, -sD};
    }
    const C D2 = cmul(fw.D, fw.D);
    fw.omd = {1.0 - D2.x, -D2.y};
    const C* z = fw.z;
    fw.PX = csub(cadd(z[1], cmul(fw.D, z[0])), cadd(z[4], cmul(fw.D, z[5])));
    fw.PY = csub(cadd(z[3], cmul(fw.D, z[2])), cadd(z[0], cmul(fw.D, z[1])));
    fw.PZ = csub(cadd(z[5], cmul(fw.D, z[4])), cadd(z[2], cmul(fw.D, z[3])));
}

constexpr double kR2 = 0.70710678118654752, kR6 = 0.40824829046386302, kR3 = 0.57735026918962576;

// template samples (values) at bit-reversed positions
__device__ void template_value(const CandG& c, const Geo& g, const OrbitTables64& tab, C* bufA, C* bufE, C* bufT,
                               int lane) {
    const int N = g.N;
    for (int n = lane; n < N; n += 32) {
        Fwd fw;
        forward(c, g, tab, n, fw);
        const C X = cmul(fw.omd, fw.PX), Y = cmul(fw.omd, fw.PY), Z = cmul(fw.omd, fw.PZ);
        const int br = (int)(__brev((unsigned)n) >> (32 - g.logN));
        bufA[br] = cscale(csub(Z, X), kR2);
        bufE[br] = cscale(cadd(csub(X, cscale(Y, 2.0)), Z), kR6);
        if (bufT) bufT[br] = cscale(cadd(cadd(X, Y), Z), kR3);
    }
    __syncwarp();
}

// Per-lane gradient accumulators: f0, fdot, beta, lambda, phi0 directly;
// A, iota, psi through the adjoints of alpha and gamma.
struct Acc {
    double f0, fd, beta, lam, phi0;
    C al, ga;
};

// Reverse-mode step of one sample: the adjoints cA, cE (and cT) of the
// channel samples s_n give Re(conj(c) d s_n/d theta) summed into acc.
__device__ void sample_adjoint(const CandG& c, const Geo& g, const OrbitTables64& tab, int n, C cA, C cE, C cT,
                               bool useT, Acc& acc) {
    const int N = g.N;
    Fwd fw;
    forward(c, g, tab, n, fw);
    // A = (Z - X)/sqrt2, E = (X - 2Y + Z)/sqrt6, T = (X + Y + Z)/sqrt3
    C Xb = cadd(cscale(cA, -kR2), cscale(cE, kR6)), Yb = cscale(cE, -2.0 * kR6), Zb = cadd(cscale(cA, kR2),
                                                                                        cscale(cE, kR6));
    if (useT) {
        Xb = cadd(Xb, cscale(cT, kR3));
        Yb = cadd(Yb, cscale(cT, kR3));
        Zb = cadd(Zb, cscale(cT, kR3));
    }
    // X = omd PX, ...
    const C omdb = cadd(cadd(cmulc(Xb, fw.PX), cmulc(Yb, fw.PY)), cmulc(Zb, fw.PZ));
    const C PXb = cmulc(Xb, fw.omd), PYb = cmulc(Yb, fw.omd), PZb = cmulc(Zb, fw.omd);
    // PX = z10 + D z01 - z20 - D z02, PY = z21 + D z12 - z01 - D z10, PZ = z02 + D z20 - z12 - D z21
    const C* z = fw.z;
    C zb[6];
    zb[0] = csub(cmulc(PXb, fw.D), PYb);   // z01
    zb[1] = csub(PXb, cmulc(PYb, fw.D));   // z10
    zb[2] = csub(cmulc(PYb, fw.D), PZb);   // z12
    zb[3] = csub(PYb, cmulc(PZb, fw.D));   // z21
    zb[4] = csub(cmulc(PZb, fw.D), PXb);   // z20
    zb[5] = csub(PZb, cmulc(PXb, fw.D));   // z02
    // D enters the combinations and omd = 1 - D^2
    C Db = cadd(cadd(cmulc(PXb, csub(z[0], z[5])), cmulc(PYb, csub(z[2], z[1]))), cmulc(PZb, csub(z[4], z[3])));
    Db = csub(Db, cmulc(omdb, cscale(fw.D, 2.0)));
    // D = exp(-i f/f*): dD = -i D df/f*
    double fb = (Db.x * fw.D.y - Db.y * fw.D.x) * g.inv_fstar;
    double ab = 0.0;
    C rxb[3] = {{0.0, 0.0}, {0.0, 0.0}, {0.0, 0.0}};
#pragma unroll
    for (int arm = 0; arm < 3; ++arm) {
        double kn, nu, nv, nw;
        arm_geometry(c, tab, arm, N, n, kn, nu, nv, nw);
        const double Fp = (nu - nv) * (nu + nv), Fx = 2.0 * nu * nv;
        const C G = cadd(cscale(c.al, Fp), cscale(c.ga, Fx));
        C Gb = {0.0, 0.0};
        double knb = 0.0;
#pragma unroll
        for (int s = 0; s < 2; ++s) {
            const int l = 2 * arm + s;
            const int j = link_rx(l);
            const double sg = s == 0 ? -1.0 : 1.0;   // X = a (1 + sg kn)
            const double Xa = fw.a * (1.0 + sg * kn);
            C V, Vd;
            transfer<true>(Xa, c.J, V, Vd);
            // z = -i a V W, W = G rx: with zz = i zbar and P = conj(zz) W,
            // abar += Re(P V), Xbar = a Re(P V'), Wbar = a zz conj(V)
            const C zz = {-zb[l].y, zb[l].x};
            const C W = cmul(G, fw.rx[j]);
            const C P = cmulc(W, zz);
            ab += P.x * V.x - P.y * V.y;
            const double Xb_ = fw.a * (P.x * Vd.x - P.y * Vd.y);
            const C Wb = cscale(cmulc(zz, V), fw.a);
            Gb = cadd(Gb, cmulc(Wb, fw.rx[j]));
            rxb[j] = cadd(rxb[j], cmulc(Wb, G));
            ab += Xb_ * (1.0 + sg * kn);
            knb += sg * fw.a * Xb_;
        }
        // G = alpha Fp + gamma Fx
        acc.al = cadd(acc.al, cscale(Gb, Fp));
        acc.ga = cadd(acc.ga, cscale(Gb, Fx));
        const double Fpb = redot(Gb, c.al), Fxb = redot(Gb, c.ga);
        const double nub = 2.0 * (nu * Fpb + nv * Fxb), nvb = 2.0 * (nu * Fxb - nv * Fpb);
        acc.beta += knb * nu - nub * kn;
        acc.lam += knb * c.cb * nv - nub * c.sb * nv + nvb * nw;
    }
    // receiver phases rx_j = exp(2 pi i cyc_j)
    const double inv_c = 1.0 / kC;
#pragma unroll
    for (int j = 0; j < 3; ++j) {
        const double pb = fw.rx[j].x * rxb[j].y - fw.rx[j].y * rxb[j].x;   // Re(conj(rxbar) i rx)
        const double cycb = 2.0 * kPi * pb;
        const double x0 = tab.x[(j * 3 + 0) * N + n], x1 = tab.x[(j * 3 + 1) * N + n],
                     x2 = tab.x[(j * 3 + 2) * N + n];
        const double ux = (c.u[0] * x0 + c.u[1] * x1 + c.u[2] * x2) * inv_c;
        const double vx = (c.v[0] * x0 + c.v[1] * x1) * inv_c;
        const double tk = fw.t - fw.kap[j], fk = fw.f - c.fd * fw.kap[j];
        acc.f0 += cycb * tk;
        acc.fd += 0.5 * cycb * (tk * tk);
        acc.beta -= cycb * fk * ux;
        acc.lam -= cycb * fk * c.cb * vx;
        acc.phi0 += pb;
    }
    // a = f/(2 f*), f = f0 + fdot t
    fb += ab * (0.5 * g.inv_fstar);
    acc.f0 += fb;
    acc.fd += fb * fw.t;
}

__device__ void fft_inplace(int N, int logN, const C* tw, C* bufA, C* bufE, C* bufT, int lane) {
    for (int s = 0; s < logN; ++s) {
        const int h = 1 << s;
        const int tstride = kTwiddles >> s;
        for (int b = lane; b < N / 2; b += 32) {
            const int j = b & (h - 1);
            const int i0 = ((b >> s) << (s + 1)) + j;
            const int i1 = i0 + h;
            const C w = tw[j * tstride];
            const C ua = bufA[i0], va = cmul(w, bufA[i1]);
            bufA[i0] = cadd(ua, va);
            bufA[i1] = csub(ua, va);
            const C ue = bufE[i0], ve = cmul(w, bufE[i1]);
            bufE[i0] = cadd(ue, ve);
            bufE[i1] = csub(ue, ve);
            if (bufT) {
                const C ut = bufT[i0], vt = cmul(w, bufT[i1]);
                bufT[i0] = cadd(ut, vt);
                bufT[i1] = csub(ut, vt);
            }
        }
        __syncwarp();
    }
}

// Gradient of one plain-double candidate (one warp); lane 0 writes row `row`.
__device__ __noinline__ void grad_plain(const CandG& c, long long q, int64_t row, const Geo& g, const OrbitTables64& tab,
                                        const C* tw, C* bufA, C* bufE, C* bufT, const gb_window_t& win, double dd,
                                        const C* __restrict__ dA, const C* __restrict__ dE,
                                        const double* __restrict__ wA, const double* __restrict__ wE,
                                        const C* __restrict__ dT, const double* __restrict__ wT,
                                        double* __restrict__ logL_out, double* __restrict__ grad_out, int lane) {
    const int N = g.N;
    const double T = g.T;
    const bool useT = bufT != nullptr;
    // (1) template
    template_value(c, g, tab, bufA, bufE, bufT, lane);
    fft_inplace(N, g.logN, tw, bufA, bufE, bufT, lane);
    // (2) logL and residual r_m = w (d - h) at DFT index m mod N, in place
    double sdh = 0.0, shh = 0.0;
    for (int idx = lane; idx < N; idx += 32) {
        const int m = idx < N / 2 ? idx : idx - N;      // signed frequency offset
        const int64_t kk = q + m - win.k0;
        const C hA = cscale(bufA[idx], g.scale), hE = cscale(bufE[idx], g.scale);
        C rA = {0.0, 0.0}, rE = {0.0, 0.0};
        if (kk >= 0 && kk < win.W) {
            const C a = dA[win.data_off + kk], e = dE[win.data_off + kk];
            const double wa = wA[win.data_off + kk], we = wE[win.data_off + kk];
            sdh += wa * (a.x * hA.x + a.y * hA.y) + we * (e.x * hE.x + e.y * hE.y);
            shh += wa * (hA.x * hA.x + hA.y * hA.y) + we * (hE.x * hE.x + hE.y * hE.y);
            rA = {wa * (a.x - hA.x), wa * (a.y - hA.y)};
            rE = {we * (e.x - hE.x), we * (e.y - hE.y)};
        }
        // conjugate for the adjoint transform: c = conj(FFT(conj(r)))
        bufA[idx] = {rA.x, -rA.y};
        bufE[idx] = {rE.x, -rE.y};
        if (useT) {
            const C hT = cscale(bufT[idx], g.scale);
            C rT = {0.0, 0.0};
            if (kk >= 0 && kk < win.W) {
                const C t = dT[win.data_off + kk];
                const double wt = wT[win.data_off + kk];
                sdh += wt * (t.x * hT.x + t.y * hT.y);
                shh += wt * (hT.x * hT.x + hT.y * hT.y);
                rT = {wt * (t.x - hT.x), wt * (t.y - hT.y)};
            }
            bufT[idx] = {rT.x, -rT.y};
        }
    }
    sdh = warp_sum(sdh) * (4.0 / T);
    shh = warp_sum(shh) * (4.0 / T);
    __syncwarp();
    // (3) bit-reversal permutation in place, then the same forward FFT
    for (int i = lane; i < N; i += 32) {
        const int j = (int)(__brev((unsigned)i) >> (32 - g.logN));
        if (i < j) {
            const C ta = bufA[i];
            bufA[i] = bufA[j];
            bufA[j] = ta;
            const C te = bufE[i];
            bufE[i] = bufE[j];
            bufE[j] = te;
            if (useT) {
                const C tt = bufT[i];
                bufT[i] = bufT[j];
                bufT[j] = tt;
            }
        }
    }
    __syncwarp();
    fft_inplace(N, g.logN, tw, bufA, bufE, bufT, lane);
    // (4) reverse-mode sweep: the adjoint of sample n is c_n = conj(buf[n])
    Acc acc = {0.0, 0.0, 0.0, 0.0, 0.0, {0.0, 0.0}, {0.0, 0.0}};
    for (int n = lane; n < N; n += 32) {
        const C cA = {bufA[n].x, -bufA[n].y}, cE = {bufE[n].x, -bufE[n].y};
        const C cT = useT ? C{bufT[n].x, -bufT[n].y} : C{0.0, 0.0};
        sample_adjoint(c, g, tab, n, cA, cE, cT, useT, acc);
    }
    double gacc[K];
    gacc[0] = acc.f0;
    gacc[1] = acc.fd;
    gacc[2] = acc.beta;
    gacc[3] = acc.lam;
#pragma unroll
    for (int k = 0; k < 3; ++k) gacc[4 + k] = redot(acc.al, c.al_i[k]) + redot(acc.ga, c.ga_i[k]);
    gacc[7] = acc.phi0;
#pragma unroll
    for (int k = 0; k < K; ++k) gacc[k] = warp_sum(gacc[k]) * (2.0 / (double)N);
    if (lane == 0) {
        if (logL_out) logL_out[row] = sdh - 0.5 * shh - 0.5 * dd;
#pragma unroll
        for (int k = 0; k < K; ++k) grad_out[8 * row + k] = gacc[k];
    }
    __syncwarp();
}

// Bits of |x|'s high word, and the largest of them over a warp: the exponent
// of the largest cotangent without an FP64 compare
__device__ __forceinline__ unsigned abs_hi(double x) { return (unsigned)__double2hiint(x) & 0x7FFFFFFFu; }

// Residual, adjoint transform and sweep of one candidate in fixed point (one
// warp), its template's bin values in buf.  Leaves adjoint_fx's sums in out,
// then <d|h> and <h|h> (before 4/T) and the value of a unit of the cotangents
// (NaN when the data are not finite).
template <int TIER, bool T3>
__device__ __noinline__ void sweep_fx(const CandGT& c, const Geo& g, const FxTab& ft, C* buf, int stride, const gb_window_t& win,
                           const C* __restrict__ dA, const C* __restrict__ dE, const double* __restrict__ wA,
                           const double* __restrict__ wE, const C* __restrict__ dT, const double* __restrict__ wT,
                           int lane, double* out) {
    const int N = g.N, lg = g.logN;
    constexpr int NCH = T3 ? 3 : 2;
    double sdh = 0.0, shh = 0.0;
    unsigned top = 0;
    // conj(r), r = w (d - h), in place at its DFT index
    for (int idx = lane; idx < N; idx += 32) {
        const int m = idx < N / 2 ? idx : idx - N;      // signed frequency offset
        const int64_t kk = c.t.q + m - win.k0;
        const bool in = kk >= 0 && kk < win.W;
        const int e = sw(idx);
#pragma unroll
        for (int ch = 0; ch < NCH; ++ch) {
            C r = {0.0, 0.0};
            if (in) {
                const C h = buf[ch * stride + e], d = (ch == 0 ? dA : ch == 1 ? dE : dT)[win.data_off + kk];
                const double w = (ch == 0 ? wA : ch == 1 ? wE : wT)[win.data_off + kk];
                sdh += w * (d.x * h.x + d.y * h.y);
                shh += w * (h.x * h.x + h.y * h.y);
                r = {w * (d.x - h.x), -(w * (d.y - h.y))};
                top = max(top, max(abs_hi(r.x), abs_hi(r.y)));
            }
            buf[ch * stride + e] = r;
        }
    }
    top = __reduce_max_sync(0xffffffffu, top);
    __syncwarp();
    // to integers, A's normalisation for every channel, and into bit-reversed order
    unsigned share[NCH] = {};
    for (int i = lane; i < N; i += 32) {
#pragma unroll
        for (int ch = 0; ch < NCH; ++ch) {
            const C r = buf[ch * stride + i];
            share[ch] += residual_share(abs_hi(r.x), top) + residual_share(abs_hi(r.y), top);
        }
    }
    unsigned sum = 0;
#pragma unroll
    for (int ch = 0; ch < NCH; ++ch) sum = max(sum, __reduce_add_sync(0xffffffffu, share[ch]));
    __syncwarp();   // every bin is read before it is overwritten
    const int k = residual_shift(sum, top);
    const double s0 = scalbn(1.0, k);
    const double sc[3] = {s0, s0 * 0.57735026918962576, s0 * 0.81649658092772603};
    Z64* z = (Z64*)buf;
    for (int i = lane; i < N; i += 32) {
        const int j = (int)(__brev((unsigned)i) >> (32 - lg));
        if (i > j) continue;
        const int ei = sw(i), ej = sw(j);
#pragma unroll
        for (int ch = 0; ch < NCH; ++ch) {
            const C a = buf[ch * stride + ei], b = buf[ch * stride + ej];
            z[ch * stride + ej] = {__double2ll_rn(a.x * sc[ch]), __double2ll_rn(a.y * sc[ch])};
            z[ch * stride + ei] = {__double2ll_rn(b.x * sc[ch]), __double2ll_rn(b.y * sc[ch])};
        }
    }
    __syncwarp();
    fft_fx<32, true>(z, stride, NCH, lg, ft.tw, sc, lane);
    // normalise: the largest component into [2^59, 2^60)
    unsigned big = 0;
    for (int n = lane; n < N; n += 32) {
        const int e = sw(n);
#pragma unroll
        for (int ch = 0; ch < NCH; ++ch) {
            const Z64 v = z[ch * stride + e];
            const int x = (int)(v.x >> 32), y = (int)(v.y >> 32);
            big = max(big, (unsigned)max(x ^ (x >> 31), y ^ (y >> 31)));
        }
    }
    big = __reduce_max_sync(0xffffffffu, big);
    const int up = __clz(big) - 4;   // left shift, or right when negative
    double acc[32];
#pragma unroll
    for (int j = 0; j < 32; ++j) acc[j] = 0.0;
    double(&sums)[kGSums] = *(double(*)[kGSums])acc;
    for (int n = lane; n < N; n += 32) {
        const int e = sw(n);
        fx gr[3], gi[3];
#pragma unroll
        for (int ch = 0; ch < NCH; ++ch) {
            const Z64 v = z[ch * stride + e];
            gr[ch] = up >= 0 ? v.x << up : v.x >> -up;
            gi[ch] = up >= 0 ? v.y << up : v.y >> -up;
        }
        const int4 a = __ldg(ft.geo + n), b = __ldg(ft.geo + N + n), f = __ldg(ft.geo + 2 * N + n),
                   h = __ldg(ft.geo + 3 * N + n);
        const GeoFx ge{{a.x, a.y}, {a.z, a.w}, {b.x, b.y}, {b.z, b.w}, {f.x, f.y}, {f.z, f.w}, {h.x, h.y}, {h.z, h.w}};
        adjoint_fx<TIER, T3>(c.t.f, c.g, ge, ft.tw, g.krho_q30, n, lg, gr, gi, sums);
    }
    acc[kGSums] = sdh;
    acc[kGSums + 1] = shh;
    // warp sums by halves: lane j ends with the total of value j
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) {
        const bool upper = (lane & o) != 0;
#pragma unroll
        for (int j = 0; j < o; ++j) {
            const double keep = upper ? acc[j + o] : acc[j], send = upper ? acc[j] : acc[j + o];
            acc[j] = keep + __shfl_xor_sync(0xffffffffu, send, o);
        }
    }
    if (lane < kGSums + 2) out[lane] = acc[0];
    if (lane == 31) out[kGSums + 2] = top >= 0x7FF00000u ? nan("") : scalbn(1.0, 60 - k - up);
    __syncwarp();
}

// Resident CTAs per SM, of two warps at 255 registers (five or six at fewer
// registers: 24% slower, from spills in the sweep).
constexpr int kMinCtasG = 4;

__global__ void __launch_bounds__(kWarpsG * 32, kMinCtasG) grad64_kernel(
    const gb_window_t* __restrict__ wins, const Tile* __restrict__ tiles, TabSet64 tabs, const C* __restrict__ tw_g,
    TabSetFx fxt, double T, double fstar, const C* __restrict__ dA, const C* __restrict__ dE,
    const double* __restrict__ wA, const double* __restrict__ wE, const double* __restrict__ theta,
    double* __restrict__ logL_out, double* __restrict__ grad_out, const C* __restrict__ dT,
    const double* __restrict__ wT, int* status, int n_max) {
    extern __shared__ __align__(16) unsigned char smem_raw[];
    FxTw* tw = (FxTw*)smem_raw;                                  // kTwiddles
    double* red = (double*)(tw + kTwiddles);                     // kWarpsG
    CandGT* cands = (CandGT*)(red + kWarpsG);                    // kWarpsG * kCapG
    double* sums = (double*)(cands + kWarpsG * kCapG);           // kWarpsG * kCapG * kSumsG
    C* bufs = (C*)(sums + kWarpsG * kCapG * kSumsG);             // kWarpsG * (2 or 3) * n_max

    const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
    const Tile tile = tiles[blockIdx.x];
    const gb_window_t win = wins[tile.win];
    load_twiddles(fxt.tw, tw);
    // T enters windows whose lowest frequency is at least f*/2 (dT given)
    const bool useT = dT != nullptr && (double)win.k0 / T >= 0.5 * fstar;
    double acc = 0.0;
    for (int i = threadIdx.x; i < win.W; i += blockDim.x) {
        const C a = dA[win.data_off + i], e = dE[win.data_off + i];
        acc += wA[win.data_off + i] * (a.x * a.x + a.y * a.y) + wE[win.data_off + i] * (e.x * e.x + e.y * e.y);
        if (useT) {
            const C t = dT[win.data_off + i];
            acc += wT[win.data_off + i] * (t.x * t.x + t.y * t.y);
        }
    }
    acc = warp_sum(acc);
    if (lane == 0) red[warp] = acc;
    __syncthreads();
    double dd = 0.0;
    for (int w = 0; w < kWarpsG; ++w) dd += red[w];
    dd *= 4.0 / T;

    const Geo g = geometry64(win.N, T, fstar, fxt.arm_c, fxt.krho_q30);
    const OrbitTables64 tab = tabs.t[g.logN - 5];
    const FxTab ft{fxt.geo[g.logN - 5], tw, tw_g};
    C* buf = bufs + (size_t)warp * (dT ? 3 : 2) * n_max;
    CandGT* mycand = cands + warp * kCapG;
    double* mysum = sums + warp * kCapG * kSumsG;
    const int64_t tlen = tile.c_end - tile.c_begin;
    const int64_t grp = (tlen + kWarpsG - 1) / kWarpsG;
    const int64_t c_lo = tile.c_begin + (int64_t)warp * grp;
    const int64_t c_hi = min(tile.c_end, c_lo + grp);
    for (int64_t c0 = c_lo; c0 < c_hi; c0 += kCapG) {
        const int cnt = (int)min((int64_t)kCapG, c_hi - c0);
        if (lane < cnt) {
            CandGT& c = mycand[lane];
            const double* th = theta + 8 * (c0 + lane);
            FxTrig t;
            double si;
            setup_lane(th, g, c.t, t, si);
            if (c.t.tier >= 0 && !setup_gfx(th, T, g.arm_c, t, c.g)) c.t.tier = -1;
            if (c.t.tier >= 0) {
                setup_fin(th, g.arm_c, g.logN, t, si, c.fin);
            } else if (!c.t.bad) {
                setup_grad(th, T, g.inv_fstar, __dadd_rn(__dmul_rn(th[0], T), -(double)c.t.q), c.d);
            }
        }
        __syncwarp();
        for (int i = 0; i < cnt; ++i) {
            const CandGT& c = mycand[i];
            if (c.t.bad) continue;
            if (c.t.tier < 0) {
                grad_plain(c.d, c.t.q, c0 + i, g, tab, tw_g, buf, buf + n_max, useT ? buf + 2 * n_max : nullptr, win,
                           dd, dA, dE, wA, wE, dT, wT, logL_out, grad_out, lane);
                continue;
            }
            template_any<32>(c.t, g, tab, ft, buf, n_max, useT, lane);
            double* s = mysum + i * kSumsG;
            if (c.t.tier == 0) {
                if (useT) sweep_fx<0, true>(c, g, ft, buf, n_max, win, dA, dE, wA, wE, dT, wT, lane, s);
                else sweep_fx<0, false>(c, g, ft, buf, n_max, win, dA, dE, wA, wE, dT, wT, lane, s);
            } else {
                if (useT) sweep_fx<1, true>(c, g, ft, buf, n_max, win, dA, dE, wA, wE, dT, wT, lane, s);
                else sweep_fx<1, false>(c, g, ft, buf, n_max, win, dA, dE, wA, wE, dT, wT, lane, s);
            }
        }
        // the sums' contraction, one candidate per lane
        if (lane < cnt) {
            const CandGT& c = mycand[lane];
            const int64_t row = c0 + lane;
            if (c.t.bad) {
                if (logL_out) logL_out[row] = nan("");
                for (int k = 0; k < K; ++k) grad_out[8 * row + k] = nan("");
                atomicOr(status, kStatusNonFinite);
            } else if (c.t.tier >= 0) {
                const double* s = mysum + lane * kSumsG;
                double gout[K];
                finish_gfx(c.fin, T, s, s[kGSums + 2], gout);
                if (logL_out) logL_out[row] = s[kGSums] * (4.0 / T) - 0.5 * (s[kGSums + 1] * (4.0 / T)) - 0.5 * dd;
                for (int k = 0; k < K; ++k) grad_out[8 * row + k] = gout[k];
            }
        }
        __syncwarp();
    }
}

}  // namespace

int launch_grad_fp64(gb_ctx* ctx, const Plan& plan, const double* dA, const double* dE, const double* wA,
                     const double* wE, const double* theta, double* logL, double* grad, const double* dT,
                     const double* wT, cudaStream_t s) {
    if (plan.n_tiles == 0) return GB_OK;
    const size_t smem = sizeof(FxTw) * kTwiddles + sizeof(double) * kWarpsG +
                        (sizeof(CandGT) + sizeof(double) * kSumsG) * kWarpsG * kCapG +
                        sizeof(C) * kWarpsG * (dT ? 3 : 2) * (size_t)plan.n_max;
    cudaError_t e = cudaFuncSetAttribute(grad64_kernel, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)smem);
    if (e != cudaSuccess) return cuda_error(ctx, e, "grad64: smem attribute");
    grad64_kernel<<<plan.n_tiles, kWarpsG * 32, smem, s>>>(plan.d_win, plan.d_tiles, tabset64(ctx),
                                                           (const C*)ctx->d_tw64, tabset_fx(ctx), ctx->obs.T_obs,
                                                           transfer_frequency(ctx), (const C*)dA, (const C*)dE,
                                                           wA, wE, theta, logL, grad, (const C*)dT, wT,
                                                           ctx->d_status, plan.n_max);
    ++ctx->launches;
    e = cudaGetLastError();
    if (e != cudaSuccess) return cuda_error(ctx, e, "grad64 launch");
    return GB_OK;
}

}  // namespace gb
