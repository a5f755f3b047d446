// The fixed-point headers compiled for the host (tests/test_fx64_host.py).
#include <vector>

#include "fx64_grad.cuh"

using namespace gb;

namespace {

// sample constants from doubles, as the device tables hold them
GeoFx geometry(const double* v) {
    return GeoFx{to_bx(v[0], 0x1p62), to_bx(v[1], 0x1p62), to_bx(v[2], 0x1p62), to_bx(v[3], 0x1p62),
                 to_bx(v[4], 0x1p62), to_bx(v[5], 0x1p62), to_bx(v[6], 0x1p62), to_bx(v[7], 0x1p62)};
}
int krho(double arm_c) { return (int)rint(arm_c / 3072.0 * 1073741824.0); }
FxTrig trig(const double* th, double arm_c) {
    const double a0 = 3.14159265358979323846 * th[0] * arm_c;
    return FxTrig{sin(th[2]), cos(th[2]), sin(th[3]), cos(th[3]), sin(2 * th[6]), cos(2 * th[6]), cos(th[5]), sin(a0), cos(a0)};
}
std::vector<FxTw> twiddles() {
    std::vector<FxTw> t(512);
    for (int k = 0; k < 512; ++k) {
        const long double x = 2.0L * 3.14159265358979323846264338327950288L * k / 1024.0L;
        t[k] = FxTw{bal((fx)llrintl(cosl(x) * 0x1p62L)), bal((fx)llrintl(sinl(x) * 0x1p62L))};
    }
    return t;
}

template <int TIER>
void samples(const CandFx& c, const std::vector<FxTw>& tw, const double* geo, double arm_c, int lg, fx* out) {
    for (int n = 0; n < 1 << lg; ++n) {
        fx o[6];
        sample_fx<TIER, true>(c, geometry(geo + 8 * n), tw.data(), krho(arm_c), n, lg, fx_shift(lg), o);
        for (int k = 0; k < 6; ++k) out[6 * n + k] = o[k];
    }
}
template <int TIER>
void sweep(const CandFx& c, const CandGFx& cg, const std::vector<FxTw>& tw, const double* geo, double arm_c, int lg,
           const fx* cot, double* sums) {
    double acc[kGSums] = {};
    for (int n = 0; n < 1 << lg; ++n) {
        fx gr[3], gi[3];
        for (int k = 0; k < 3; ++k) {
            gr[k] = cot[6 * n + 2 * k];
            gi[k] = cot[6 * n + 2 * k + 1];
        }
        adjoint_fx<TIER, true>(c, cg, geometry(geo + 8 * n), tw.data(), krho(arm_c), n, lg, gr, gi, acc);
    }
    for (int k = 0; k < kGSums; ++k) sums[k] = acc[k];
}

// what the compiler calls at a signed overflow: counted, with the last line
int g_overflows = 0, g_line = 0;
struct Location {
    const char* file;
    unsigned line, column;
};
void overflow(void* at) {
    ++g_overflows;
    g_line = (int)((Location*)at)->line;
}

}  // namespace

extern "C" {

void __ubsan_handle_add_overflow(void* at, void*, void*) { overflow(at); }
void __ubsan_handle_sub_overflow(void* at, void*, void*) { overflow(at); }
void __ubsan_handle_mul_overflow(void* at, void*, void*) { overflow(at); }
void __ubsan_handle_negate_overflow(void* at, void*) { overflow(at); }

// signed overflows since the last call, and the line of the last one
int host_overflows(int* line) {
    const int n = g_overflows;
    *line = g_line;
    g_overflows = 0;
    return n;
}

// tier of each of B candidates, and the samples A, E, T (re, im) of those in
// the fixed-point ranges; scale: a channel's bin value per unit of its transform
void host_samples(int B, const double* theta, const double* delta, double T, double arm_c, int lg, const double* geo,
                  int* tier, fx* out, double* scale) {
    const auto tw = twiddles();
    for (int b = 0; b < B; ++b) {
        CandFx c{};
        setup_fx(theta + 8 * b, T, arm_c, delta[b], lg, trig(theta + 8 * b, arm_c), c);
        tier[b] = c.tier;
        scale[3 * b] = c.sA;
        scale[3 * b + 1] = c.sE;
        scale[3 * b + 2] = c.sT;
        fx* o = out + (size_t)b * 6 * (1 << lg);
        if (c.tier == 0) samples<0>(c, tw, geo, arm_c, lg, o);
        else if (c.tier == 1) samples<1>(c, tw, geo, arm_c, lg, o);
    }
}

// gradients of B candidates for cotangents cot (N x 3 complex per candidate, Q60, |re|, |im| <= 1)
void host_gradients(int B, const double* theta, const double* delta, double T, double arm_c, int lg, const double* geo,
                    const fx* cot, int* tier, double* grad) {
    const auto tw = twiddles();
    for (int b = 0; b < B; ++b) {
        const double* th = theta + 8 * b;
        CandFx c{};
        CandGFx cg{};
        FinGFx fin{};
        const FxTrig t = trig(th, arm_c);
        setup_fx(th, T, arm_c, delta[b], lg, t, c);
        tier[b] = c.tier;
        if (c.tier < 0 || !setup_gfx(th, T, arm_c, t, cg)) continue;
        setup_fin(th, arm_c, lg, t, sin(th[5]), fin);
        double sums[kGSums];
        const fx* g = cot + (size_t)b * 6 * (1 << lg);
        if (c.tier == 0) sweep<0>(c, cg, tw, geo, arm_c, lg, g, sums);
        else sweep<1>(c, cg, tw, geo, arm_c, lg, g, sums);
        finish_gfx(fin, T, sums, 0x1p-60 * 0x1p60, grad + 8 * b);
    }
}

// transform of B residuals (N complex each): N integers and the power of two that they carry
void host_transform(int B, int lg, const double* r, fx* out, int* power) {
    const auto tw = twiddles();
    const int N = 1 << lg;
    const double one[3] = {1.0, 1.0, 1.0};
    std::vector<Z64> z(N);
    for (int b = 0; b < B; ++b) {
        const double* x = r + (size_t)b * 2 * N;
        auto high = [&](int i) { return (unsigned)((uint64_t)double_bits(fabs(x[i])) >> 32); };
        unsigned top = 0, sum = 0;
        for (int i = 0; i < 2 * N; ++i) top = high(i) > top ? high(i) : top;
        for (int i = 0; i < 2 * N; ++i) sum += residual_share(high(i), top);
        const int k = power[b] = residual_shift(sum, top);
        for (int i = 0; i < N; ++i) {
            int j = 0;
            for (int q = 0; q < lg; ++q) j |= ((i >> q) & 1) << (lg - 1 - q);
            z[sw(j)] = Z64{to_fx(ldexp(x[2 * i], k), 1.0), to_fx(ldexp(x[2 * i + 1], k), 1.0)};
        }
        fft_fx<1, true>(z.data(), N, 1, lg, tw.data(), one, 0);
        for (int i = 0; i < N; ++i) {
            out[((size_t)b * N + i) * 2] = z[sw(i)].x;
            out[((size_t)b * N + i) * 2 + 1] = z[sw(i)].y;
        }
    }
}
}
