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
#include "fp64_common.cuh"

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
            if (warp == 0) setup_warp(theta + 8 * row, 1, g, cands, lane);
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

// Sum, minimum over the NT threads that work on a window (a warp or the CTA;
// `red`: kWarps64 doubles of the CTA).
template <int NT>
__device__ __forceinline__ double group_sum(double v, double* red) {
    v = warp_sum(v);
    if (NT == 32) return v;
    __syncthreads();
    if ((threadIdx.x & 31) == 0) red[threadIdx.x >> 5] = v;
    __syncthreads();
    double s = 0.0;
    for (int w = 0; w < kWarps64; ++w) s += red[w];
    return s;
}
template <int NT>
__device__ __forceinline__ int group_min(int v, double* red) {
    v = __reduce_min_sync(0xffffffffu, v);
    if (NT == 32) return v;
    int* r = (int*)red;
    __syncthreads();
    if ((threadIdx.x & 31) == 0) r[threadIdx.x >> 5] = v;
    __syncthreads();
    for (int w = 0; w < kWarps64; ++w) v = min(v, r[w]);
    return v;
}
// a template in its buffers (bin values in natural order at sw(index)), its
// carrier bin and the window bins [lo, hi) that it reaches
struct WinTpl {
    C64 *A, *E;
    long long q;
    int lo, hi;
    bool bad;
};
__device__ __forceinline__ void place(WinTpl& t, const CandT& c, const gb_window_t& win) {
    t.q = c.q;
    t.bad = c.bad;
    const long long l = c.q - win.N / 2 - win.k0, h = l + win.N;
    t.lo = (int)min(max(l, 0LL), (long long)win.W);
    t.hi = (int)min(max(h, 0LL), (long long)win.W);
}
__device__ __forceinline__ int tpl_index(const WinTpl& t, const gb_window_t& win, int i) {
    return sw((int)((win.k0 + i - t.q) & (win.N - 1)));
}
__device__ __forceinline__ bool finite_bits(double x) { return (~__double2hiint(x) & 0x7ff00000) != 0; }

// Gram matrix G_ij = <s_i|s_j>, b_i = <d|s_i> and the multi-signal SNR
// rho = sum_i b_i / sqrt(sum_ij G_ij) (Eq. 11) of each window's sources (the
// sources are the window's candidate rows), with <x|y> = (4/T) Re sum_k w_k
// x_k y_k* in a fixed order.  NT threads work on a window, a warp or a CTA.
// Template i is held in buffer P while the templates j > i pass through Q, the
// next one last, so that it is P's content for i + 1: K (K-1)/2 + 1 templates.
// A sum runs over the bins that its templates share; a weight or datum outside
// them counts only by being non-finite (its product with zero is NaN), for
// which the window is looked through once.
// Bound by the FP64 and integer pipes and the set-ups' latency; 4,096 pairs,
// N = 64-256, W = 2 N: 0.80 ms with one set-up at a time, template 1 computed
// twice and five passes over all W bins, 0.50 ms now with a CTA per window,
// 0.44 ms with a warp per window.
constexpr int kGramSlots = kSetupWarp + 2;      // candidate slots of a window: those set up together, one for later ones
static_assert(sizeof(CandT) * kGramSlots % 16 == 0, "the buffers behind the slots are read in 16-byte elements");
template <int NT>
__global__ void __launch_bounds__(kWarps64 * 32, kMinCtas64) multi_gram_kernel(
    const gb_window_t* __restrict__ wins, int n_win, TabSet64 tabs, const C64* __restrict__ tw_g, TabSetFx fxt,
    double T, double fstar, const C64* __restrict__ dA, const C64* __restrict__ dE, const double* __restrict__ wA,
    const double* __restrict__ wE, const double* __restrict__ theta, int kmax, double* __restrict__ gram,
    double* __restrict__ dh_out, double* __restrict__ rho_out, int* status, int n_max) {
    constexpr int GROUPS = kWarps64 * 32 / NT;  // windows in work per CTA
    extern __shared__ __align__(16) unsigned char smem_raw[];
    FxTw* tw = (FxTw*)smem_raw;                 // kTwiddles
    double* red = (double*)(tw + kTwiddles);    // kWarps64
    const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31, tid = threadIdx.x & (NT - 1);
    const int group = GROUPS == 1 ? 0 : warp;
    CandT* cand = (CandT*)(red + kWarps64) + group * kGramSlots;
    C64* bufs = (C64*)((CandT*)(red + kWarps64) + GROUPS * kGramSlots) + (size_t)group * 4 * n_max;
    load_twiddles(fxt.tw, tw);
    __syncthreads();
    const bool data = dA != nullptr;
    for (int w = blockIdx.x * GROUPS + group; w < n_win; w += gridDim.x * GROUPS) {
        const gb_window_t win = wins[w];
        const int K = win.n_cand;
        const double* th = theta + 8 * win.cand_off;
        double* G = gram + (size_t)w * kmax * kmax;
        const Geo64 g = geometry64(win.N, T, fstar, fxt.arm_c, fxt.krho_q30);
        const OrbitTables64 tab = tabs.t[g.logN - 5];
        const FxTab ft{fxt.geo[g.logN - 5], tw, tw_g};
        const double* pwA = wA + win.data_off;
        const double* pwE = wE + win.data_off;
        // first and last bin with a non-finite weight, with a non-finite datum
        int w_first = win.W, w_last = 0, d_first = win.W, d_last = 0;
        if (K > 0) {
            for (int i = tid; i < win.W; i += NT) {
                if (!finite_bits(pwA[i]) || !finite_bits(pwE[i])) {
                    w_first = min(w_first, i);
                    w_last = min(w_last, -i - 1);
                }
                if (data) {
                    const C64 a = dA[win.data_off + i], e = dE[win.data_off + i];
                    if (!finite_bits(a.x) || !finite_bits(a.y) || !finite_bits(e.x) || !finite_bits(e.y)) {
                        d_first = min(d_first, i);
                        d_last = min(d_last, -i - 1);
                    }
                }
            }
            w_first = group_min<NT>(w_first, red);
            w_last = -group_min<NT>(w_last, red);    // one past the last
            d_first = group_min<NT>(d_first, red);
            d_last = -group_min<NT>(d_last, red);
        }
        sync_nt<NT>();                          // the slots and buffers of the window before are done with
        if (K > 0 && (GROUPS > 1 || warp == 0)) setup_warp(th, min(K, kSetupWarp), g, cand, lane);
        sync_nt<NT>();
        // template k into t's buffers
        auto compute = [&](int k, WinTpl& t) {
            if (k >= kSetupWarp) {
                sync_nt<NT>();
                if (GROUPS > 1 || warp == 0) setup_warp(th + 8 * k, 1, g, cand + kSetupWarp, lane);
                sync_nt<NT>();
            }
            const CandT& c = cand[k < kSetupWarp ? k : kSetupWarp];
            place(t, c, win);
            sync_nt<NT>();                      // the buffer's last reads
            if (!t.bad) template_any<NT>(c, g, tab, ft, t.A, n_max, false, tid);
            sync_nt<NT>();
        };
        WinTpl P, Q;
        P.A = bufs;
        P.E = bufs + n_max;
        Q.A = bufs + 2 * n_max;
        Q.E = bufs + 3 * n_max;
        double sum_b = 0.0, sum_g = 0.0;
        bool bad_any = false;
        for (int i = 0; i < K; ++i) {
            if (i == 0) compute(0, P);
            double gii = nan(""), bi = nan("");
            if (!P.bad) {
                const bool odd = w_first < P.lo || w_last > P.hi;
                double sg = 0.0, sb = 0.0;
                for (int k = P.lo + tid; k < P.hi; k += NT) {
                    const int idx = tpl_index(P, win, k);
                    const C64 xa = P.A[idx], xe = P.E[idx];
                    const double va = pwA[k], ve = pwE[k];
                    sg += va * (xa.x * xa.x + xa.y * xa.y) + ve * (xe.x * xe.x + xe.y * xe.y);
                    if (data) {
                        const C64 ya = dA[win.data_off + k], ye = dE[win.data_off + k];
                        sb += va * (xa.x * ya.x + xa.y * ya.y) + ve * (xe.x * ye.x + xe.y * ye.y);
                    }
                }
                gii = odd ? nan("") : group_sum<NT>(sg, red) * (4.0 / T);
                if (data)
                    bi = odd || d_first < P.lo || d_last > P.hi ? nan("") : group_sum<NT>(sb, red) * (4.0 / T);
            }
            if (tid == 0) {
                G[i * kmax + i] = gii;
                if (dh_out) dh_out[win.cand_off + i] = bi;
                if (P.bad) atomicOr(status, kStatusNonFinite);
                sum_b += bi;
                sum_g += gii;
                bad_any |= P.bad;
            }
            for (int j = K - 1; j > i; --j) {
                compute(j, Q);
                double gij = nan("");
                if (!P.bad && !Q.bad) {
                    const int lo = max(P.lo, Q.lo), hi = min(P.hi, Q.hi);
                    const bool odd = lo < hi ? w_first < lo || w_last > hi : w_last > 0;
                    double sg = 0.0;
                    for (int k = lo + tid; k < hi; k += NT) {
                        const int ip = tpl_index(P, win, k), iq = tpl_index(Q, win, k);
                        const C64 xa = P.A[ip], xe = P.E[ip], ya = Q.A[iq], ye = Q.E[iq];
                        sg += pwA[k] * (xa.x * ya.x + xa.y * ya.y) + pwE[k] * (xe.x * ye.x + xe.y * ye.y);
                    }
                    gij = odd ? nan("") : group_sum<NT>(sg, red) * (4.0 / T);
                }
                if (tid == 0) {
                    G[i * kmax + j] = gij;
                    G[j * kmax + i] = gij;
                    sum_g += 2.0 * gij;
                }
            }
            if (i + 1 < K) {
                const WinTpl t = P;
                P = Q;
                Q = t;
            }
        }
        if (tid == 0 && rho_out) rho_out[w] = (K == 0 || bad_any || !data) ? nan("") : sum_b / sqrt(sum_g);
    }
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
    int sms = 152;
    cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, ctx->device);
    // a warp per window needs windows for all SMs' warps, and short templates
    // (four buffers each) to have eight of them resident
    const bool by_warp = n_max <= 256 && n_win >= 4 * sms;
    const int groups = by_warp ? kWarps64 : 1;
    const size_t smem = sizeof(FxTw) * kTwiddles + sizeof(double) * kWarps64 +
                        groups * (sizeof(CandT) * kGramSlots + sizeof(C64) * 4 * (size_t)n_max);
    const auto kfn = by_warp ? multi_gram_kernel<32> : multi_gram_kernel<kWarps64 * 32>;
    cudaError_t e = cudaFuncSetAttribute(kfn, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)smem);
    if (e != cudaSuccess) return cuda_error(ctx, e, "multi_gram: smem attribute");
    int bpsm = 0;
    if (cudaOccupancyMaxActiveBlocksPerMultiprocessor(&bpsm, kfn, kWarps64 * 32, smem) != cudaSuccess || bpsm < 1) bpsm = 1;
    const int grid = std::min((n_win + groups - 1) / groups, sms * bpsm);
    kfn<<<grid, kWarps64 * 32, smem, s>>>(d_win, n_win, tabset64(ctx), (const C64*)ctx->d_tw64, tabset_fx(ctx),
                                          ctx->obs.T_obs, transfer_frequency(ctx), (const C64*)dA, (const C64*)dE, wA,
                                          wE, theta, kmax, gram, dh, rho, ctx->d_status, n_max);
    ++ctx->launches;
    e = cudaGetLastError();
    if (e != cudaSuccess) return cuda_error(ctx, e, "multi_gram launch");
    return GB_OK;
}

}  // namespace gb
