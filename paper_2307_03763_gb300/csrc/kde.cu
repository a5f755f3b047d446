// kde.cu -- paired two-dimensional kernel-density proposals of the annealed
// posterior (Sec. III.G, Alg. 4).
//
// The posterior of a recovered signal is sampled over a reduced box around
// the MLE.  The first temperature draws uniformly from the box; afterwards the
// chain obtained at one temperature, smoothed by a kernel density estimate,
// is the proposal of the next.  The estimates are two-dimensional, one per
// parameter pair: (f0, fdot), (lambda, beta), (A, iota); psi and phi0 stay
// uniform over their narrow ranges.
//
// Each pair's estimate is a G x G grid.  It spans the chain's own range on
// each axis, [max(lo, a - 3h - c0), min(hi, b + 3h + c0)] for entries in
// [a, b], bandwidth h and box cell c0 = (hi - lo)/G, so that its resolution
// follows the posterior (the first temperature's grids span the box):
//   * the chain's n entries are counted per cell, cell index
//     floor((x - lo') / (hi' - lo') * G) clamped to the grid;
//   * the counts are smoothed per axis by a Gaussian kernel of Scott's
//     bandwidth for two dimensions, h = s n_eff^(-1/6) (s the standard
//     deviation of the n entries, n_eff the accepted moves + 1), truncated at
//     min(ceil(3 h / cell), G - 1) cells and normalised to sum one; mass
//     pushed past the grid edge is dropped;
//   * the result is normalised and mixed with a uniform floor eps, and
//     stored as cumulative sums C over the flattened cells c = i G + j.
// A draw takes the first cell with C_c > u and a uniform point in it; its
// density is (C_c - C_(c-1)) / cell area, exactly the probability the draw
// has.  A cluster of eight CTAs builds one pair of one window (counts, both
// smoothing passes and the prefix sums in shared memory); one thread draws one
// proposal.
#include <cooperative_groups.h>

#include <cmath>

#include "gb_internal.cuh"

namespace cg = cooperative_groups;

namespace gb {
namespace {

constexpr int kKdeThreads = 256;
constexpr int kKdeCtas = 8;                  // CTAs of a build cluster
constexpr int kKdeVirt = 32 * kKdeCtas;      // partial sums of an ordered sum

__device__ __forceinline__ void pair_dims(int p, int& dx, int& dy) {
    dx = p == 0 ? 0 : p == 1 ? 3 : 4;
    dy = p == 0 ? 1 : p == 1 ? 2 : 5;
}

// cell of value v in [lo, hi] with G cells, clamped (a non-finite value goes to cell 0)
__device__ __forceinline__ int kde_cell(double v, double lo, double hi, int G) {
    const double t = __dmul_rn(__ddiv_rn(__dadd_rn(v, -lo), __dadd_rn(hi, -lo)), (double)G);
    if (!(t >= 0.0)) return 0;
    if (t >= (double)(G - 1)) return G - 1;
    return (int)floor(t);
}

// the same cell, in float when the value is well inside one (t in float is
// within 3e-5 of the exact quotient times G <= 128); gi = G/(hi - lo)
__device__ __forceinline__ int kde_cell_fast(double v, double lo, double hi, int G, float gi) {
    const float t = (float)__dadd_rn(v, -lo) * gi;
    const int c = (int)t;
    const float fr = t - (float)c;
    if (t > 1e-3f && t < (float)(G - 1) && fr > 1e-3f && fr < 0.999f) return c;
    return kde_cell(v, lo, hi, G);
}

// grid extent of one axis: the entries' range [a, b] widened by 3h and a box cell, inside the box
__device__ __forceinline__ void grid_extent(double a, double b, double h, double lo, double hi, int G, double& e0,
                                            double& e1) {
    const double c0 = __ddiv_rn(__dadd_rn(hi, -lo), (double)G), h3 = __dmul_rn(3.0, h);
    e0 = fmax(lo, __dadd_rn(__dadd_rn(a, -h3), -c0));
    e1 = fmin(hi, __dadd_rn(__dadd_rn(b, h3), c0));
}

// Truncation of the Gaussian kernel of width sigma (in cells): offsets -r..r;
// r = 0 for sigma = 0 or non-finite
__device__ __forceinline__ int kernel_radius(double sigma, int G) {
    return sigma > 0.0 && isfinite(sigma) ? (int)fmin(ceil(3.0 * sigma), (double)(G - 1)) : 0;
}

// What the CTAs of a cluster tell each other: sums and range of their entries
// (pass 0), spreads (pass 1), the totals of the smoothed cells and of the
// chunks of cumulative sums.
struct KdeShare {
    double sx[kKdeCtas], sy[kKdeCtas], ax[kKdeCtas], bx[kKdeCtas], ay[kKdeCtas], by[kKdeCtas];
    double vx[kKdeCtas], vy[kKdeCtas], tot[kKdeCtas];
    double part[kKdeVirt];   // chunk sums, then their exclusive prefix sums (CTA 0)
    int acc[kKdeCtas];
};

__device__ __forceinline__ double wsum_kde(double v) {
    for (int o = 16; o > 0; o >>= 1) v += __shfl_xor_sync(0xffffffffu, v, o);
    return v;
}
__device__ __forceinline__ double sum_ranks(const double* v) {
    double s = v[0];
    for (int w = 1; w < kKdeCtas; ++w) s += v[w];
    return s;
}

// One cluster of 8 CTAs builds one pair of one window.  Bound by latency: a
// few FP64 chains (the ordered sums, exp, pow) and the gathers behind the
// chain.  The sums keep the order of 256 partial sums (entry i in partial sum
// i mod 256, each in order of i, combined by a shuffle tree per 32 and in order
// over the eight): CTA r holds partial sums 32 r .. 32 r + 31, so the FP64 work
// and the gathers spread over eight SMs.  Counts go to the CTA that owns the
// cell's row block by distributed-shared-memory atomics.  16 windows of 10,000
// entries, grid 64: 80 us (332 us for one CTA per pair: a division per entry,
// serial exponentials, one SM's FP64 pipe).
__global__ void __cluster_dims__(kKdeCtas, 1, 1) __launch_bounds__(kKdeThreads)
    kde_build_kernel(int n, int G, const double* __restrict__ theta, const int32_t* __restrict__ chain,
                     const double* __restrict__ box, double eps, double* __restrict__ cdf, double* __restrict__ ext,
                     int store) {
    cg::cluster_group cl = cg::this_cluster();
    const int r = (int)cl.block_rank();
    const int w = blockIdx.x / kKdeCtas, p = blockIdx.y, GG = G * G;
    const int tid = threadIdx.x, warp = tid >> 5, lane = tid & 31;
    int dx, dy;
    pair_dims(p, dx, dy);
    // rows of the grid this CTA smooths: [i0, i1)
    const int rows = (G + kKdeCtas - 1) / kKdeCtas;
    const int i0 = min(G, r * rows), i1 = min(G, i0 + rows);
    extern __shared__ __align__(16) unsigned char smem_raw[];
    KdeShare* sh = (KdeShare*)smem_raw;
    double* we = (double*)(sh + 1);                        // 2 x 2G: kernel weights before normalisation
    double* par = we + 4 * G;                              // extents, 1/cell factors, weight totals
    float* kx = (float*)(par + 8);                         // 2G
    float* ky = kx + 2 * G;                                // 2G
    int* own = (int*)(ky + 2 * G);                         // rows x G: counts of the own rows
    int* cnt = own + rows * G;                             // GG: all counts
    float* S1 = (float*)(cnt + GG);                        // rows x G
    float* S2 = S1 + rows * G;                             // rows x G
    double2* ent = (double2*)(((uintptr_t)(S2 + rows * G) + 15) & ~(uintptr_t)15);   // the CTA's entries (x, y), if stored
    const double* bx = box + 16 * (size_t)w;
    const double lox = bx[dx], hix = bx[8 + dx], loy = bx[dy], hiy = bx[8 + dy];
    for (int c = tid; c < rows * G; c += kKdeThreads) own[c] = 0;
    const double* th = theta + 8 * (size_t)w * n;
    const int32_t* ch = chain + (size_t)w * n;
    // entry e of this CTA is entry i = 32 r + (e mod 32) + 256 (e / 32) of the chain
    const int ne = n > 32 * r ? ((n - 32 * r + kKdeVirt - 1) / kKdeVirt) * 32 : 0;
    auto index = [&](int e) { return 32 * r + (e & 31) + kKdeVirt * (e >> 5); };
    auto entry = [&](int e, int i) {
        if (store) return ent[e];
        const int s = min(max(ch[i], 0), n - 1);
        return make_double2(th[8 * (size_t)s + dx], th[8 * (size_t)s + dy]);
    };
    double ax = INFINITY, bx_ = -INFINITY, ay = INFINITY, by_ = -INFINITY;
    int acc = 0;
    for (int e = tid; e < ne; e += kKdeThreads) {
        const int i = index(e);
        if (i >= n) continue;
        const int s = min(max(ch[i], 0), n - 1);
        if (i >= 1 && s == i) ++acc;
        const double2 v = make_double2(th[8 * (size_t)s + dx], th[8 * (size_t)s + dy]);
        if (store) ent[e] = v;
        ax = fmin(ax, v.x);
        bx_ = fmax(bx_, v.x);
        ay = fmin(ay, v.y);
        by_ = fmax(by_, v.y);
    }
    __shared__ double red[4][kKdeThreads / 32];
    __shared__ int redc[kKdeThreads / 32];
    for (int o = 16; o > 0; o >>= 1) {
        ax = fmin(ax, __shfl_xor_sync(0xffffffffu, ax, o));
        bx_ = fmax(bx_, __shfl_xor_sync(0xffffffffu, bx_, o));
        ay = fmin(ay, __shfl_xor_sync(0xffffffffu, ay, o));
        by_ = fmax(by_, __shfl_xor_sync(0xffffffffu, by_, o));
        acc += __shfl_xor_sync(0xffffffffu, acc, o);
    }
    if (lane == 0) {
        red[0][warp] = ax;
        red[1][warp] = bx_;
        red[2][warp] = ay;
        red[3][warp] = by_;
        redc[warp] = acc;
    }
    // a CTA's shared memory may be reached only once it runs: no remote store
    // before this barrier (behind the gathers, whose latency hides it)
    cl.sync();
    // ordered sums: x in warp 0, y in warp 1; range and moves in warp 2
    if (warp < 2) {
        double s = 0.0;
        for (int e = lane; e < ne; e += 32) {
            const int i = index(e);
            if (i >= n) break;
            const double2 v = entry(e, i);
            s += warp == 0 ? v.x : v.y;
        }
        s = wsum_kde(s);
        if (lane < kKdeCtas) {
            KdeShare* o = cl.map_shared_rank(sh, lane);
            if (warp == 0) o->sx[r] = s;
            else o->sy[r] = s;
        }
    } else if (warp == 2 && lane < kKdeCtas) {
        double v[4];
        for (int m = 0; m < 4; ++m) {
            v[m] = red[m][0];
            for (int q = 1; q < kKdeThreads / 32; ++q) v[m] = m & 1 ? fmax(v[m], red[m][q]) : fmin(v[m], red[m][q]);
        }
        int a = 0;
        for (int q = 0; q < kKdeThreads / 32; ++q) a += redc[q];
        KdeShare* o = cl.map_shared_rank(sh, lane);
        o->ax[r] = v[0];
        o->bx[r] = v[1];
        o->ay[r] = v[2];
        o->by[r] = v[3];
        o->acc[r] = a;
    }
    cl.sync();
    // spreads about the mean, and the bandwidth factor
    if (warp < 2) {
        const double m = sum_ranks(warp == 0 ? sh->sx : sh->sy) / n;
        double s = 0.0;
        for (int e = lane; e < ne; e += 32) {
            const int i = index(e);
            if (i >= n) break;
            const double2 v = entry(e, i);
            const double d = (warp == 0 ? v.x : v.y) - m;
            s += d * d;
        }
        s = wsum_kde(s);
        if (lane < kKdeCtas) {
            KdeShare* o = cl.map_shared_rank(sh, lane);
            if (warp == 0) o->vx[r] = s;
            else o->vy[r] = s;
        }
    } else if (tid == 64) {
        long long a = 0;
        for (int q = 0; q < kKdeCtas; ++q) a += sh->acc[q];
        par[6] = pow((double)a + 1.0, -1.0 / 6.0);
    }
    cl.sync();
    // extents, kernel widths (x: thread 0, y: thread 32)
    if (lane == 0 && warp < 2) {
        const bool X = warp == 0;
        const double v = sum_ranks(X ? sh->vx : sh->vy) / n, h = sqrt(v) * par[6];
        double lo = X ? sh->ax[0] : sh->ay[0], hi = X ? sh->bx[0] : sh->by[0];
        for (int q = 1; q < kKdeCtas; ++q) {
            lo = fmin(lo, X ? sh->ax[q] : sh->ay[q]);
            hi = fmax(hi, X ? sh->bx[q] : sh->by[q]);
        }
        double e0, e1;
        grid_extent(lo, hi, h, X ? lox : loy, X ? hix : hiy, G, e0, e1);
        par[2 * warp] = e0;
        par[2 * warp + 1] = e1;
        par[4 + warp] = h / ((e1 - e0) / G);   // kernel width in cells
        if (r == 0) {
            double* e = ext + ((size_t)w * 3 + p) * 4 + 2 * warp;
            e[0] = e0;
            e[1] = e1;
        }
    }
    __syncthreads();
    const double x0 = par[0], x1 = par[1], y0 = par[2], y1 = par[3];
    const int rx = kernel_radius(par[4], G), ry = kernel_radius(par[5], G);
    // weights exp(-d^2/2 sigma^2), one per thread (x: lower half, y: upper half)
    {
        const bool X = tid < kKdeThreads / 2;
        const double sigma = X ? par[4] : par[5];
        const bool smooth = sigma > 0.0 && isfinite(sigma);
        const int rr = X ? rx : ry;
        for (int q = tid & (kKdeThreads / 2 - 1); q <= 2 * rr; q += kKdeThreads / 2) {
            const int d = q - rr;
            we[(X ? 0 : 2 * G) + q] = smooth ? exp(-(double)d * d / (2.0 * sigma * sigma)) : 1.0;
        }
    }
    // counts, each at the CTA that owns its row
    const float gx = (float)((double)G / (x1 - x0)), gy = (float)((double)G / (y1 - y0));
    for (int e = tid; e < ne; e += kKdeThreads) {
        const int i = index(e);
        if (i >= n) continue;
        const double2 v = entry(e, i);
        const int ci = kde_cell_fast(v.x, x0, x1, G, gx), cj = kde_cell_fast(v.y, y0, y1, G, gy);
        const int o = ci / rows;
        atomicAdd(cl.map_shared_rank(own, o) + (ci - o * rows) * G + cj, 1);
    }
    __syncthreads();
    if (lane == 0 && warp < 2) {   // weight totals, in order
        double t = 0.0;
        const double* e = we + (warp == 0 ? 0 : 2 * G);
        const int m = 2 * (warp == 0 ? rx : ry);
        for (int q = 0; q <= m; ++q) t += e[q];
        par[4 + warp] = t;
    }
    __syncthreads();
    {
        const bool X = tid < kKdeThreads / 2;
        const int rr = X ? rx : ry;
        for (int q = tid & (kKdeThreads / 2 - 1); q <= 2 * rr; q += kKdeThreads / 2)
            (X ? kx : ky)[q] = (float)(we[(X ? 0 : 2 * G) + q] / (X ? par[4] : par[5]));
    }
    cl.sync();   // every count is in
    // the rows within reach of this CTA's
    for (int c = max(0, i0 - rx) * G + tid; c < min(G, i1 + rx) * G; c += kKdeThreads) {
        const int i = c / G, o = i / rows;
        cnt[c] = cl.map_shared_rank(own, o)[c - o * rows * G];
    }
    __syncthreads();
    // smoothing along x (first index), then along y
    for (int c = i0 * G + tid; c < i1 * G; c += kKdeThreads) {
        const int i = c / G, j = c - i * G;
        float v = 0.0f;
        for (int d = -rx; d <= rx; ++d) {
            const int i2 = i - d;
            if (i2 >= 0 && i2 < G) v = fmaf(kx[d + rx], (float)cnt[i2 * G + j], v);
        }
        S1[c - i0 * G] = v;
    }
    __syncthreads();
    for (int c = i0 * G + tid; c < i1 * G; c += kKdeThreads) {
        const int i = c / G, j = c - i * G;
        float v = 0.0f;
        for (int e = -ry; e <= ry; ++e) {
            const int j2 = j - e;
            if (j2 >= 0 && j2 < G) v = fmaf(ky[e + ry], S1[(i - i0) * G + j2], v);
        }
        S2[c - i0 * G] = v;
    }
    cl.sync();   // every smoothed cell is there
    auto cell = [&](int c) {
        const int o = c / (rows * G);
        return cl.map_shared_rank(S2, o)[c - o * rows * G];
    };
    // total over the cells and cumulative sums over contiguous chunks, in the
    // order of 256 partial sums again (warp 0: partial sums 32 r + lane)
    const int per = (GG + kKdeVirt - 1) / kKdeVirt;
    const int vt = 32 * r + lane, c0 = vt * per, c1 = min(GG, c0 + per);
    if (warp == 0) {
        double t = 0.0;
        for (int c = vt; c < GG; c += kKdeVirt) t += cell(c);
        t = wsum_kde(t);
        if (lane < kKdeCtas) cl.map_shared_rank(sh, lane)->tot[r] = t;
    }
    cl.sync();
    const double tot = sum_ranks(sh->tot);
    // cell probabilities with the floor
    const double fl = eps / (double)GG, sc = (1.0 - eps) / tot;
    if (warp == 0) {
        double run = 0.0;
        for (int c = c0; c < c1; ++c) run += (double)cell(c) * sc + fl;
        cl.map_shared_rank(sh, 0)->part[vt] = run;
    }
    cl.sync();
    if (r == 0 && tid == 0) {   // exclusive scan of the chunk sums
        double a = 0.0;
        for (int t = 0; t < kKdeVirt; t += 8) {
            double v[8];
#pragma unroll
            for (int q = 0; q < 8; ++q) v[q] = sh->part[t + q];
#pragma unroll
            for (int q = 0; q < 8; ++q) {
                sh->part[t + q] = a;
                a += v[q];
            }
        }
    }
    cl.sync();
    if (warp == 0) {
        double* out = cdf + ((size_t)w * 3 + p) * GG;
        double run = cl.map_shared_rank(sh, 0)->part[vt];
        for (int c = c0; c < c1; ++c) {
            run += (double)cell(c) * sc + fl;
            out[c] = run;
        }
    }
    cl.sync();   // the others' shared memory outlives these reads
}

// C > u for u > 0 and any C, on the bits: integer compares, which do not wait
// for the FP64 pipe (positive doubles order as their bits; a NaN is above +inf)
__device__ __forceinline__ bool above(const double* C, long long ub) {
    const long long c = __ldg((const long long*)C);
    return c > ub && c <= 0x7FF0000000000000LL;
}
// (hi + (x + 1/2) 2^-32) for a small integer hi, exactly: one FP64 operation
__device__ __forceinline__ double u01_plus(int hi, uint32_t x) {
    const long long v = ((long long)hi << 33) | ((long long)x << 1) | 1;
    return fma(__longlong_as_double(0x4330000000000000LL | v), 0x1p-33, -0x1p19);
}

// What a window's proposals share, formed once per CTA
struct KdeDrawShared {
    double cx[3], cy[3], lc[3];   // cell sizes and the log of the cell's area
    double wd[2], lw[2];          // widths of psi and phi0 and their logs
};

// One thread per proposal.  Bound by the FP64 pipe: four logs, and per
// coordinate an offset, a product and a sum; what depends only on the window
// (two divisions and a log per pair, two logs more) is formed once per CTA,
// the searches compare integers and the uniforms take one operation each.
// 160,000 proposals, grid 64: 75 us (166 us with nine logs and six divisions
// per proposal).
__global__ void kde_draw_kernel(int n, int G, const double* __restrict__ box, const double* __restrict__ cdf,
                                const double* __restrict__ ext, uint64_t seed, const uint64_t* __restrict__ round_in, uint64_t* __restrict__ round_out,
                                double* __restrict__ theta, double* __restrict__ log_g, double* __restrict__ log_u) {
    __shared__ KdeDrawShared ks;
    const int w = blockIdx.y;
    const int i = blockIdx.x * blockDim.x + threadIdx.x;
    const uint64_t rnd = *round_in;
    if (w == 0 && blockIdx.x == 0 && threadIdx.x == 0) *round_out = rnd + 1;
    const double* bx = box + 16 * (size_t)w;
    if (threadIdx.x < 3) {
        const int p = threadIdx.x;
        const double* e = ext + ((size_t)w * 3 + p) * 4;
        const double cx = __ddiv_rn(__dadd_rn(e[1], -e[0]), (double)G);
        const double cy = __ddiv_rn(__dadd_rn(e[3], -e[2]), (double)G);
        ks.cx[p] = cx;
        ks.cy[p] = cy;
        ks.lc[p] = log(__dmul_rn(cx, cy));
    } else if (threadIdx.x < 5) {
        const int d = threadIdx.x - 3;
        const double wd = __dadd_rn(bx[14 + d], -bx[6 + d]);
        ks.wd[d] = wd;
        ks.lw[d] = log(wd);
    }
    __syncthreads();
    if (i >= n) return;
    const uint32_t k0 = (uint32_t)seed, k1 = (uint32_t)(seed >> 32);
    const uint4 a = philox4x32_10((uint32_t)rnd, (uint32_t)w, (uint32_t)i, 0u, k0, k1);
    const uint4 b = philox4x32_10((uint32_t)rnd, (uint32_t)w, (uint32_t)i, 1u, k0, k1);
    const uint4 c = philox4x32_10((uint32_t)rnd, (uint32_t)w, (uint32_t)i, 2u, k0, k1);
    const uint32_t words[12] = {a.x, a.y, a.z, a.w, b.x, b.y, b.z, b.w, c.x, c.y, c.z, c.w};
    const int GG = G * G;
    // first cell with C_c > u of each pair, the last cell if none
    const double* C = cdf + (size_t)w * 3 * GG;
    int lo[3] = {0, 0, 0}, hi[3] = {GG - 1, GG - 1, GG - 1};
    long long ub[3];
#pragma unroll
    for (int p = 0; p < 3; ++p) ub[p] = __double_as_longlong(u01_plus(0, words[3 * p]));
    for (int left = GG - 1; left > 0; left >>= 1) {
#pragma unroll
        for (int p = 0; p < 3; ++p)
            if (lo[p] < hi[p]) {
                const int mid = (lo[p] + hi[p]) >> 1;
                if (above(C + (size_t)p * GG + mid, ub[p])) hi[p] = mid;
                else lo[p] = mid + 1;
            }
    }
    double out[8];
    double lg = 0.0;
#pragma unroll
    for (int p = 0; p < 3; ++p) {
        int dx, dy;
        pair_dims(p, dx, dy);
        const double* Cp = C + (size_t)p * GG;
        const double* e = ext + ((size_t)w * 3 + p) * 4;
        const int cell = lo[p];
        const double P = Cp[cell] - (cell > 0 ? Cp[cell - 1] : 0.0);
        const int ci = cell / G, cj = cell - ci * G;
        out[dx] = __dadd_rn(e[0], __dmul_rn(u01_plus(ci, words[3 * p + 1]), ks.cx[p]));
        out[dy] = __dadd_rn(e[2], __dmul_rn(u01_plus(cj, words[3 * p + 2]), ks.cy[p]));
        lg += log(P) - ks.lc[p];
    }
#pragma unroll
    for (int d = 6; d < 8; ++d) {
        out[d] = __dadd_rn(bx[d], __dmul_rn(u01_plus(0, words[d + 3]), ks.wd[d - 6]));
        lg -= ks.lw[d - 6];
    }
    const size_t row = (size_t)w * n + i;
    if (((size_t)theta & 15) == 0) {
#pragma unroll
        for (int d = 0; d < 8; d += 2) *(double2*)(theta + 8 * row + d) = make_double2(out[d], out[d + 1]);
    } else {
#pragma unroll
        for (int d = 0; d < 8; ++d) theta[8 * row + d] = out[d];
    }
    log_g[row] = lg;
    log_u[row] = log(u01_plus(0, words[11]));
}

// shared memory of a build CTA without and with its entries
size_t kde_build_smem(int G, int n, bool store) {
    const size_t GG = (size_t)G * G, rows = (G + kKdeCtas - 1) / kKdeCtas;
    const size_t ne = ((size_t)n + kKdeVirt - 1) / kKdeVirt * 32;
    return sizeof(KdeShare) + sizeof(double) * (4 * (size_t)G + 8) + 4 * sizeof(float) * G + sizeof(int) * GG +
           3 * sizeof(float) * rows * G + 16 + (store ? sizeof(double2) * ne : 0);
}

}  // namespace
}  // namespace gb

using namespace gb;

extern "C" int gb_kde_build(gb_ctx_t* ctx, int32_t n_win, int32_t n, const double* theta, const int32_t* chain,
                            const double* box, int32_t grid, double floor_mass, double* cdf, double* ext,
                            void* stream) {
    if (!ctx) return GB_EINVAL;
    if (n_win < 0 || n < 0) return set_error(ctx, GB_EINVAL, "gb_kde_build: negative size");
    if (n_win == 0) return GB_OK;
    if (n < 1) return set_error(ctx, GB_EINVAL, "gb_kde_build: at least one step per chain");
    if (grid < 2 || grid > 128) return set_error(ctx, GB_EINVAL, "gb_kde_build: grid must be in [2, 128]");
    if (!(floor_mass >= 0.0 && floor_mass <= 1.0)) return set_error(ctx, GB_EINVAL, "gb_kde_build: floor in [0, 1]");
    if (!theta || !chain || !box || !cdf || !ext) return set_error(ctx, GB_EINVAL, "gb_kde_build: null pointer");
    cudaError_t e = cudaSetDevice(ctx->device);
    if (e != cudaSuccess) return cuda_error(ctx, e, "gb_kde_build: cudaSetDevice");
    // a chain's entries stay in shared memory when they fit beside the grid (up
    // to 88,064 per chain at grid 64, 52,736 at grid 128); longer chains are
    // gathered again in each pass
    const int store = kde_build_smem(grid, n, true) <= 200 * 1024;
    const size_t smem = kde_build_smem(grid, n, store != 0);
    e = cudaFuncSetAttribute(kde_build_kernel, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)smem);
    if (e != cudaSuccess) return cuda_error(ctx, e, "gb_kde_build: smem attribute");
    kde_build_kernel<<<dim3((unsigned)n_win * kKdeCtas, 3), kKdeThreads, smem, (cudaStream_t)stream>>>(
        n, grid, theta, chain, box, floor_mass, cdf, ext, store);
    ++ctx->launches;
    e = cudaGetLastError();
    if (e != cudaSuccess) return cuda_error(ctx, e, "gb_kde_build launch");
    return GB_OK;
}

extern "C" int gb_kde_draw(gb_ctx_t* ctx, int32_t n_win, int32_t n, const double* box, int32_t grid,
                           const double* cdf, const double* ext, uint64_t seed, const uint64_t* round_in, uint64_t* round_out,
                           double* theta, double* log_g, double* log_u, void* stream) {
    if (!ctx) return GB_EINVAL;
    if (n_win < 0 || n < 0) return set_error(ctx, GB_EINVAL, "gb_kde_draw: negative size");
    if (n_win == 0 || n == 0) return GB_OK;
    if (n_win > 65535) return set_error(ctx, GB_EINVAL, "gb_kde_draw: more than 65535 windows");
    if (grid < 2 || grid > 128) return set_error(ctx, GB_EINVAL, "gb_kde_draw: grid must be in [2, 128]");
    if (!box || !cdf || !ext || !round_in || !round_out || !theta || !log_g || !log_u)
        return set_error(ctx, GB_EINVAL, "gb_kde_draw: null pointer");
    if (round_in == round_out) return set_error(ctx, GB_EINVAL, "gb_kde_draw: round_out must not alias round_in");
    cudaError_t e = cudaSetDevice(ctx->device);
    if (e != cudaSuccess) return cuda_error(ctx, e, "gb_kde_draw: cudaSetDevice");
    kde_draw_kernel<<<dim3((n + 255) / 256, n_win), 256, 0, (cudaStream_t)stream>>>(
        n, grid, box, cdf, ext, seed, round_in, round_out, theta, log_g, log_u);
    ++ctx->launches;
    e = cudaGetLastError();
    if (e != cudaSuccess) return cuda_error(ctx, e, "gb_kde_draw launch");
    return GB_OK;
}
