// Gabor time-frequency analysis of the dipole bins and emission times of a
// burst (Sec. III.A, the time-frequency maps of the dipole velocity and the
// burst centres as functions of the harmonic energy).
//
//   G(t_j, w_m) = sum_k x(t_k) exp(-(t_k - t_j)^2 / (2 sigma^2)) e^{i w_m t_k} dt_out
//
// summed over the bins with |t_k - t_j| <= 9 sigma (the window is below
// e^{-40} beyond).
//
// Bound by FP64 instructions (64 cycles of a sub-partition each on GB300), so the kernel
// is built to need few per (time, frequency, bin).  About the window's bin c nearest to t_j
// the windowed bins y of a pair c + m, c - m enter as
//   e^{i w t_c} [ (y_{c+m} + y_{c-m}) cos(w m dt) + i (y_{c+m} - y_{c-m}) sin(w m dt) ]:
// 2 FMAs a pair, and cos and sin depend on the frequency and m only, so a warp (one lane
// per frequency) that holds 8 times forms them once for all 8: (16 + 4) / 16 = 1.25
// FMAs per time and bin instead of 6.  The Gaussian of a pair is
//   e^{-delta^2/2s^2} e^{-(m dt)^2/2s^2} (e^{-delta dt/s^2})^{+-m},  delta = t_c - t_j:
// one exponential per m for all times, and powers of one number per time (near 1 where
// t_j lies among the bins).  The index arithmetic is in gabor_window.h: c stays within the
// bins, so m and the work do too, and a time that is not a number takes no part in the sums
// and has a row of NaN.  Block = 8 times x 64 frequencies x 4 parts of half of the m range;
// the parts meet in shared memory, the halves (a cluster of two blocks) in the first
// block's.  Twice as many blocks even out what the SMs get: 1300 blocks on 152 SMs are 9 at
// most for a mean of 8.6, 650 were 5 for 4.3 (1937 us).
// Measured, 6620 bins, 400 times x 800 frequencies, windows of 2107 bins: 8387 us with a
// rotation per time, frequency and bin, 1816 us now (8.4e8 FMAs: 1.4 ms).
//
// Short windows and few bins (direct_is_faster): one thread per frequency and time with a
// rotation per bin, as the eight times' tables and the cluster's barriers take 21 to 28 us
// however short the window.
//
// Emission time: a block of 16 warps per 32 frequencies scans |G(t_j, w)|^2 over the
// analysis times in [t_a, t_b] for the centroid and the peak (vertex of the parabola
// through ln|G|^2 at the maximum and its two neighbours); 122 -> 28 us at
// the same size (one thread per frequency before, which is still the faster form for few
// times or very many frequencies: launch_emission_time).
#include <cooperative_groups.h>

#include <algorithm>

#include "gabor_window.h"
#include "sfhk_device.cuh"

namespace sfhk {
namespace {

constexpr int kTimes = 8;           // analysis times per block
constexpr int kParts = 4;           // parts of the m range (warps per 32 frequencies)
constexpr int kGroups = 2;          // groups of 32 frequencies per block
constexpr int kGThreads = 32 * kParts * kGroups;
constexpr int kSpan = 64;           // m values between exact anchors of the rotation
constexpr int kGTile = kParts * kSpan;

constexpr int kHalves = 2;          // blocks of a cluster, along the m range
static_assert(kGThreads == 2 * kTimes * 16 && kGThreads == kGTile, "one table entry and one m per thread");

struct GaborShared {
    double2 ab[kGTile][kTimes];               // (y_{c+m} + y_{c-m}, y_{c+m} - y_{c-m}) of the tile
    double2 part[kGroups][kParts - 1][32];    // sums of parts 1..3, one time at a time
    double run[2][kTimes][kGTile / 16];       // e^{-+ 16 a delta dt/s^2} of the tile's runs of 16 m
    double in_run[2][kTimes][16];             // dt e^{-delta^2/2s^2} e^{-+ b delta dt/s^2}
    double delta[kTimes];                     // t_c - t_j
    long long c[kTimes], lo[kTimes], hi[kTimes];
    long long reach, m_lo, m_hi;
};

constexpr int kDirectTile = 1024;

// block = one analysis time x 128 frequencies
__global__ void gabor_direct_kernel(const double* __restrict__ x, int64_t n_bins, double t0, double dt, double sigma,
                                    const double* __restrict__ times, int64_t n_t, const double* __restrict__ omega,
                                    int64_t n_omega, double* out_re, double* out_im) {
    __shared__ double sx[kDirectTile];
    const int64_t m = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
    const double w = m < n_omega ? omega[m] : 0.0;
    double rs, rc;
    sincos(w * dt, &rs, &rc);
    const double inv2s2 = 1.0 / (2.0 * sigma * sigma);
    for (int64_t j = blockIdx.y; j < n_t; j += gridDim.y) {
        const double tj = times[j];
        const GaborBins v = gabor_bins(tj, t0, dt, sigma, n_bins);
        double sr = 0.0, si = 0.0;
        for (int64_t k0 = v.lo; k0 <= v.hi; k0 += kDirectTile) {
            const int nt = (int)(v.hi - k0 + 1 < kDirectTile ? v.hi - k0 + 1 : kDirectTile);
            __syncthreads();
            for (int u = threadIdx.x; u < nt; u += blockDim.x) {
                const double d = (t0 + (double)(k0 + u) * dt) - tj;
                sx[u] = x[k0 + u] * exp(-d * d * inv2s2) * dt;
            }
            __syncthreads();
            direct_sum(sx, nt, w, t0, dt, k0, rc, rs, sr, si);
        }
        if (m < n_omega) {
            out_re[j * n_omega + m] = v.nan ? tj : sr;
            out_im[j * n_omega + m] = v.nan ? tj : si;
        }
    }
}

// The faster kernel for a call, by what their times in microseconds were found to be on 152
// SMs (windows of W bins, reach R of the pairs): the larger of one block's latency and of the
// chip's throughput.  Measured against this estimate's choice, direct and blocked: 10 times x
// 20 frequencies, W 91: 28 and 36, W 217: 58 and 46; 400 x 800, W 19: 136 and 181, W 55: 275
// and 205; 100 bins under a window of 1054, 100 x 100: 31 and 44, 400 x 800: 474 and 267.
bool direct_is_faster(int64_t n_bins, double half_width, int64_t n_t, int64_t n_omega) {
    if (n_bins < 1) return true;
    const double R = std::min((double)(n_bins - 1), half_width), W = std::min((double)n_bins, 2.0 * half_width + 1.0);
    const double direct_pairs = (double)n_t * (double)((n_omega + 127) / 128 * 128);
    const double blocked_pairs = (double)((n_t + 7) / 8 * 8) * (double)((n_omega + 63) / 64 * 64);
    const double direct = std::max(8.5 + 0.216 * W, direct_pairs * (1.9e-4 + 1.08e-5 * W));
    const double blocked = std::max((n_t < 8 ? 20.5 : 27.5) + 0.18 * R, blocked_pairs * (4.7e-4 + 4.9e-6 * R));
    return direct <= blocked;
}

__global__ void __cluster_dims__(1, 1, kHalves) __launch_bounds__(kGThreads)
    gabor_kernel(const double* __restrict__ x, int64_t n_bins, double t0, double dt, double sigma,
                 const double* __restrict__ times, int64_t n_t, const double* __restrict__ omega, int64_t n_omega,
                 double* out_re, double* out_im) {
    __shared__ GaborShared sm;
    const cooperative_groups::cluster_group cluster = cooperative_groups::this_cluster();
    const int half = (int)cluster.block_rank();
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5, part = warp % kParts, group = warp / kParts;
    const int64_t m_w = ((int64_t)blockIdx.x * kGroups + group) * 32 + lane;   // this lane's frequency
    const double w = m_w < n_omega ? omega[m_w] : 0.0;
    const double inv2s2 = 1.0 / (2.0 * sigma * sigma);
    for (int64_t jt = (int64_t)blockIdx.y * kTimes; jt < n_t; jt += (int64_t)gridDim.y * kTimes) {
        __syncthreads();
        if (threadIdx.x < kTimes) {
            const int u = threadIdx.x;
            // no bins for a time past the end of the list
            GaborWindow v{1, 0, 0, 0.0};
            if (jt + u < n_t) v = gabor_window(times[jt + u], t0, dt, sigma, n_bins);
            sm.c[u] = v.c;
            sm.lo[u] = v.lo;
            sm.hi[u] = v.hi;
            sm.delta[u] = v.delta;
        }
        __syncthreads();
        if (threadIdx.x == 0) {
            // this block's half of the m range of all eight windows
            long long reach = -1;
            for (int u = 0; u < kTimes; ++u) {
                const long long r = gabor_reach(sm.lo[u], sm.hi[u], sm.c[u]);
                reach = r > reach ? r : reach;
            }
            const long long mid = gabor_middle(reach);
            sm.reach = reach;
            sm.m_lo = half ? mid : 0;
            sm.m_hi = half ? reach : mid - 1;
        }
        __syncthreads();
        if (sm.reach < 0) {   // no bins for any of the times (in both blocks of the cluster)
            if (half == 0 && m_w < n_omega)
                for (int u = part; u < kTimes && jt + u < n_t; u += kParts)   // (0, or NaN)
                    out_re[(jt + u) * n_omega + m_w] = out_im[(jt + u) * n_omega + m_w] = sm.delta[u];
            continue;
        }
        const int64_t m_lo = sm.m_lo, m_hi = sm.m_hi;
        double rs, rc;
        sincos(w * dt, &rs, &rc);   // rotation per bin
        // this thread's entry of the two tables: side, time, place in the run or run
        const int e_side = threadIdx.x >> 7, e_u = (threadIdx.x >> 4) & (kTimes - 1), e_b = threadIdx.x & 15;
        const double e_d = sm.delta[e_u], theta = (e_side ? 2.0 : -2.0) * dt * e_d * inv2s2;
        sm.in_run[e_side][e_u][e_b] = exp(fma((double)e_b, theta, -e_d * e_d * inv2s2)) * dt;
        double gr[kTimes], gi[kTimes];
#pragma unroll
        for (int u = 0; u < kTimes; ++u) gr[u] = gi[u] = 0.0;
        for (int64_t mt = m_lo; mt <= m_hi; mt += kGTile) {
            const int nm = (int)(m_hi - mt + 1 < kGTile ? m_hi - mt + 1 : kGTile);
            __syncthreads();   // the last tile is read, the time's table written
            sm.run[e_side][e_u][e_b] = exp((double)(mt + 16 * e_b) * theta);
            __syncthreads();
            // the pairs of the tile: thread i takes every time of m = mt + i
            if ((int)threadIdx.x < nm) {
                const int i = threadIdx.x;
                const int64_t m = mt + i;
                const double md = (double)m * dt, g0 = exp(-md * md * inv2s2);
#pragma unroll
                for (int u = 0; u < kTimes; ++u) {
                    const int64_t kp = sm.c[u] + m, kq = sm.c[u] - m, lo = sm.lo[u], hi = sm.hi[u];
                    double yp = 0.0, yq = 0.0;
                    if (kp >= lo && kp <= hi) yp = x[kp] * (g0 * (sm.run[0][u][i >> 4] * sm.in_run[0][u][i & 15]));
                    if (m > 0 && kq >= lo && kq <= hi)
                        yq = x[kq] * (g0 * (sm.run[1][u][i >> 4] * sm.in_run[1][u][i & 15]));
                    sm.ab[i][u] = make_double2(yp + yq, yp - yq);
                }
            }
            __syncthreads();
            const int a = nm * part / kParts, b = nm * (part + 1) / kParts;
            if (a < b) {
                double es, ec;
                sincos(w * ((double)(mt + a) * dt), &es, &ec);
                for (int i = a; i < b; ++i) {
#pragma unroll
                    for (int u = 0; u < kTimes; ++u) {
                        const double2 v = sm.ab[i][u];
                        gr[u] = fma(v.x, ec, gr[u]);
                        gi[u] = fma(v.y, es, gi[u]);
                    }
                    const double nc = fma(ec, rc, -es * rs);
                    es = fma(ec, rs, es * rc);
                    ec = nc;
                }
            }
        }
        // the parts of the m range, in order; the second block's sums go to the first one,
        // into the place of its pairs
        double2* const other = cluster.map_shared_rank(&sm.ab[0][0], 0);
        double2 sum[kTimes];
#pragma unroll
        for (int u = 0; u < kTimes; ++u) {
            __syncthreads();
            if (part > 0) sm.part[group][part - 1][lane] = make_double2(gr[u], gi[u]);
            __syncthreads();
            if (part == 0) {
                sum[u] = make_double2(gr[u], gi[u]);
                for (int q = 0; q < kParts - 1; ++q) {
                    sum[u].x += sm.part[group][q][lane].x;
                    sum[u].y += sm.part[group][q][lane].y;
                }
            }
        }
        cluster.sync();   // the first block has read its last tile
        if (half == 1 && part == 0)
#pragma unroll
            for (int u = 0; u < kTimes; ++u) other[(u * kGroups + group) * 32 + lane] = sum[u];
        cluster.sync();
        if (half == 0 && part == 0 && m_w < n_omega) {
#pragma unroll
            for (int u = 0; u < kTimes; ++u) {
                if (jt + u >= n_t) continue;
                const double2 o = other[(u * kGroups + group) * 32 + lane];
                double vr = sum[u].x + o.x, vi = sum[u].y + o.y;
                if (sm.lo[u] <= sm.hi[u]) {   // times e^{i w t_c}
                    double s, c;
                    sincos(w * (t0 + (double)sm.c[u] * dt), &s, &c);
                    const double zr = fma(vr, c, -vi * s);
                    vi = fma(vr, s, vi * c);
                    vr = zr;
                } else if (isnan(sm.delta[u])) {
                    vr = vi = sm.delta[u];
                }
                out_re[(jt + u) * n_omega + m_w] = vr;
                out_im[(jt + u) * n_omega + m_w] = vi;
            }
        }
    }
    cluster.sync();   // no block leaves while the other may write to it
}

constexpr int kEWarps = 16;
constexpr int kEDirect = 128;   // threads of a block with one thread per frequency

// kWarps warps per 32 frequencies (kEWarps: a block; 1: every warp by itself)
template <int kWarps>
__global__ void __launch_bounds__(kWarps == 1 ? kEDirect : 32 * kWarps)
    emission_kernel(const double* __restrict__ g_re, const double* __restrict__ g_im, int64_t n_t, int64_t n_omega,
                    const double* __restrict__ times, double t_a, double t_b, double* centroid, double* peak) {
    const int lane = threadIdx.x & 31, warp = kWarps == 1 ? 0 : threadIdx.x >> 5;
    const int64_t m = kWarps == 1 ? (int64_t)blockIdx.x * kEDirect + threadIdx.x : (int64_t)blockIdx.x * 32 + lane;
    const bool have = m < n_omega;
    auto P = [&](int64_t j) {
        const double r = g_re[j * n_omega + m], i = g_im[j * n_omega + m];
        return r * r + i * i;
    };
    // warp q takes the times q, q + kWarps, ...
    double s0 = 0.0, s1 = 0.0, pmax = -1.0;
    int64_t jmax = -1, j_first = LLONG_MAX, j_last = -1;
    for (int64_t j = warp; j < n_t; j += kWarps) {
        const double t = times[j];
        if (!(t >= t_a && t <= t_b)) continue;
        if (j < j_first) j_first = j;
        j_last = j;
        if (!have) continue;
        const double p = P(j);
        s0 += p;
        s1 = fma(t, p, s1);
        if (p > pmax) {
            pmax = p;
            jmax = j;
        }
    }
    if constexpr (kWarps > 1) {
        __shared__ double s_s0[kWarps][32], s_s1[kWarps][32], s_p[kWarps][32];
        __shared__ long long s_j[kWarps][32], s_first[kWarps], s_last[kWarps];
        s_s0[warp][lane] = s0;
        s_s1[warp][lane] = s1;
        s_p[warp][lane] = pmax;
        s_j[warp][lane] = jmax;
        if (lane == 0) {
            s_first[warp] = j_first;
            s_last[warp] = j_last;
        }
        __syncthreads();
        if (warp != 0) return;
        for (int q = 1; q < kWarps; ++q) {
            s0 += s_s0[q][lane];
            s1 += s_s1[q][lane];
            const double p = s_p[q][lane];
            const int64_t j = s_j[q][lane];
            // the first of equal maxima
            if (j >= 0 && (p > pmax || (p == pmax && j < jmax))) {
                pmax = p;
                jmax = j;
            }
            if (s_first[q] < j_first) j_first = s_first[q];
            if (s_last[q] > j_last) j_last = s_last[q];
        }
    }
    if (!have) return;
    double cen = nan(""), pk = nan("");
    if (jmax >= 0 && s0 > 0.0) {
        cen = s1 / s0;
        pk = times[jmax];
        if (jmax > j_first && jmax < j_last) {
            const double pm = P(jmax - 1), pp = P(jmax + 1);
            if (pm > 0.0 && pp > 0.0) {
                const double ym = log(pm), y0 = log(pmax), yp = log(pp);
                const double h = times[jmax + 1] - times[jmax];
                const double curv = ym - 2.0 * y0 + yp;
                if (curv < 0.0 && fabs(times[jmax] - times[jmax - 1] - h) <= 1e-9 * fabs(h))
                    pk = times[jmax] + 0.5 * h * (ym - yp) / curv;
            }
        }
    }
    centroid[m] = cen;
    peak[m] = pk;
}

}  // namespace

cudaError_t launch_gabor(const double* bins, int64_t n_bins, double t0, double dt_out, double sigma,
                         const double* times, int64_t n_t, const double* omega, int64_t n_omega, double* out_re,
                         double* out_im, cudaStream_t s) {
    if (n_omega == 0 || n_t == 0) return cudaSuccess;
    if (direct_is_faster(n_bins, floor(kGaborCut * sigma / dt_out), n_t, n_omega)) {
        const int block = 128;
        const dim3 grid((unsigned)((n_omega + block - 1) / block), (unsigned)std::min<int64_t>(n_t, 65535));
        gabor_direct_kernel<<<grid, block, 0, s>>>(bins, n_bins, t0, dt_out, sigma, times, n_t, omega, n_omega, out_re,
                                                   out_im);
        return cudaGetLastError();
    }
    const unsigned gx = (unsigned)((n_omega + 32 * kGroups - 1) / (32 * kGroups));
    const unsigned gy = (unsigned)std::min<int64_t>((n_t + kTimes - 1) / kTimes, 65535);
    gabor_kernel<<<dim3(gx, gy, kHalves), kGThreads, 0, s>>>(bins, n_bins, t0, dt_out, sigma, times, n_t, omega, n_omega,
                                                    out_re, out_im);
    return cudaGetLastError();
}

cudaError_t launch_emission_time(const double* g_re, const double* g_im, int64_t n_t, int64_t n_omega,
                                 const double* times, double t_a, double t_b, double* centroid, double* peak,
                                 cudaStream_t s) {
    if (n_omega == 0) return cudaSuccess;
    // One thread per frequency where its few times, or its many frequencies, leave 16 warps
    // nothing to share (152 SMs; its time over that of 16 warps): 3 times 0.92, 10 times 1.2 up
    // to 5000 frequencies; 20000: 0.76 at 20 times, 0.99 at 50; 1e5: 0.90 at 100, 1.15 at 400.
    if (n_t < std::max<int64_t>(6, (n_omega - 3000) / 400))
        emission_kernel<1><<<(unsigned)((n_omega + kEDirect - 1) / kEDirect), kEDirect, 0, s>>>(
            g_re, g_im, n_t, n_omega, times, t_a, t_b, centroid, peak);
    else
        emission_kernel<kEWarps><<<(unsigned)((n_omega + 31) / 32), 32 * kEWarps, 0, s>>>(
            g_re, g_im, n_t, n_omega, times, t_a, t_b, centroid, peak);
    return cudaGetLastError();
}

}  // namespace sfhk
