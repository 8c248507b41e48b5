// Hanning-windowed Fourier transform of the dipole bins (App. D):
//   X(w_m) = sum_k x(t_k) W_H(t_k) e^{i w_m t_k} dt_out,
//   W_H(t) = (1 + cos(pi t / tau_H)) / 2 for |t| <= tau_H, else 0.
//
// Bound by FP64 instructions: a warp's FP64 instruction takes 64 cycles of its
// sub-partition on GB300, so the count per (frequency, bin) pair and the number of
// sub-partitions at work decide.  One lane per frequency; the bins are cut into runs
// of 16, and a run's sum over u of y_u e^{i w u dt} takes the 16 factors from
// registers (they are the same for every run): 2 FMAs a pair instead of the 6 of a
// rotation per bin.  Runs are joined by Horner's rule with e^{i 16 w dt}, 4 FMAs per
// run, and anchored with an exact sincos once per part.  A frequency's bins are
// spread over the warps of a block and the blocks of a cluster (kParts parts or more),
// whose sums meet in the first block's shared memory in a fixed order.  The window
// comes from two angle sums over three small tables of cosines (4 FP64 instructions a
// bin instead of a cosine).
// Measured, 8826 bins x 1200 frequencies: 2044 us with one thread per frequency in 10
// blocks, 111 us now (the pairs' FMAs alone take 45 us on all sub-partitions).  4 us of
// them carry the phases' roundings (anchor): relative error against 64 bits, the worst
// output, 8.6e-14; 2.7e-13 without, 1.4e-13 with one thread per frequency.  The clusters of
// four put two blocks on some SMs and none on others: an SM is at work for 58 % of the
// launch on average, its FP64 pipe then 80 % busy, and the fullest sub-partition holds 3300
// FP64 instructions for a mean of 1620 (ncu).
//
// Few bins (direct_bins): one thread per frequency with a rotation per bin.  The factors,
// anchors and cluster barriers above take 24 us however few the bins (10 bins x 20: 24 us
// against 9 us), and a warp's ~140 FP64 instructions for them in 16 warps per 32
// frequencies outweigh the pairs where frequencies are many (500 bins x 2e5: 1.9 ms
// against 1.25 ms).
#include <cooperative_groups.h>

#include <algorithm>

#include "sfhk_device.cuh"

namespace sfhk {
namespace {

constexpr int kRun = 16;         // bins per run
constexpr int kTileRuns = 160;   // runs of a block in shared memory at a time
constexpr int kMaxWarps = 8;

// e^{i w (t0 + k dt)} with the roundings of the phase carried: a part of some 500 bins has
// one anchor and one factor between its runs, so errors of their phases (1e-13 where |w t|
// is 1500) would not average out.
__device__ __forceinline__ void anchor(double w, double t0, double dt, int64_t k, double* s, double* c) {
    const double kd = __dmul_rn((double)k, dt), kl = fma((double)k, dt, -kd);
    const double t = __dadd_rn(t0, kd), b = __dadd_rn(t, -t0);
    const double tl = __dadd_rn(__dadd_rn(t0, -__dadd_rn(t, -b)), __dadd_rn(kd, -b)) + kl;   // t0 + k dt - t
    const double p = __dmul_rn(w, t), e = fma(w, tl, fma(w, t, -p));
    double sp, cp;
    sincos(p, &sp, &cp);
    *s = fma(cp, e, sp);
    *c = fma(-sp, e, cp);
}

constexpr int kDirectTile = 1024;

__global__ void spectrum_direct_kernel(const double* __restrict__ x, int64_t n_bins, double t0, double dt, double tau,
                                       const double* __restrict__ omega, int64_t n_omega, double* out_re,
                                       double* out_im) {
    __shared__ double sx[kDirectTile];
    const int64_t m = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
    const double w = m < n_omega ? omega[m] : 0.0;
    double sr = 0.0, si = 0.0, rs, rc;
    sincos(w * dt, &rs, &rc);
    for (int64_t k0 = 0; k0 < n_bins; k0 += kDirectTile) {
        const int nt = (int)(n_bins - k0 < kDirectTile ? n_bins - k0 : kDirectTile);
        __syncthreads();
        for (int u = threadIdx.x; u < nt; u += blockDim.x) {
            const double t = t0 + (double)(k0 + u) * dt;
            const double W = fabs(t) <= tau ? 0.5 * (1.0 + cospi(t / tau)) : 0.0;
            sx[u] = x[k0 + u] * W * dt;
        }
        __syncthreads();
        direct_sum(sx, nt, w, t0, dt, k0, rc, rs, sr, si);
    }
    if (m < n_omega) {
        out_re[m] = sr;
        out_im[m] = si;
    }
}

// Most bins for that kernel, where its time meets the other one's (152 SMs; its time over
// the other's): up to 1200 frequencies 0.87 at 64 bins, 1.25 at 100; 5000: 0.93 at 200, 1.14
// at 256; 20000: 0.97 at 400, 1.23 at 552; 1e5: 0.76 at 552, 1.14 at 1000.
int64_t direct_bins(int64_t n_omega) {
    return std::max<int64_t>(80, std::min<int64_t>(n_omega / 24, 400 + n_omega / 400));
}

__global__ void __launch_bounds__(32 * kMaxWarps)
    spectrum_kernel(const double* __restrict__ x, int64_t n_bins, double t0, double dt, double tau,
                    const double* __restrict__ omega, int64_t n_omega, double* out_re, double* out_im) {
    namespace cg = cooperative_groups;
    const cg::cluster_group cluster = cg::this_cluster();
    __shared__ double sy[kTileRuns * kRun];
    // cos and sin of pi/tau times: a bin's place in its run, a run's place in its row of 16
    // runs, the start of a row of the tile
    __shared__ double s_bin[2][kRun], s_run[2][16], s_row[2][kTileRuns / 16];
    __shared__ double sum[kMaxWarps][2][32];       // per warp, then (first block) per block of the cluster
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5, warps = blockDim.x >> 5;
    const int part = (int)cluster.block_rank(), parts = (int)cluster.num_blocks();
    const int64_t m = (int64_t)(blockIdx.x / parts) * 32 + lane;
    const double w = m < n_omega ? omega[m] : 0.0;
    const double h = 0.5 * dt;
    // |t| <= tau as a range of bins (the window is 0 at the ends)
    const int64_t k_in = (int64_t)fmin(fmax(ceil((-tau - t0) / dt), 0.0), (double)n_bins);
    const int64_t k_out = (int64_t)fmin(fmax(floor((tau - t0) / dt), -1.0), (double)n_bins);
    // e^{i w u dt}, u < 16, by products of two (at most 4 roundings deep), and e^{i 16 w dt}
    double er[kRun], ei[kRun], rr, ri;
    er[0] = 1.0;
    ei[0] = 0.0;
    anchor(w, 0.0, dt, 1, &ei[1], &er[1]);
#pragma unroll
    for (int u = 2; u < kRun; ++u) {
        const int p = u / 2, q = u - p;
        er[u] = fma(er[p], er[q], -ei[p] * ei[q]);
        ei[u] = fma(er[p], ei[q], ei[p] * er[q]);
    }
    anchor(w, 0.0, dt, kRun, &ri, &rr);   // (Horner's rule takes its error to the number of runs)
    // the angle sums lose nothing while a row of 16 runs is not long against the window
    const bool fine = 16.0 * kRun * dt <= 4.0 * tau;
    const int64_t runs = (n_bins + kRun - 1) / kRun;
    const int64_t j_lo = runs * part / parts, j_hi = runs * (part + 1) / parts;   // this block's runs
    double sr = 0.0, si = 0.0;
    for (int64_t j0 = j_lo; j0 < j_hi; j0 += kTileRuns) {
        const int nr = (int)(j_hi - j0 < kTileRuns ? j_hi - j0 : kTileRuns);
        __syncthreads();
        {
            const int v = threadIdx.x;
            double s0, c0, ang = 0.0;
            if (v < kRun) ang = (double)v * dt;
            else if (v < 32) ang = (double)((v - 16) * kRun) * dt;
            else if (v < 32 + kTileRuns / 16) ang = t0 + (double)((j0 + (v - 32) * 16) * kRun) * dt;
            if (v < 32 + kTileRuns / 16) {
                sincospi(ang / tau, &s0, &c0);
                double(*const dst)[16] = v < kRun ? s_bin : s_run;
                if (v < 32) {
                    dst[0][v & 15] = c0;
                    dst[1][v & 15] = s0;
                } else {
                    s_row[0][v - 32] = c0;
                    s_row[1][v - 32] = s0;
                }
            }
        }
        __syncthreads();
        // the windowed bins of the tile, a thread on one place of the run throughout
        {
            const int u = threadIdx.x & (kRun - 1);
            const double cu = s_bin[0][u], su = s_bin[1][u];
            for (int v = threadIdx.x / kRun; v < nr; v += blockDim.x / kRun) {
                const double cj = s_run[0][v & 15], sj = s_run[1][v & 15], cr = s_row[0][v >> 4], sr_ = s_row[1][v >> 4];
                const double cs = fma(cr, cj, -sr_ * sj), sn = fma(sr_, cj, cr * sj);
                const int64_t k = (j0 + v) * kRun + u;
                double W = 0.0;   // W_H dt
                if (k >= k_in && k <= k_out) {
                    if (fine) W = fma(h, fma(cs, cu, -sn * su), h);
                    else W = h * (1.0 + cospi((t0 + (double)k * dt) / tau));
                }
                sy[v * kRun + u] = k < n_bins ? x[k] * W : 0.0;
            }
        }
        __syncthreads();
        // this warp's runs [a, b) of the tile, last first
        const int a = nr * warp / warps, b = nr * (warp + 1) / warps;
        if (a < b) {
            double hr = 0.0, hi = 0.0;
            for (int j = b - 1; j >= a; --j) {
                const double2* y2 = reinterpret_cast<const double2*>(sy + j * kRun);
                double pr = 0.0, pi = 0.0;
#pragma unroll
                for (int u = 0; u < kRun; u += 2) {
                    const double2 y = y2[u / 2];
                    pr = fma(y.x, er[u], pr);
                    pi = fma(y.x, ei[u], pi);
                    pr = fma(y.y, er[u + 1], pr);
                    pi = fma(y.y, ei[u + 1], pi);
                }
                const double nr2 = fma(hr, rr, fma(-hi, ri, pr));
                hi = fma(hr, ri, fma(hi, rr, pi));
                hr = nr2;
            }
            double es, ec;
            anchor(w, t0, dt, (j0 + a) * kRun, &es, &ec);
            sr = fma(hr, ec, fma(-hi, es, sr));
            si = fma(hr, es, fma(hi, ec, si));
        }
    }
    // warps of the block, then blocks of the cluster, in order
    sum[warp][0][lane] = sr;
    sum[warp][1][lane] = si;
    __syncthreads();
    double tr = 0.0, ti = 0.0;
    if (warp == 0) {
        for (int q = 0; q < warps; ++q) {
            tr += sum[q][0][lane];
            ti += sum[q][1][lane];
        }
        __syncwarp();
    }
    cluster.sync();   // every block's warps have read their sums
    if (warp == 0) {
        double* const dst = cluster.map_shared_rank(&sum[part][0][0], 0);   // row `part` of the first block
        dst[lane] = tr;
        dst[32 + lane] = ti;
    }
    cluster.sync();
    if (part == 0 && warp == 0 && m < n_omega) {
        double vr = 0.0, vi = 0.0;
        for (int q = 0; q < parts; ++q) {
            vr += sum[q][0][lane];
            vi += sum[q][1][lane];
        }
        out_re[m] = vr;
        out_im[m] = vi;
    }
}

}  // namespace

cudaError_t launch_spectrum(const double* bins, int64_t n_bins, double t0, double dt_out, double tau_h,
                            const double* omega, int64_t n_omega, double* out_re, double* out_im,
                            cudaStream_t s) {
    if (n_omega == 0) return cudaSuccess;
    if (n_bins <= direct_bins(n_omega)) {
        const int block = 128;
        spectrum_direct_kernel<<<(unsigned)((n_omega + block - 1) / block), block, 0, s>>>(
            bins, n_bins, t0, dt_out, tau_h, omega, n_omega, out_re, out_im);
        return cudaGetLastError();
    }
    // Blocks per group of 32 frequencies: as many as bring the grid to one block on each of
    // 152 SMs, at least 4 (16 warps: the parts' anchors still cost a tenth of the sums) and
    // at most 8 (the portable cluster size), those with 8 warps where even that leaves half
    // the SMs idle.
    const int64_t groups = (n_omega + 31) / 32;
    const int parts = (int)std::max<int64_t>(4, std::min<int64_t>(8, 152 / groups));
    const int warps = groups * parts <= 76 ? 8 : 4;
    cudaLaunchConfig_t cfg = {};
    cfg.gridDim = dim3((unsigned)(groups * parts));
    cfg.blockDim = dim3(32 * warps);
    cfg.stream = s;
    cudaLaunchAttribute attr[1];
    attr[0].id = cudaLaunchAttributeClusterDimension;
    attr[0].val.clusterDim.x = parts;
    attr[0].val.clusterDim.y = 1;
    attr[0].val.clusterDim.z = 1;
    cfg.attrs = attr;
    cfg.numAttrs = 1;
    return cudaLaunchKernelEx(&cfg, spectrum_kernel, bins, n_bins, t0, dt_out, tau_h, omega, n_omega, out_re, out_im);
}

}  // namespace sfhk
