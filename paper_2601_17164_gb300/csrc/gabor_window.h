// Index arithmetic of the Gabor map (gabor.cu): the window of one analysis time and the
// range of pairs that a block sums.  Plain functions, compiled for the host too, where a
// test runs them over times that are not numbers, infinite or far from the bins and over
// windows wider than the bins: whatever a caller's array holds, every index stays within
// the bins and the work within their number.
#pragma once
#include <math.h>

#ifdef __CUDACC__
#define SFHK_HD __host__ __device__ __forceinline__
#else
#define SFHK_HD inline
#endif

namespace sfhk {

constexpr double kGaborCut = 9.0;   // window half-width in units of sigma

// Bins [lo, hi] of a time's window, none when lo > hi.  A time that is not a number has no
// bins, and a row of NaN (where there are bins at all).
struct GaborBins {
    long long lo, hi;
    bool nan;
};
SFHK_HD GaborBins gabor_bins(double tj, double t0, double dt, double sigma, long long n_bins) {
    GaborBins w{1, 0, false};
    if (n_bins < 1) return w;
    if (tj != tj) {
        w.nan = true;
        return w;
    }
    const double lo = fmax(ceil((tj - kGaborCut * sigma - t0) / dt), 0.0);
    const double hi = fmin(floor((tj + kGaborCut * sigma - t0) / dt), (double)(n_bins - 1));
    if (lo <= hi) {
        w.lo = (long long)lo;
        w.hi = (long long)hi;
    }
    return w;
}
// the same with the window's bin c nearest to the time and delta = t_c - t_j (NaN for a time
// that is not a number, 0 without bins)
struct GaborWindow {
    long long lo, hi, c;
    double delta;
};
SFHK_HD GaborWindow gabor_window(double tj, double t0, double dt, double sigma, long long n_bins) {
    const GaborBins b = gabor_bins(tj, t0, dt, sigma, n_bins);
    GaborWindow w{b.lo, b.hi, 0, b.nan ? tj : 0.0};
    if (b.lo > b.hi) return w;
    const double c = fmin(fmax(rint((tj - t0) / dt), (double)b.lo), (double)b.hi);
    w.c = (long long)c;
    w.delta = (t0 + c * dt) - tj;
    return w;
}
// the last m of which c + m or c - m is in the window, -1 when it is empty
SFHK_HD long long gabor_reach(long long lo, long long hi, long long c) {
    if (lo > hi) return -1;
    return hi - c > c - lo ? hi - c : c - lo;
}
// the first of two halves of [0, reach] ends before this m
SFHK_HD long long gabor_middle(long long reach) { return (reach + 1) / 2; }

}  // namespace sfhk
