// Importance sampling of births in proportion to |I0| (App. A, Eq. Int: the
// weight |I0| of a momentum that solves the saddle-point equation turns the
// Monte Carlo integral into importance sampling), as systematic resampling of
// a proposal pool of m births down to n.
//
//   w_i = |a_i| (a_i = the pool amplitude, |I0| times the proposal weight),
//   q_i = floor(w_i 2^B / max w) with B = 62 - ceil(log2 m), Q = sum q_i < 2^62,
//   one uniform U in [0, 2^32) (Philox4x64-10, key (seed, 1), counter 0, the
//   high half of word 0), thresholds t_j = floor((j 2^32 + U) Q / (n 2^32)),
//   m_i = #{j : C_{i-1} <= t_j < C_i} with C_i = q_0 + ... + q_i,
//   output: the births with m_i > 0 in pool order, amplitude a_i m_i Q / (n q_i).
//
// Every integer step is exact (64-bit sums, 128-bit threshold counts) and the
// few floating-point steps are single correctly rounded operations, so the
// result does not depend on the launch configuration.  The count of
// thresholds below c has the closed form
//   J(c) = clamp(ceil((ceil(c n 2^32 / Q) - U) / 2^32), 0, n),
// so m_i = J(C_i) - J(C_{i-1}) needs only the inclusive prefix sum of q.
//
// Launches: the largest |a|^2 (its root is the largest weight: a correctly rounded root is
// monotone); quantisation with per-block sums; a one-block scan of the block sums;
// multiplicities with per-block counts of the drawn births; a one-block scan of the
// counts; the gather in pool order with the amplitude rescaling, and the padding.
//
// Bound by FP64 instructions (64 cycles of a sub-partition each on GB300) where the
// weights are formed and by HBM elsewhere, so the root is taken once per birth and only
// where it can reach q_i >= 1 (births far from a field crest cannot: whole warps skip),
// floors are shifts of the significand, and the thresholds are counted by 128-bit
// multiplications with a fixed-point reciprocal of Q, each prefix once.  Measured, 4e6 ->
// 1e6 births: 477 us with a root per birth in a pass of its own, an FP64 floor, two
// 128-bit divisions per birth and a 128-thread scan; 245 us now.
#include "sfhk_device.cuh"
#include "sfhk_internal.cuh"

namespace sfhk {
namespace {

constexpr int kRB = 1024;   // pool entries per block of the scan kernels (= threads)

// |a|^2 with separate products and sum (no fused multiply-add)
__device__ __forceinline__ double abs2(double re, double im) {
    return __dadd_rn(__dmul_rn(re, re), __dmul_rn(im, im));
}

// the largest |a|^2 as its bit pattern: non-negative doubles order as integers; a NaN
// (either sign) is above them all
__global__ void max_kernel(const double* __restrict__ re, const double* __restrict__ im, int64_t m,
                           unsigned long long* amax_bits) {
    unsigned long long mb = 0;
    for (int64_t i = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; i < m; i += (int64_t)gridDim.x * blockDim.x) {
        const unsigned long long b = (unsigned long long)__double_as_longlong(abs2(re[i], im[i]));
        if (b > mb) mb = b;
    }
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) {
        const unsigned long long t = __shfl_xor_sync(0xffffffffu, mb, o);
        if (t > mb) mb = t;
    }
    if ((threadIdx.x & 31) == 0 && mb) atomicMax(amax_bits, mb);
}

// 2^B / A (one correctly rounded division); 0 when A is zero, infinite or NaN
__device__ __forceinline__ double quant_scale(unsigned long long amax_bits, int B) {   // of the largest |a|^2
    const double A = __dsqrt_rn(__longlong_as_double((long long)amax_bits));
    if (!(A > 0.0) || !isfinite(A)) return 0.0;
    return __ddiv_rn(ldexp(1.0, B), A);
}

__device__ __forceinline__ unsigned long long block_sum_u64(unsigned long long v, unsigned long long* sh) {
    const int lane = threadIdx.x & 31, wp = threadIdx.x >> 5;
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) v += __shfl_xor_sync(0xffffffffu, v, o);
    if (lane == 0) sh[wp] = v;
    __syncthreads();
    unsigned long long t = 0;
    if (threadIdx.x == 0)
        for (int k = 0; k < (int)(blockDim.x >> 5); ++k) t += sh[k];
    return t;
}

// floor of a non-negative double below 2^63, by its significand
__device__ __forceinline__ unsigned long long floor_u64(double x) {
    const unsigned long long b = (unsigned long long)__double_as_longlong(x);
    const int e = (int)(b >> 52) - 1023;
    if (e < 0) return 0;
    const unsigned long long f = (b & 0xfffffffffffffull) | 0x10000000000000ull;
    return e <= 52 ? f >> (52 - e) : f << (e - 52);
}

__global__ void quant_kernel(const double* __restrict__ re, const double* __restrict__ im, int64_t m,
                             const unsigned long long* amax_bits, int B, unsigned long long* __restrict__ q,
                             unsigned long long* __restrict__ blk) {
    __shared__ unsigned long long sh[32];
    __shared__ double s_scale;
    __shared__ unsigned long long s_least;
    if (threadIdx.x == 0) {
        const double s = quant_scale(*amax_bits, B);
        s_scale = s;
        // |a|^2 below this gives |a| s < 1 - 1e-3, whatever the roundings
        // (not used near underflow, where r^2 is not good to 1e-3)
        const double r = s > 0.0 ? 0.999 / s : 0.0;
        s_least = r * r > 1e-290 ? (unsigned long long)__double_as_longlong(r * r) : 0ull;
    }
    __syncthreads();
    const double s = s_scale;
    const int64_t i = (int64_t)blockIdx.x * kRB + threadIdx.x;
    unsigned long long v = 0;
    if (i < m) {
        const double a2 = abs2(re[i], im[i]);
        if (s > 0.0 && (unsigned long long)__double_as_longlong(a2) >= s_least)
            v = floor_u64(__dmul_rn(__dsqrt_rn(a2), s));
        q[i] = v;
    }
    const unsigned long long t = block_sum_u64(v, sh);
    if (threadIdx.x == 0) blk[blockIdx.x] = t;
}

// inclusive scan of 1024 values per block (warp scans, then the warp totals)
__device__ __forceinline__ unsigned long long block_incl_scan_u64(unsigned long long v, unsigned long long* wt) {
    const int lane = threadIdx.x & 31, wp = threadIdx.x >> 5;
    unsigned long long x = v;
#pragma unroll
    for (int o = 1; o < 32; o <<= 1) {
        const unsigned long long y = __shfl_up_sync(0xffffffffu, x, o);
        if (lane >= o) x += y;
    }
    if (lane == 31) wt[wp] = x;
    __syncthreads();
    if (wp == 0) {
        unsigned long long t = wt[lane];
#pragma unroll
        for (int o = 1; o < 32; o <<= 1) {
            const unsigned long long y = __shfl_up_sync(0xffffffffu, t, o);
            if (lane >= o) t += y;
        }
        wt[lane] = t;
    }
    __syncthreads();
    return x + (wp > 0 ? wt[wp - 1] : 0ull);
}

// exclusive scan of blk[0..nb) in place; the total Q into blk[nb]
__global__ void scan_u64_kernel(unsigned long long* blk, int64_t nb) {
    __shared__ unsigned long long wt[32];
    __shared__ unsigned long long carry;
    if (threadIdx.x == 0) carry = 0;
    __syncthreads();
    for (int64_t base = 0; base < nb; base += kRB) {
        const int64_t k = base + threadIdx.x;
        const unsigned long long v = k < nb ? blk[k] : 0ull;
        const unsigned long long incl = block_incl_scan_u64(v, wt);
        const unsigned long long c = carry;
        if (k < nb) blk[k] = c + incl - v;
        __syncthreads();
        if (threadIdx.x == kRB - 1) carry = c + incl;
        __syncthreads();
    }
    if (threadIdx.x == 0) blk[nb] = carry;
}

// J(c) = #{j < n : t_j < c}: the smallest j with (j 2^32 + U) Q >= c n 2^32, at most n (the
// products are below 2^125).  R = floor(n 2^64 / Q), saturated, gives a start at or below
// it: c n / Q - U / 2^32 > floor(c R / 2^64) - 1, so J is at least that floor, and the two
// floors and U / 2^32 leave it at most 2 below.
__device__ __forceinline__ int64_t thresholds_below(unsigned long long c, unsigned long long Q, int64_t n,
                                                    unsigned long long U, unsigned long long R) {
    if (c == 0) return 0;
    unsigned long long j = __umul64hi(c, R);
    if (j >= (unsigned long long)n) j = (unsigned long long)n;
    const unsigned __int128 x = ((unsigned __int128)c * (unsigned long long)n) << 32;
    unsigned __int128 t = (unsigned __int128)((j << 32) + U) * Q;
    while (t < x && j < (unsigned long long)n) {
        t += (unsigned __int128)Q << 32;
        ++j;
    }
    return (int64_t)j;
}

__device__ __forceinline__ unsigned long long resample_uniform(uint64_t seed) {
    uint64_t c[4] = {0, 0, 0, 0};
    philox4x64_10(c, seed, 1);
    return (unsigned long long)(c[0] >> 32);
}

// m_i into mult[i], and the block's number of drawn births (m_i >= 1)
__global__ void mult_kernel(const unsigned long long* __restrict__ q, int64_t m, const unsigned long long* blk,
                            int64_t nb, int64_t n, uint64_t seed, int32_t* __restrict__ mult,
                            unsigned long long* __restrict__ cnt) {
    __shared__ unsigned long long wt[32];
    __shared__ unsigned long long sU, sR;
    __shared__ int64_t s_j[kRB / 32];
    const unsigned long long Q = blk[nb];
    if (threadIdx.x == 0) {
        sU = resample_uniform(seed);
        // floor(n 2^64 / Q), saturated at 2^64 - 1
        sR = Q == 0 ? 0ull
                    : ((unsigned long long)n < Q
                           ? (unsigned long long)((((unsigned __int128)(unsigned long long)n) << 64) / Q)
                           : ~0ull);
    }
    const int64_t i = (int64_t)blockIdx.x * kRB + threadIdx.x;
    const unsigned long long v = i < m ? q[i] : 0ull;
    const unsigned long long incl = block_incl_scan_u64(v, wt);   // (its barriers publish sU and sR)
    const unsigned long long first = blk[blockIdx.x], c = first + incl;
    // J of this prefix; the previous one's is the left neighbour's
    const int lane = threadIdx.x & 31, wp = threadIdx.x >> 5;
    const int64_t J = Q > 0 ? thresholds_below(c, Q, n, sU, sR) : 0;
    if (lane == 31) s_j[wp] = J;
    __syncthreads();
    int64_t Jp = __shfl_up_sync(0xffffffffu, J, 1);
    if (lane == 0) Jp = wp > 0 ? s_j[wp - 1] : (Q > 0 ? thresholds_below(first, Q, n, sU, sR) : 0);
    const int32_t k = (i < m && v > 0) ? (int32_t)(J - Jp) : 0;
    const int drawn = __syncthreads_count(k > 0);
    if (i < m) mult[i] = k;
    if (threadIdx.x == 0) cnt[blockIdx.x] = (unsigned long long)drawn;
}

// Block b gathers the drawn births of its pool entries to cnt[b] (exclusive sum), ...
__global__ void gather_kernel(BirthArgs pool, int64_t m, int64_t n, const int32_t* __restrict__ mult,
                              const unsigned long long* __restrict__ cnt, const unsigned long long* __restrict__ q,
                              const unsigned long long* Qp, BirthArgs out) {
    __shared__ int s_w[kRB / 32];
    const int lane = threadIdx.x & 31, wp = threadIdx.x >> 5;
    const int64_t i = (int64_t)blockIdx.x * kRB + threadIdx.x;
    const int32_t k = i < m ? mult[i] : 0;
    const unsigned mask = __ballot_sync(0xffffffffu, k > 0);
    if (lane == 0) s_w[wp] = __popc(mask);
    __syncthreads();
    if (k <= 0) return;
    int before = __popc(mask & ((1u << lane) - 1u));
    for (int w = 0; w < wp; ++w) before += s_w[w];
    const int64_t j = (int64_t)cnt[blockIdx.x] + before;
    const double f = __ddiv_rn(__dmul_rn((double)k, __ull2double_rn(*Qp)), __dmul_rn((double)n, __ull2double_rn(q[i])));
    out.n0[j] = pool.n0[i];
    out.t0[j] = pool.t0[i];
    out.px[j] = pool.px[i];
    out.py[j] = pool.py[i];
    out.pz[j] = pool.pz[i];
    out.qz[j] = pool.qz[i];
    out.amp_re[j] = __dmul_rn(pool.amp_re[i], f);
    out.amp_im[j] = __dmul_rn(pool.amp_im[i], f);
}

// ... and the rest of the output repeats the last drawn birth (the pool's first when none
// was drawn) with amplitude 0.
__global__ void pad_kernel(BirthArgs pool, int64_t n, const unsigned long long* Rp, BirthArgs out,
                           int64_t* n_distinct) {
    const int64_t r = (int64_t)*Rp;
    const int64_t t = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
    if (t == 0 && n_distinct) *n_distinct = r;
    const BirthArgs& src = r > 0 ? out : pool;
    const int64_t i = r > 0 ? r - 1 : 0;
    for (int64_t j = r + t; j < n; j += (int64_t)gridDim.x * blockDim.x) {
        out.n0[j] = src.n0[i];
        out.t0[j] = src.t0[i];
        out.px[j] = src.px[i];
        out.py[j] = src.py[i];
        out.pz[j] = src.pz[i];
        out.qz[j] = src.qz[i];
        out.amp_re[j] = 0.0;
        out.amp_im[j] = 0.0;
    }
}

size_t al256(size_t x) { return (x + 255) / 256 * 256; }

}  // namespace

int resample_scale_bits(int64_t m) {
    int k = 0;   // ceil(log2 max(2, m)), at least 1
    while (((int64_t)1 << k) < (m < 2 ? 2 : m)) ++k;
    return 62 - (k < 1 ? 1 : k);
}

size_t resample_scratch_bytes(int64_t m) {
    const int64_t nb = (m + kRB - 1) / kRB;
    return al256((size_t)m * 8) + al256((size_t)m * 4) + 2 * al256((size_t)(nb + 1) * 8) + 256;
}

cudaError_t launch_resample(const BirthArgs& pool, int64_t m, int64_t n, uint64_t seed, const BirthArgs& out,
                            unsigned char* scratch, int64_t* n_distinct, cudaStream_t s) {
    const int64_t nb = (m + kRB - 1) / kRB;
    unsigned char* p = scratch;
    unsigned long long* q = reinterpret_cast<unsigned long long*>(p);
    p += al256((size_t)m * 8);
    unsigned long long* blk = reinterpret_cast<unsigned long long*>(p);
    p += al256((size_t)(nb + 1) * 8);
    unsigned long long* cnt = reinterpret_cast<unsigned long long*>(p);
    p += al256((size_t)(nb + 1) * 8);
    int32_t* mult = reinterpret_cast<int32_t*>(p);
    p += al256((size_t)m * 4);
    unsigned long long* amax = reinterpret_cast<unsigned long long*>(p);

    cudaError_t e = cudaMemsetAsync(amax, 0, sizeof(unsigned long long), s);
    if (e != cudaSuccess) return e;
    const int64_t want = (m + 255) / 256;
    max_kernel<<<(unsigned)(want < 1216 ? want : 1216), 256, 0, s>>>(pool.amp_re, pool.amp_im, m, amax);
    quant_kernel<<<(unsigned)nb, kRB, 0, s>>>(pool.amp_re, pool.amp_im, m, amax, resample_scale_bits(m), q, blk);
    scan_u64_kernel<<<1, kRB, 0, s>>>(blk, nb);
    mult_kernel<<<(unsigned)nb, kRB, 0, s>>>(q, m, blk, nb, n, seed, mult, cnt);
    scan_u64_kernel<<<1, kRB, 0, s>>>(cnt, nb);
    gather_kernel<<<(unsigned)nb, kRB, 0, s>>>(pool, m, n, mult, cnt, q, blk + nb, out);
    const int64_t pad = (n + 255) / 256;
    pad_kernel<<<(unsigned)(pad < 1216 ? pad : 1216), 256, 0, s>>>(pool, n, cnt + nb, out, n_distinct);
    return cudaGetLastError();
}

}  // namespace sfhk
