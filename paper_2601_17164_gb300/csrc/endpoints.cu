// FP64 endpoints (sfhk_propagate): the full 43-component state, 32 trajectories per block
// of eight warps.
//
// A trajectory-step of the full state is about 700 FP64 instructions, each of which holds
// a sub-partition's FP64 unit for 64 cycles whatever it computes on (GB300).  With one
// thread per trajectory a call of some thousand births keeps a few warps on a part of
// the SMs busy; here a group of 32 is spread over the four sub-partitions of an SM:
//   dynamics  RK4 stages of (q, p, S) and the stage Hessian data,
//   columns   six warps, one stability column each, through the stages,
//   det       det Z, its branch, removal and the results,
// one grid point apart, with one barrier per grid point and double-buffered slots.
// Warps w and w + 4 share a sub-partition: (dynamics, column), (det, column) and two
// pairs of columns, 190, 180, 164 and 164 instructions.
// Measured, 4096 births over 11029 steps: 283 ms with one thread per trajectory (32 SMs at
// work), 84 ms now.
//
// The expressions are those of Traj<double>::step, so that the values are too.  A removed
// trajectory keeps the state of its removal bin: the det warp, which decides it, writes
// the state that belongs to its grid point.
#include <algorithm>

#include "sfhk_internal.cuh"
#include "traj_block.cuh"

namespace sfhk {
namespace {

constexpr int kW = 32;
constexpr int kThreads = 256;

struct EShared {
    double stage[2][20][kW];    // of the step n -> n + 1: positions (4 x 3), g (4), h (4)
    double state[4][7][kW];     // q, p, S at grid point n
    double col[2][6][6][kW];    // columns at grid point n: column, component (x, then y)
    long long last;             // the last iteration when the block ends early, else -1
};
constexpr int kStretch = 8;    // iterations between the points at which a block may end early

template <int POT>
__global__ void __launch_bounds__(kThreads, 2) endpoints_kernel(FieldDev f, TargetDev tg, TrajArgs a) {
    extern __shared__ __align__(16) unsigned char smem[];
    EShared& sm = *reinterpret_cast<EShared*>(smem);
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    const int64_t i = (int64_t)blockIdx.x * kW + lane;
    const bool have = i < a.n;
    const int64_t n0 = have ? (int64_t)a.n0[i] : 0;
    const int64_t n_last = a.n_last;
    const bool alive0 = have && n0 <= n_last && n0 >= 0;
    long long m = alive0 ? (long long)n0 : LLONG_MAX;   // first grid point of the block
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) {
        const long long u = __shfl_xor_sync(0xffffffffu, m, o);
        m = u < m ? u : m;
    }
    // a block without a trajectory in range writes its initial states at n_last
    const int64_t n_first = m == LLONG_MAX ? n_last : m;
    const int n_out = (int)f.n_out;
    const StepK<double> hk = f.k64;
    const double h = hk.h, hh = hk.hh, h6 = hk.h6;

    // The iterations run in stretches of 8.  The block ends early when every trajectory has
    // its results: at the start of a stretch, before the first barrier of it, the det warp
    // names its last iteration, after which all warps look (a reduction at every barrier
    // instead costs 0.7 %).
    const int64_t n_stop = n_last + 2;
    if (threadIdx.x == 0) sm.last = -1;
    volatile long long* const last = &sm.last;
    auto stretch = [&](int64_t n) { return n_stop - n + 1 < kStretch ? (int)(n_stop - n + 1) : kStretch; };

    if (warp == 0) {
        // dynamics
        PotConst<double> pc;
        pc.a2 = (POT == POT_SOFTCORE || POT == POT_HARMONIC) ? tg.pot_param[0] * tg.pot_param[0] : 0.0;
        pc.Zc = tg.pot_param[0]; pc.a1 = tg.pot_param[1]; pc.a2t = tg.pot_param[2];
        pc.a3 = tg.pot_param[3]; pc.a4 = tg.pot_param[4]; pc.a5 = tg.pot_param[5];
        pc.a6 = tg.pot_param[6];
        double q[3] = {(have && a.qx) ? a.qx[i] : 0.0, (have && a.qy) ? a.qy[i] : 0.0, have ? a.qz[i] : 0.0};
        double p[3] = {have ? a.px[i] : 0.0, have ? a.py[i] : 0.0, have ? a.pz[i] : 0.0};
        double S = 0.0;
        const double* E = f.E64;
        auto e_at = [&](int64_t j) { return j < f.table_len ? __ldg(E + j) : 0.0; };
        double Ea = e_at(2 * n_first), Eb = e_at(2 * n_first + 1), Ec = e_at(2 * n_first + 2);
        for (int64_t n = n_first; n <= n_stop;) {
            int left = stretch(n);
            for (; left > 0; --left, ++n) {
                if (n <= n_last) {
                    double(*const st)[kW] = sm.state[n & 3];
#pragma unroll
                    for (int c = 0; c < 3; ++c) {
                        st[c][lane] = q[c];
                        st[3 + c][lane] = p[c];
                    }
                    st[6][lane] = S;
                }
                if (n < n_last) {
                    const double Fa = e_at(2 * n + 2), Fb = e_at(2 * n + 3), Fc = e_at(2 * n + 4);
                    double qs[4][3], gs[4], hs[4];
                    double V, g, hc;
                    // the stages of Traj::step
                    potential<double, POT>(q[0], q[1], q[2], pc, V, g, hc);
                    double kp1[3] = {-g * q[0], -g * q[1], -fma(g, q[2], Ea)};
                    double kS1 = fma(0.5, fma(p[0], p[0], fma(p[1], p[1], p[2] * p[2])), -fma(q[2], Ea, V));
#pragma unroll
                    for (int c = 0; c < 3; ++c) qs[0][c] = q[c];
                    gs[0] = g; hs[0] = hc;
                    double p2[3];
#pragma unroll
                    for (int c = 0; c < 3; ++c) { qs[1][c] = fma(hh, p[c], q[c]); p2[c] = fma(hh, kp1[c], p[c]); }
                    potential<double, POT>(qs[1][0], qs[1][1], qs[1][2], pc, V, g, hc);
                    gs[1] = g; hs[1] = hc;
                    double kp2[3] = {-g * qs[1][0], -g * qs[1][1], -fma(g, qs[1][2], Eb)};
                    double kS2 = fma(0.5, fma(p2[0], p2[0], fma(p2[1], p2[1], p2[2] * p2[2])), -fma(qs[1][2], Eb, V));
                    double p3[3];
#pragma unroll
                    for (int c = 0; c < 3; ++c) { qs[2][c] = fma(hh, p2[c], q[c]); p3[c] = fma(hh, kp2[c], p[c]); }
                    potential<double, POT>(qs[2][0], qs[2][1], qs[2][2], pc, V, g, hc);
                    gs[2] = g; hs[2] = hc;
                    double kp3[3] = {-g * qs[2][0], -g * qs[2][1], -fma(g, qs[2][2], Eb)};
                    double kS3 = fma(0.5, fma(p3[0], p3[0], fma(p3[1], p3[1], p3[2] * p3[2])), -fma(qs[2][2], Eb, V));
                    double p4[3];
#pragma unroll
                    for (int c = 0; c < 3; ++c) { qs[3][c] = fma(h, p3[c], q[c]); p4[c] = fma(h, kp3[c], p[c]); }
                    potential<double, POT>(qs[3][0], qs[3][1], qs[3][2], pc, V, g, hc);
                    gs[3] = g; hs[3] = hc;
                    double kp4[3] = {-g * qs[3][0], -g * qs[3][1], -fma(g, qs[3][2], Ec)};
                    double kS4 = fma(0.5, fma(p4[0], p4[0], fma(p4[1], p4[1], p4[2] * p4[2])), -fma(qs[3][2], Ec, V));
                    double(*const sl)[kW] = sm.stage[n & 1];
#pragma unroll
                    for (int k = 0; k < 4; ++k) {
#pragma unroll
                        for (int c = 0; c < 3; ++c) sl[3 * k + c][lane] = qs[k][c];
                        sl[12 + k][lane] = gs[k];
                        sl[16 + k][lane] = hs[k];
                    }
                    if (alive0 && n >= n0) {
#pragma unroll
                        for (int c = 0; c < 3; ++c) {
                            const double sq = fma(2.0, p2[c] + p3[c], p[c]) + p4[c];
                            const double sp = fma(2.0, kp2[c] + kp3[c], kp1[c]) + kp4[c];
                            q[c] = fma(h6, sq, q[c]);
                            p[c] = fma(h6, sp, p[c]);
                        }
                        S += h6 * (fma(2.0, kS2 + kS3, kS1) + kS4);
                    }
                    Ea = Fa;
                    Eb = Fb;
                    Ec = Fc;
                }
                __syncthreads();
            }
            if (*last == n - 1) break;
        }
    } else if (warp != 1) {
        // columns: warps 2..7 hold the derivatives to q0 (x, y, z) and p0 (x, y, z), at grid
        // point n - 1 in iteration n
        const int c = warp - 2;
        double X[3], Y[3];
#pragma unroll
        for (int k = 0; k < 3; ++k) {
            X[k] = c == k ? 1.0 : 0.0;
            Y[k] = c == k + 3 ? 1.0 : 0.0;
        }
        for (int64_t n = n_first; n <= n_stop;) {
            int left = stretch(n);
            for (; left > 0; --left, ++n) {
                const int64_t u = n - 1;
                if (u >= n_first && u <= n_last) {
                    double(*const o)[kW] = sm.col[u & 1][c];
#pragma unroll
                    for (int k = 0; k < 3; ++k) {
                        o[k][lane] = X[k];
                        o[3 + k][lane] = Y[k];
                    }
                }
                if (u >= n_first && u < n_last) {
                    const double(*const sl)[kW] = sm.stage[u & 1];
                    double xs[3], ys[3], ky[3], ay[3], ax[3];
#pragma unroll
                    for (int s = 0; s < 4; ++s) {
                        const double q0 = sl[3 * s][lane], q1 = sl[3 * s + 1][lane], q2 = sl[3 * s + 2][lane];
                        const double qv[3] = {q0, q1, q2}, g = sl[12 + s][lane], hs = sl[16 + s][lane];
                        const double* const xv = s == 0 ? X : xs;
                        const double d = fma(q0, xv[0], fma(q1, xv[1], q2 * xv[2])) * hs;
#pragma unroll
                        for (int k = 0; k < 3; ++k) {
                            ky[k] = -fma(g, xv[k], d * qv[k]);
                            if (s == 0) {
                                ax[k] = Y[k];
                                ay[k] = ky[k];
                            } else if (s < 3) {
                                ax[k] = fma(2.0, ys[k], ax[k]);
                                ay[k] = fma(2.0, ky[k], ay[k]);
                            } else {
                                ax[k] += ys[k];
                                ay[k] += ky[k];
                            }
                        }
                        if (s < 3) {
                            const double w = s < 2 ? hh : h;
#pragma unroll
                            for (int k = 0; k < 3; ++k) {
                                xs[k] = fma(w, s == 0 ? Y[k] : ys[k], X[k]);
                                ys[k] = fma(w, ky[k], Y[k]);
                            }
                        }
                    }
                    if (alive0 && u >= n0) {
#pragma unroll
                        for (int k = 0; k < 3; ++k) {
                            X[k] = fma(h6, ax[k], X[k]);
                            Y[k] = fma(h6, ay[k], Y[k]);
                        }
                    }
                }
                __syncthreads();
            }
            if (*last == n - 1) break;
        }
    } else {
        // det: grid point n - 2 in iteration n
        const double rg = a.gamma;
        const double zh = 0.5, zg = -rg, zq = 1.0 / (4.0 * rg);
        bool alive = alive0;
        unsigned flags = (have && !alive) ? 8u : 0u;
        Cx2<double> Dp{1.0, 0.0};
        double sgn = 1.0;
        cd Cacc{1.0, 0.0};
        unsigned long long steps = 0;
        bool written = false;
        int rem = (int)(n_first % n_out);
        for (int64_t n = n_first; n <= n_stop;) {
            int left = stretch(n);
            if (__all_sync(0xffffffffu, written || !have) && lane == 0) *last = n + left - 1;
            for (; left > 0; --left, ++n) {
                const int64_t u = n - 2;
                if (u >= n_first) {
                    const double(*const st)[kW] = sm.state[u & 3];
                    const double(*const co)[6][kW] = sm.col[u & 1];
                    const bool live = alive && u >= n0;
                    if (u > n_first) {
                        // the step into u: det Z of its columns
                        Traj<double, POT> T;
#pragma unroll
                        for (int c = 0; c < 6; ++c)
#pragma unroll
                            for (int k = 0; k < 3; ++k) {
                                T.X[c][k] = co[c][k][lane];
                                T.Y[c][k] = co[c][3 + k][lane];
                            }
                        if (alive && u - 1 >= n0) {
                            const Cx2<double> D = T.detc(zh, zg, zq);
                            follow_branch<double>(Dp, D, sgn, flags);
                            ++steps;
                        }
                    }
                    bool write = false;
                    if ((rem == 0 || u == n_last) && live) {
                        const double fs = st[0][lane] + st[1][lane] + st[2][lane] + st[3][lane] + st[4][lane] + st[5][lane];
                        const bool ok = isfinite(fs) && isfinite(st[6][lane]);
                        const cd D{Dp.re, Dp.im};
                        const double m2 = D.re * D.re + D.im * D.im;
                        if (!ok || !(m2 <= a.d_t * a.d_t)) {
                            alive = false;
                            flags |= 1u;
                            if (!ok || !isfinite(m2)) flags |= 2u;
                            write = true;
                        } else {
                            cd C = c_sqrt(D);
                            if (sgn < 0.0) C = -C;
                            Cacc = C;
                        }
                    }
                    // a trajectory that never started has its results at the end of the others
                    if (u == n_last || !__any_sync(0xffffffffu, alive)) write = have && !written;
                    if (write) {
                        written = true;
                        const size_t nn = (size_t)a.n;
#pragma unroll
                        for (int c = 0; c < 6; ++c) a.st_out[(size_t)c * nn + i] = st[c][lane];
#pragma unroll
                        for (int r = 0; r < 3; ++r)
#pragma unroll
                            for (int c = 0; c < 3; ++c) {
                                a.st_out[(size_t)(6 + 3 * r + c) * nn + i] = co[c][r][lane];            // Mqq
                                a.st_out[(size_t)(15 + 3 * r + c) * nn + i] = co[3 + c][r][lane];       // Mqp
                                a.st_out[(size_t)(24 + 3 * r + c) * nn + i] = co[c][3 + r][lane];       // Mpq
                                a.st_out[(size_t)(33 + 3 * r + c) * nn + i] = co[3 + c][3 + r][lane];   // Mpp
                            }
                        a.st_out[(size_t)42 * nn + i] = st[6][lane];
                        a.c_re[i] = Cacc.re;
                        a.c_im[i] = Cacc.im;
                        a.flags[i] = (uint8_t)flags;
                    }
                    rem = rem + 1 == n_out ? 0 : rem + 1;
                }
                __syncthreads();
            }
            if (*last == n - 1) break;
        }
        if (a.stats) {
            unsigned rm = __reduce_add_sync(0xffffffffu, (flags & 1u) ? 1u : 0u);
            unsigned nf = __reduce_add_sync(0xffffffffu, (flags & 2u) ? 1u : 0u);
            unsigned bg = __reduce_add_sync(0xffffffffu, (flags & 4u) ? 1u : 0u);
            unsigned sk = __reduce_add_sync(0xffffffffu, (flags & 8u) ? 1u : 0u);
            unsigned long long sp = steps;
#pragma unroll
            for (int o = 16; o > 0; o >>= 1) sp += __shfl_xor_sync(0xffffffffu, sp, o);
            if (lane == 0) {
                if (rm) atomicAdd(&a.stats->removed, (unsigned long long)rm);
                if (nf) atomicAdd(&a.stats->nonfinite, (unsigned long long)nf);
                if (bg) atomicAdd(&a.stats->branch_guard, (unsigned long long)bg);
                if (sk) atomicAdd(&a.stats->skipped, (unsigned long long)sk);
                if (sp) atomicAdd(&a.stats->traj_steps, sp);
            }
        }
    }
}

template <int POT>
cudaError_t launch_pot(const FieldDev& f, const TargetDev& t, const TrajArgs& a, cudaStream_t s) {
    auto kern = endpoints_kernel<POT>;
    const int bytes = (int)sizeof(EShared);
    cudaError_t e = cudaFuncSetAttribute(kern, cudaFuncAttributeMaxDynamicSharedMemorySize, bytes);
    if (e != cudaSuccess) return e;
    kern<<<(unsigned)((a.n + kW - 1) / kW), kThreads, bytes, s>>>(f, t, a);
    return cudaGetLastError();
}

}  // namespace

// Longest call for this kernel.  Where the one-thread kernel's warps fill the chip it needs
// no hand-offs and no barriers, and its warps skip the steps after their last removal, of
// which Tong-Lin trajectories have many (27 % below).  Measured, one-thread over this
// kernel's time (800 nm 1 cycle, d_t 1e30, 152 SMs): soft-core 1.01 at 160,000, 0.99 at
// 180,000, 0.98 at 400,000; harmonic 1.00 at 156,000 and 200,000; Tong-Lin 1.05 at 60,000,
// 0.99 at 66,000, 0.85 at 100,000.
int64_t endpoints_limit(int pot, int sms) { return (int64_t)kW * sms * (pot == POT_TONGLIN ? 13 : 34); }

cudaError_t launch_endpoints(const FieldDev& f, const TargetDev& t, const TrajArgs& a, cudaStream_t s) {
    if (a.n == 0) return cudaSuccess;
    switch (t.pot) {
        case POT_SOFTCORE: return launch_pot<POT_SOFTCORE>(f, t, a, s);
        case POT_TONGLIN: return launch_pot<POT_TONGLIN>(f, t, a, s);
        case POT_HARMONIC: return launch_pot<POT_HARMONIC>(f, t, a, s);
        default: return launch_pot<POT_ZERO>(f, t, a, s);
    }
}

}  // namespace sfhk
