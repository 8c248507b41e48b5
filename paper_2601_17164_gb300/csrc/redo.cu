// FP64 redo of the escalated births of a mixed-precision pass, planar form,
// with the work of one trajectory-step split across four warps.
//
// Same arithmetic as the FP64 planar trajectory block (traj_block.cuh: App. A
// propagation, Eq. C_HK prefactor with per-step branch tracking, Sec. III.A
// removal, App. C recombination terms), reorganised for latency: an escalation
// list is short (a few per cent of the births) and its longest members run
// the whole pulse, so the redo is bound by the chain of dependent FP64
// operations of one trajectory, not by the number of trajectories (one warp's
// FP64 instruction occupies its sub-partition's FP64 unit for 64 cycles).  A
// block of 128 threads holds 32 trajectories (one per lane) and gives each of
// its four warps about a quarter of the FP64 work of every step:
//   dynamics  RK4 stages of (q, p) and the stage Hessian data,
//   matrix    the in-plane step matrix [[A, B], [C, D]],
//   columns   the in-plane stability columns advanced by the step matrix, and the
//             action increment,
//   bins      the out-of-plane block, det Z and the branch of sqrt det Z, the
//             partial-wave labels, removal and the prefactor at the bins, and
//             the GTO recombination sums, spread over the steps between bins,
//             with the warp reduction and the atomic bin update.
// The warps form a pipeline, each handing data on to the next through two slots in
// shared memory on named barriers of the two warps (redo_warps.cuh), so that a warp can
// run up to two grid points ahead of the next one.
// The roles rotate with the block index so that the heavier roles of the
// blocks resident on one SM spread over its four sub-partitions.  Removal is
// decided by the bins warp; the warps ahead of it learn of it a few grid
// points late and only skip work that no longer counts.
//
// Lists long enough to fill the chip at 32 trajectories a block come here (quad_limit);
// then the FP64 instructions of all roles decide, 19 cycles of the SM each: 301 per step of
// a group, bins left out (soft-core; Tong-Lin 604; ncu), 15 fewer since the branch compares
// the bits of doubles and follows 8 det Z of 2 Z (no halves).  Measured, mixed H 8 cycles,
// 1e6 births (12,200 redone): 496 -> 472 ms; FP64 H 1600 nm 3 cycles, 20011 births: 471 to
// 483 ms with one thread per trajectory, 237 to 287 ms here by the sample (271 instead of
// 242 ms with every GTO term of every bin).
//
// Each part runs the same device functions as the one-thread-per-trajectory
// kernel (TrajP::stages_qp / action_term / action_sum, TrajP::step_matrix,
// TrajP::apply_step_matrix, TrajP::detc, follow_branch, gto_terms,
// contribution_final), so trajectories, branches, labels and removals are the
// same; only the order of the final bin sums (one warp per block instead of
// four) differs.
#include <algorithm>

#include "redo_warps.cuh"
#include "sfhk_internal.cuh"

namespace sfhk {
namespace {

constexpr int kW = 32;            // trajectories per block
constexpr int kThreads = 128;     // four warps
// dynamics -> matrix: stage positions (8), g (4), h (4), stage momenta 2..4 (6), stage
// potentials (4), three unused words, state (q0, q2, p0, p2)
constexpr int kS01 = 33;
// matrix -> columns: 15 matrix entries, g (4), state (q0, q2, p0, p2), then the action
// increment's inputs: stage z of stages 2..4 (3), stage momenta of stages 2..4 (6),
// stage potentials (4); the columns warp reads E itself (static shared memory stays
// within 48 KB per block)
constexpr int kS12 = 36;
constexpr int kS23 = 25;          // columns -> bins: in-plane columns after the step (16), g of the stages (4), state

// barrier bases of the three hand-offs
constexpr int kHand0 = 1, kHand1 = 5, kHand2 = 9;

struct Shared {
    double s01[2][kS01][kW];
    double s12[2][kS12][kW];
    double s23[2][kS23][kW];
    int alive[kW];   // written by the bins warp, read late and without order by the warps ahead
    long long last;  // the group's last grid point when it ends early, else -1 (GroupEnd)
};

struct Common {
    int64_t n_first, n_last;   // first and last grid point of the block
    int n_out;
    bool have;
    int64_t i, n0, k_cnt;
    bool alive0;
};

// dynamics: the state at grid point n and the stages of the step n -> n + 1
template <int POT>
__device__ void run_dynamics(const FieldDev& f, const TargetDev& tg, const TrajArgs& a, const Common& c, Shared& sm,
                             int lane) {
    PotConst<double> pc;
    if (POT == POT_SOFTCORE || POT == POT_HARMONIC) pc.a2 = tg.pot_param[0] * tg.pot_param[0];
    pc.Zc = tg.pot_param[0]; pc.a1 = tg.pot_param[1]; pc.a2t = tg.pot_param[2];
    pc.a3 = tg.pot_param[3]; pc.a4 = tg.pot_param[4]; pc.a5 = tg.pot_param[5];
    pc.a6 = tg.pot_param[6];
    TrajP<double, POT> T;
    T.init(0.0, 0.0, c.have ? a.qz[c.i] : 0.0, c.have ? a.px[c.i] : 0.0, c.have ? a.py[c.i] : 0.0,
           c.have ? a.pz[c.i] : 0.0);
    const StepK<double> hk = f.k64;
    const double* E = f.E64;
    auto e_at = [&](int64_t j) { return j < f.table_len ? __ldg(E + j) : 0.0; };
    double e0 = e_at(2 * c.n_first), e1 = e_at(2 * c.n_first + 1), e2 = e_at(2 * c.n_first + 2);
    const volatile int* alive = sm.alive;
    Producer<2> out(kHand0);
    for (int64_t n = c.n_first; n <= c.n_last;) {
        int left = GroupEnd::stretch(n, c.n_last);
        GroupEnd::decide(sm.last, n + left - 1, alive[lane]);
        for (; left > 0; --left, ++n) {
            {
                const int d = out.acquire();
                double* o = &sm.s01[d][0][lane];
                o[29 * kW] = T.q[0];
                o[30 * kW] = T.q[2];
                o[31 * kW] = T.p[0];
                o[32 * kW] = T.p[2];
                // the E values of the next step, loaded one step ahead
                const double f0 = e_at(2 * n + 2), f1 = e_at(2 * n + 3), f2 = e_at(2 * n + 4);
                const bool step = c.have && n >= c.n0 && n < c.n_last && alive[lane];
                if (step) {
                    double qs[4][2], gs[4], hs[4], ps[4][2], Vs[4];
                    T.stages_qp(e0, e1, e2, hk, pc, qs, gs, hs, ps, Vs);
#pragma unroll
                    for (int k = 0; k < 4; ++k) {
                        o[(2 * k) * kW] = qs[k][0];
                        o[(2 * k + 1) * kW] = qs[k][1];
                        o[(8 + k) * kW] = gs[k];
                        o[(12 + k) * kW] = hs[k];
                        o[(22 + k) * kW] = Vs[k];
                    }
#pragma unroll
                    for (int k = 1; k < 4; ++k) {
                        o[(14 + 2 * k) * kW] = ps[k][0];
                        o[(15 + 2 * k) * kW] = ps[k][1];
                    }
                }
                out.publish(d);
                e0 = f0;
                e1 = f1;
                e2 = f2;
            }
        }
        if (GroupEnd::here(sm.last, n - 1)) break;
    }
    out.drain();
}

// matrix: the step matrix of grid point n (one iteration behind the dynamics); the
// action increment's inputs go on to the columns warp
template <int POT>
__device__ void run_matrix(const FieldDev& f, const Common& c, Shared& sm, int lane) {
    const StepK<double> hk = f.k64;
    Consumer<2> in_q(kHand0);
    Producer<2> out(kHand1);
    for (int64_t n = c.n_first; n <= c.n_last;) {
        int left = GroupEnd::stretch(n, c.n_last);
        for (; left > 0; --left, ++n) {
            {
                const int di = in_q.wait();
                const int dq = out.acquire();
                const double* in = &sm.s01[di][0][lane];
                double* o = &sm.s12[dq][0][lane];
#pragma unroll
                for (int k = 0; k < 4; ++k) o[(19 + k) * kW] = in[(29 + k) * kW];
                if (c.have && n >= c.n0 && n < c.n_last) {
                    double qs[4][2], gs[4], hs[4];
#pragma unroll
                    for (int k = 0; k < 4; ++k) {
                        qs[k][0] = in[(2 * k) * kW];
                        qs[k][1] = in[(2 * k + 1) * kW];
                        gs[k] = in[(8 + k) * kW];
                        hs[k] = in[(12 + k) * kW];
                    }
                    const StepMat<double> M = TrajP<double, POT>::step_matrix(qs, gs, hs, hk);
#pragma unroll
                    for (int k = 0; k < 15; ++k) o[k * kW] = M.m[k];   // (its out-of-plane part is left out)
#pragma unroll
                    for (int k = 0; k < 4; ++k) o[(15 + k) * kW] = gs[k];
                    // the action increment's inputs
#pragma unroll
                    for (int k = 1; k < 4; ++k) {
                        o[(22 + k) * kW] = qs[k][1];
                        o[(24 + 2 * k) * kW] = in[(14 + 2 * k) * kW];
                        o[(25 + 2 * k) * kW] = in[(15 + 2 * k) * kW];
                    }
#pragma unroll
                    for (int k = 0; k < 4; ++k) o[(32 + k) * kW] = in[(22 + k) * kW];
                }
                in_q.release(di);
                out.publish(dq);
            }
        }
        if (GroupEnd::here(sm.last, n - 1)) break;
    }
    out.drain();
}

// columns: the stability columns advanced by the step matrix of grid point n, and
// the action S (its increment from the stage data the matrix warp hands on)
template <int POT>
__device__ void run_columns(const FieldDev& f, const Common& c, Shared& sm, int lane) {
    TrajP<double, POT> T;
    T.init(0.0, 0.0, 0.0, 0.0, 0.0, 0.0);   // columns: identity (the state is read from the slots)
    const double h6 = f.k64.h6;
    Action<double> S;
    S.init();
    const volatile int* alive = sm.alive;
    Consumer<2> in_q(kHand1);
    Producer<2> out(kHand2);
    for (int64_t n = c.n_first; n <= c.n_last;) {
        int left = GroupEnd::stretch(n, c.n_last);
        for (; left > 0; --left, ++n) {
            {
                const int di = in_q.wait();
                const int dq = out.acquire();
                const double* in = &sm.s12[di][0][lane];
                double* o = &sm.s23[dq][0][lane];
                const double s_n = S.value();   // the action at grid point n
                if (c.have && n >= c.n0 && n < c.n_last && alive[lane]) {
                    StepMat<double> M;
#pragma unroll
                    for (int k = 0; k < 15; ++k) M.m[k] = in[k * kW];
#pragma unroll
                    for (int k = 15; k < 19; ++k) M.m[k] = 0.0;   // the bins warp advances the out-of-plane block
                    T.apply_step_matrix(M);
                }
                if (c.have && n >= c.n0 && n < c.n_last) {
                    double qs[4][2], ps[4][2], Vs[4];
                    qs[0][1] = in[20 * kW];   // the state at n: q_z, p_x', p_z
                    ps[0][0] = in[21 * kW];
                    ps[0][1] = in[22 * kW];
#pragma unroll
                    for (int k = 1; k < 4; ++k) {
                        qs[k][1] = in[(22 + k) * kW];
                        ps[k][0] = in[(24 + 2 * k) * kW];
                        ps[k][1] = in[(25 + 2 * k) * kW];
                    }
#pragma unroll
                    for (int k = 0; k < 4; ++k) {
                        qs[k][0] = 0.0;   // not read by the action terms
                        Vs[k] = in[(32 + k) * kW];
                    }
                    auto e_at = [&](int64_t j) { return j < f.table_len ? __ldg(f.E64 + j) : 0.0; };
                    S.add(TrajP<double, POT>::action_increment(ps, qs, Vs, e_at(2 * n), e_at(2 * n + 1), e_at(2 * n + 2),
                                                               h6));
                }
#pragma unroll
                for (int k = 0; k < 4; ++k) {
                    o[(4 * k) * kW] = T.X[k][0];
                    o[(4 * k + 1) * kW] = T.X[k][1];
                    o[(4 * k + 2) * kW] = T.Y[k][0];
                    o[(4 * k + 3) * kW] = T.Y[k][1];
                }
#pragma unroll
                for (int k = 0; k < 8; ++k) o[(16 + k) * kW] = in[(15 + k) * kW];   // g of the stages, state
                o[24 * kW] = s_n;
                in_q.release(di);
                out.publish(dq);
            }
        }
        if (GroupEnd::here(sm.last, n - 1)) break;
    }
    out.drain();
}

// bins: det Z and its branch, labels, removal, prefactor and the recombination
// sums of the bins, a few GTO terms per grid point
template <int POT>
__device__ void run_bins(const FieldDev& f, const TargetDev& tg, const GtoTerms& gt, const TrajArgs& a,
                         const Common& c, Shared& sm, int lane) {
    const Cx<double> amp{c.have ? a.amp_re[c.i] : 0.0, c.have ? a.amp_im[c.i] : 0.0};
    const bool fbins = a.float_bins != 0;   // recombination terms in float (as the float pass forms them)
    const float gamf = (float)a.gamma;
    const int tps = (gt.n + c.n_out - 1) / c.n_out > 0 ? (gt.n + c.n_out - 1) / c.n_out : 1;
    TrajP<double, POT> T;                    // holds the columns read from the slots for detc
    T.init(0.0, 0.0, 0.0, 0.0, 0.0, 0.0);
    bool alive = c.alive0;
    unsigned flags = (c.have && !alive) ? 8u : 0u;
    Cx2<double> Dp{8.0, 0.0};               // 8 det Z (of 2 Z: powers of two, exact)
    double sgn = 1.0;
    const double rg = a.gamma;
    const StepK<double> hk = f.k64;
    const bool pw = a.pw_mask != 0;
    const double pw_r2 = a.pw_radius * a.pw_radius;
    int pw_cls = -1;
    bool pw_in = false;
    unsigned long long all_steps = 0, steps = 0;
    // the bin in progress
    bool pending = false, valid = false;
    int64_t k_bin = 0;
    int j_next = 0;
    double bq0 = 0, bq2 = 0, bp0 = 0, bp2 = 0, bS = 0, p2s = 0, q2s = 0, pqs = 0;
    float p2f = 0.f, q2f = 0.f, pqf = 0.f, most = 0.f;   // most: size of the largest GTO term (FP64 bins)
    Cx<double> C{0.0, 0.0};
    GtoSums<double> acc{};
    GtoSums<float> accf{};
    auto terms = [&](int j0, int j1) {
        if (fbins) {
            gto_terms<float>(gt, p2f, q2f, pqf, j0, j1, accf);
        } else {
            for (int j = j0; j < j1; ++j)
                if (!(gto_size(gt, p2f, q2f, j) < most - kGtoNothing)) gto_terms<double>(gt, p2s, q2s, pqs, j, j + 1, acc);
        }
    };
    auto finish = [&]() {
        double cl = 0.0, cv = 0.0;
        if (valid) {
            terms(j_next, gt.n);
            const int64_t nb = k_bin * c.n_out;
            const double tk = f.t_start + (double)nb * f.dt;
            double sn, cs;
            sincos(fmod_2pi(tg.ip * tk), &sn, &cs);
            if (fbins) {
                float fl, fv;
                contribution_final<float>(FloatState(bq0, 0.0, bq2, bp0, 0.0, bp2, bS), gt, gamf,
                                          Cx<float>{(float)C.re, (float)C.im}, Cx<float>{(float)amp.re, (float)amp.im},
                                          Cx<float>{(float)cs, (float)(-sn)}, accf, fl, fv);
                cl = (double)fl;
                cv = (double)fv;
            } else {
                contribution_final<double>(PView(bq0, bq2, bp0, bp2, bS), gt, a.gamma, C, amp, Cx<double>{cs, -sn},
                                           acc, cl, cv);
            }
        }
        if (__any_sync(0xffffffffu, cl != 0.0 || cv != 0.0)) {
#pragma unroll
            for (int o = 16; o > 0; o >>= 1) {
                cl += __shfl_xor_sync(0xffffffffu, cl, o);
                cv += __shfl_xor_sync(0xffffffffu, cv, o);
            }
            const double sl = 0.0 + cl, sv = 0.0 + cv;
            if (lane == 0 && k_bin < f.n_bins && (sl != 0.0 || sv != 0.0)) {
                atomicAdd(&a.d_len[k_bin], sl);
                atomicAdd(&a.d_vel[k_bin], sv);
            }
        }
        pending = false;
    };
    int rem = (int)(c.n_first % c.n_out);
    int64_t k_next = (c.n_first + c.n_out - 1) / c.n_out;   // bin index of the next output point
    volatile int* alive_out = sm.alive;
    Consumer<2> in_q(kHand2);
    for (int64_t n = c.n_first; n <= c.n_last;) {
        int left = GroupEnd::stretch(n, c.n_last);
        for (; left > 0; --left, ++n) {
            {
                const int di = in_q.wait();
                const double* in = &sm.s23[di][0][lane];
                const double q0 = in[20 * kW], q2 = in[21 * kW], p0 = in[22 * kW], p2 = in[23 * kW], S = in[24 * kW];
                const bool on_bin = rem == 0;
                // partial waves (Sec. III.A-B): class at each entry into r < R, labels at
                // every grid point from birth on while the trajectory is integrated
                if (pw && alive && n >= c.n0) {
                    const double qx = q0, qy = 0.0, qz = q2;
                    const bool inside = qx * qx + qy * qy + qz * qz < pw_r2;
                    if (inside && !pw_in) {
                        const double px = p0, py = 0.0, pz = p2;
                        const double lx = qy * pz - qz * py, ly = qz * px - qx * pz, lz = qx * py - qy * px;
                        const double L2 = lx * lx + ly * ly + lz * lz;
                        pw_cls = L2 < 0.25 ? 0 : (L2 < 2.25 ? 1 : (L2 < 6.25 ? 2 : 3));
                    }
                    pw_in = inside;
                }
                const bool pw_ok = !pw || (pw_cls >= 0 && ((a.pw_mask >> pw_cls) & 1));
                if (on_bin) {
                    if (pending) finish();
                    valid = false;
                    if (alive && n >= c.n0) {
                        const double fs = q0 + q2 + p0 + p2;
                        const bool ok = isfinite(fs) && isfinite(S);
                        const cd D = 0.125 * cd{Dp.re, Dp.im};
                        const double m2 = D.re * D.re + D.im * D.im;
                        if (!ok || !(m2 <= a.d_t * a.d_t)) {
                            alive = false;
                            flags |= 1u;
                            if (!ok || !isfinite(m2)) flags |= 2u;
                        } else if (n >= c.k_cnt && pw_ok) {
                            cd Cz = root_det(D, m2);
                            if (sgn < 0.0) Cz = -Cz;
                            C = Cx<double>{Cz.re, Cz.im};
                            valid = true;
                            bq0 = q0;
                            bq2 = q2;
                            bp0 = p0;
                            bp2 = p2;
                            bS = S;
                            if (fbins)
                                recomb_invariants<float>(FloatState(bq0, 0.0, bq2, bp0, 0.0, bp2, bS), p2f, q2f, pqf);
                            else {
                                recomb_invariants<double>(PView(bq0, bq2, bp0, bp2, bS), p2s, q2s, pqs);
                                p2f = (float)p2s;
                                q2f = (float)q2s;
                                most = -INFINITY;
                                for (int j = 0; j < gt.n; ++j) most = fmaxf(most, gto_size(gt, p2f, q2f, j));
                            }
                        }
                    }
                    k_bin = k_next++;
                    pending = true;
                    j_next = 0;
                    acc = GtoSums<double>{};
                    accf = GtoSums<float>{};
                }
                // the step n -> n + 1: det Z of the advanced columns and its branch
                if (alive && n >= c.n0 && n < c.n_last) {
#pragma unroll
                    for (int k = 0; k < 4; ++k) {
                        T.X[k][0] = in[(4 * k) * kW];
                        T.X[k][1] = in[(4 * k + 1) * kW];
                        T.Y[k][0] = in[(4 * k + 2) * kW];
                        T.Y[k][1] = in[(4 * k + 3) * kW];
                    }
                    // the out-of-plane block, H_s = g_s (TrajP::step_matrix and apply_step_matrix)
                    const double g0 = in[16 * kW], g1 = in[17 * kW], g2 = in[18 * kW], g3 = in[19 * kW];
                    const double g23 = g1 + g2;
                    const double oa = fma(hk.c4, g2 * g0, -hk.c2 * (g23 + g0)), ob = fma(-hk.c3, g23, hk.h);
                    const double oc = fma(hk.c3, fma(g2, g0, g3 * g1), -hk.h6 * (fma(2.0, g23, g0) + g3));
                    const double od = fma(hk.c4, g3 * g1, -hk.c2 * (g23 + g3));
                    const double ya = T.aq, pa = T.ap, yb = T.bq, pb = T.bp;
                    T.aq = fma(oa, ya, fma(ob, pa, ya));
                    T.ap = fma(oc, ya, fma(od, pa, pa));
                    T.bq = fma(oa, yb, fma(ob, pb, yb));
                    T.bp = fma(oc, yb, fma(od, pb, pb));
                    const Cx2<double> D = T.detc(1.0, -2.0 * rg, 2.0 * a.qg64);
                    follow_branch<double>(Dp, D, sgn, flags);
                    ++all_steps;
                    if (n >= c.k_cnt) ++steps;
                }
                in_q.release(di);
                alive_out[lane] = alive ? 1 : 0;
                rem = (rem + 1 == c.n_out) ? 0 : rem + 1;
            }
            if (pending) {
                const int j_end = j_next + tps < gt.n ? j_next + tps : gt.n;
                if (valid) terms(j_next, j_end);
                j_next = j_end;
                if (j_next >= gt.n) finish();
            }
        }
        if (GroupEnd::here(sm.last, n - 1)) break;
    }
    if (pending) finish();
    if (a.stats) {
        unsigned rm = __reduce_add_sync(0xffffffffu, (flags & 1u) ? 1u : 0u);
        unsigned nf = __reduce_add_sync(0xffffffffu, (flags & 2u) ? 1u : 0u);
        unsigned bg = __reduce_add_sync(0xffffffffu, (flags & 4u) ? 1u : 0u);
        unsigned sk = __reduce_add_sync(0xffffffffu, (flags & 8u) ? 1u : 0u);
        unsigned long long st = steps, ast = all_steps;
#pragma unroll
        for (int o = 16; o > 0; o >>= 1) {
            st += __shfl_xor_sync(0xffffffffu, st, o);
            ast += __shfl_xor_sync(0xffffffffu, ast, o);
        }
        if (lane == 0) {
            if (rm) atomicAdd(&a.stats->removed, (unsigned long long)rm);
            if (nf) atomicAdd(&a.stats->nonfinite, (unsigned long long)nf);
            if (bg) atomicAdd(&a.stats->branch_guard, (unsigned long long)bg);
            if (sk) atomicAdd(&a.stats->skipped, (unsigned long long)sk);
            if (a.idx && ast) atomicAdd(&a.stats->esc_steps, ast);
            if (a.idx && ast > st) atomicAdd(&a.stats->esc_steps_pre, ast - st);
            if (st) atomicAdd(&a.stats->traj_steps, st);
        }
    }
}

// One group of 32 list entries (list positions 32 g .. 32 g + 31).
template <int POT>
__device__ void redo_group(const FieldDev& f, const TargetDev& tg, const GtoTerms& gt, const TrajArgs& a,
                           int64_t g, int64_t n_list, Shared& sm, int lane, int warp) {
    Common c;
    c.n_out = (int)f.n_out;
    c.n_last = a.n_last;
    const int64_t j = g * kW + lane;
    c.have = j < n_list;
    c.i = c.have ? (a.idx ? (int64_t)a.idx[j] : j) : 0;
    const int64_t k_min = (c.have && a.k_from) ? (int64_t)a.k_from[j] : 0;
    c.k_cnt = k_min * c.n_out;
    c.n0 = c.have ? (int64_t)a.n0[c.i] : 0;
    const double ar = c.have ? a.amp_re[c.i] : 0.0, ai = c.have ? a.amp_im[c.i] : 0.0;
    c.alive0 = c.have && c.n0 <= a.n_last && c.n0 >= 0 && (ar != 0.0 || ai != 0.0);
    // first grid point of the block: the earliest birth among its live trajectories
    long long m = c.alive0 ? (long long)c.n0 : LLONG_MAX;
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) {
        const long long t = __shfl_xor_sync(0xffffffffu, m, o);
        m = t < m ? t : m;
    }
    if (m == LLONG_MAX) {
        // nothing to integrate; one warp still reports skipped births
        if (a.stats && warp == 0) {
            const unsigned sk = __reduce_add_sync(0xffffffffu, c.have ? 1u : 0u);
            if (lane == 0 && sk) atomicAdd(&a.stats->skipped, (unsigned long long)sk);
        }
        return;
    }
    c.n_first = m;
    if (warp == 0) sm.alive[lane] = c.alive0 ? 1 : 0;
    if (threadIdx.x == 0) sm.last = -1;
    __syncthreads();
    const int role = (warp + (int)(g & 3)) & 3;
    if (role == 0) run_dynamics<POT>(f, tg, a, c, sm, lane);
    else if (role == 1) run_matrix<POT>(f, c, sm, lane);
    else if (role == 2) run_columns<POT>(f, c, sm, lane);
    else run_bins<POT>(f, tg, gt, a, c, sm, lane);
}

// Groups to SMs.  The list is in birth order, so group g's length (grid points from
// its earliest birth to the end) falls with g.  One warp plans the launch: it takes
// the groups longest first and gives each to the list (one per SM) with the least
// length so far (longest-processing-time-first), then lays the lists out in the
// scratch (plan: [0, L) counters, [K, K + L) list lengths, [2K, 2K + L) list starts,
// [3K, 3K + G) the groups list by list, longest first, then the assignment of each
// group; K = kRedoLists).  A block takes the groups of its own SM's list (one atomic
// counter per list), longest first, and then those left on the other lists, so
// every group is taken exactly once whatever the SMs' numbering and the blocks'
// placement.
__global__ void redo_plan_kernel(const int32_t* __restrict__ idx, const int32_t* __restrict__ n0,
                                 const int32_t* __restrict__ count, int64_t n_last, int L, int64_t quad_limit, int64_t g_max,
                                 int* plan) {
    __shared__ long long load[kRedoLists];
    __shared__ int cursor[kRedoLists];
    const int lane = threadIdx.x;   // one warp
    int* const len = plan + kRedoLists;
    int* const start = plan + 2 * kRedoLists;
    int* const grp = plan + 3 * kRedoLists;
    int* const asg = grp + g_max;
    const int64_t n_list = *count;
    const int W = n_list <= quad_limit ? kQuadWidth : kW;   // trajectories per group
    const int64_t G = min((n_list + W - 1) / W, g_max);
    for (int l = lane; l < L; l += 32) {
        load[l] = 0;
        cursor[l] = 0;
    }
    __syncwarp();
    for (int64_t g = 0; g < G; ++g) {
        // the group's length: from its earliest birth in range to the end
        const int64_t j = g * W + lane;
        long long m = LLONG_MAX;
        if (lane < W && j < n_list) {
            const long long b = n0[idx[j]];
            if (b >= 0 && b <= n_last) m = b;
        }
#pragma unroll
        for (int o = 16; o > 0; o >>= 1) m = min(m, (long long)__shfl_xor_sync(0xffffffffu, m, o));
        const long long lg = m == LLONG_MAX ? 1 : n_last - m + 1;
        // the least loaded list (ties: the lowest index)
        long long bv = LLONG_MAX;
        int bl = 0;
        for (int l = lane; l < L; l += 32)
            if (load[l] < bv) {
                bv = load[l];
                bl = l;
            }
#pragma unroll
        for (int o = 16; o > 0; o >>= 1) {
            const long long ov = __shfl_xor_sync(0xffffffffu, bv, o);
            const int ol = __shfl_xor_sync(0xffffffffu, bl, o);
            if (ov < bv || (ov == bv && ol < bl)) {
                bv = ov;
                bl = ol;
            }
        }
        if (lane == 0) {
            load[bl] += lg;
            ++cursor[bl];
            asg[g] = bl;
        }
        __syncwarp();
    }
    // list starts: exclusive prefix of the list lengths
    if (lane == 0) {
        int acc = 0;
        for (int l = 0; l < L; ++l) {
            len[l] = cursor[l];
            start[l] = acc;
            acc += cursor[l];
            cursor[l] = 0;
        }
        // the groups list by list, in order of g (longest first)
        for (int64_t g = 0; g < G; ++g) {
            const int l = asg[g];
            grp[start[l] + cursor[l]++] = (int)g;
        }
    }
}

template <int POT>
__global__ void __launch_bounds__(kThreads, 4) redo_kernel(FieldDev f, TargetDev tg, GtoTerms gt, TrajArgs a) {
    __shared__ Shared sm;
    __shared__ long long s_g;
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    const int64_t n_list = a.count ? (int64_t)*a.count : a.n;
    if (a.count && n_list <= a.quad_limit) return;   // a short list: quad.cu takes it
    GroupSource src(a, (n_list + kW - 1) / kW);
    for (;;) {
        const int64_t g = src.next(a, s_g);
        if (g < 0) break;
        redo_group<POT>(f, tg, gt, a, g, n_list, sm, lane, warp);
        __syncthreads();   // every role has drained its hand-offs before the next group
    }
}

template <int POT>
cudaError_t launch_pot(const FieldDev& f, const TargetDev& t, const GtoTerms& gt, const TrajArgs& a, cudaStream_t s) {
    // with a plan: persistent, as many blocks as fit on every SM (4), each looping over the
    // groups of its SM's list; without one: a block per group
    const int64_t blocks = a.redo_ctr ? (int64_t)a.redo_lists * 4 : (a.n + kW - 1) / kW;
    redo_kernel<POT><<<(unsigned)blocks, kThreads, 0, s>>>(f, t, gt, a);
    return cudaGetLastError();
}

cudaError_t launch_wide(const FieldDev& f, const TargetDev& t, const TrajArgs& a, cudaStream_t s) {
    const GtoTerms gt = make_gto_terms(t, a.gamma);
    switch (t.pot) {
        case POT_SOFTCORE: return launch_pot<POT_SOFTCORE>(f, t, gt, a, s);
        case POT_TONGLIN: return launch_pot<POT_TONGLIN>(f, t, gt, a, s);
        case POT_HARMONIC: return launch_pot<POT_HARMONIC>(f, t, gt, a, s);
        default: return launch_pot<POT_ZERO>(f, t, gt, a, s);
    }
}

}  // namespace

int redo_lists() {
    int dev = 0, sms = 0;
    if (cudaGetDevice(&dev) != cudaSuccess) return 1;
    if (cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, dev) != cudaSuccess) return 1;
    return std::max(1, std::min(sms, kRedoLists));
}

// Longest list for the four-lane kernel.  Set by FP64 instructions per step of a group, 64
// cycles each on the longest role and 19 of the SM for all roles: m groups of 8 per SM take
// at least m x 114 x 19 cycles (soft-core; Tong-Lin m x 211 x 19), one group of 32 takes 6,300
// (24,700).  Measured on both sides, 800 nm 1 cycle, 152 SMs, bins every fifth step:
//   lists, float bins     soft-core  9.2 ms at 2175 entries, 32-wide 17.7 ms at 2507;
//                         Tong-Lin  29.7 ms at 5369, 64.2 ms at 6191;
//   FP64 calls and bins   soft-core 10.6 ms at 2432, 26.5 ms at 2433;
//                         harmonic  10.9 and 30.2 ms; Tong-Lin 29.3 ms at 6080, 66.0 ms at 6081.
// The lines lie on the safe side of where the two meet.
int64_t quad_limit(int pot, int lists) { return (int64_t)kQuadWidth * lists * (pot == POT_TONGLIN ? 5 : 2); }

// Longest FP64 dipole call for the warp-specialised kernels.  The harmonic force leaves the
// bins warp with most of the work, and the one-thread kernel is even from 80,000 births on
// 152 SMs and faster beyond: its time over the 32-wide kernel's is 1.36 at 50,000, 1.00 at
// 80,000, 0.98 at 100,000, 0.96 at 1e6; soft-core 1.05, Tong-Lin 1.01 and free 1.07 at 1e6
// (800 nm, 1 cycle).
int64_t fp64_limit(int pot, int sms) { return pot == POT_HARMONIC ? (int64_t)kW * sms * 16 : INT64_MAX; }

cudaError_t launch_fp64(const FieldDev& f, const TargetDev& t, const TrajArgs& a, cudaStream_t s) {
    if (a.n == 0) return cudaSuccess;
    if (a.redo_lists < 1 || a.redo_lists > kRedoLists) return cudaErrorInvalidValue;
    if (a.n <= a.quad_limit) return launch_quad(f, t, a, s);
    return launch_wide(f, t, a, s);
}

cudaError_t launch_redo(const FieldDev& f, const TargetDev& t, const TrajArgs& a, cudaStream_t s) {
    if (a.n == 0) return cudaSuccess;
    if (a.redo_lists < 1 || a.redo_ctr == nullptr) return cudaErrorInvalidValue;
    if (a.redo_lists > kRedoLists) return cudaErrorInvalidValue;
    cudaError_t e = cudaMemsetAsync(a.redo_ctr, 0, (size_t)a.redo_lists * sizeof(int), s);
    if (e != cudaSuccess) return e;
    redo_plan_kernel<<<1, 32, 0, s>>>(a.idx, a.n0, a.count, a.n_last, a.redo_lists, a.quad_limit,
                                      redo_groups(a.n, a.quad_limit), a.redo_ctr);
    e = cudaGetLastError();
    // the list's length is on the device: the kernel that it is not meant for returns at once
    if (e == cudaSuccess && a.quad_limit > 0) e = launch_quad(f, t, a, s);
    if (e == cudaSuccess && a.n > a.quad_limit) e = launch_wide(f, t, a, s);
    return e;
}

}  // namespace sfhk
