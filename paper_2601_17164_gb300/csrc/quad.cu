// FP64 planar trajectories with four lanes per trajectory, for short lists.
//
// On GB300 a warp's FP64 instruction holds its sub-partition's FP64 unit for 64
// cycles however many of its 32 lanes are active and however independent the
// instructions are (measured: 64.1 cycles for chains of 1 to 8 independent FMAs, 1
// to 32 lanes; 76 with all four sub-partitions busy).  A trajectory's speed is
// therefore the number of FP64 warp instructions of one step, and a list too short
// to fill the chip with 32 trajectories a block (redo.cu) runs at the pace of the
// dynamics warp while most SMs idle.  Here a block of four warps holds 8
// trajectories and every trajectory has four lanes, which split the work inside a
// step so that one instruction does four parts of it:
//   dynamics  lanes = {x', z} x {stages 1 and 3, stages 2 and 4}: the force does not
//             depend on the momentum, so two stages run side by side; the RK4
//             combination of q in the one pair, of p in the other;
//   matrix    lane s forms stage s's Hessian and action integrand, then lane (i, j)
//             the entries (i, j) of A, B, C and D;
//   columns   lane c advances column c, lane k one entry of the out-of-plane block;
//   bins      labels, removal and the recombination terms, those of an FP64 bin in four
//             parts, with the two phases of the bin in one sincos;
// det Z (lane j forms column j of Z, even lanes the real and odd lanes the imaginary part)
// goes to the bins warp when the recombination terms are formed in float, to the columns
// warp when FP64 terms load the bins warp.
// FP64 instructions of the longest chain, the dynamics: 84 -> 29 a step (soft-core), 380 ->
// 111 (Tong-Lin); of all four warps 114 and 211 (ncu, FP64 bins left out).  A block alone on
// its SM steps in 2,900 cycles (float bins; FP64 3,800) where 32 trajectories a block take
// 6,300 (Tong-Lin: 8,000 to 8,500 and 24,700), with 1.5 times the FP64 work per trajectory,
// so the host and the plan choose by list length (quad_limit).  Measured: mixed H 8 cycles,
// 4096 births (110 redone) 333 -> 169 ms; mixed Ar 6 cycles, 5e4 births 1730 -> 650 ms; FP64
// H 2 cycles, 1024 births 143 -> 22 ms.
//
// Every value is formed by the same operations in the same order as in TrajP
// (traj_block.cuh): trajectories, columns, determinants, branches and removals are
// those of the other FP64 kernels bit for bit; sums over trajectories differ in
// order.
#include <algorithm>

#include "redo_warps.cuh"
#include "sfhk_internal.cuh"

namespace sfhk {
namespace {

constexpr int kT = kQuadWidth;   // trajectories per block
constexpr int kThreads = 128;
// dynamics -> matrix, per stage: q (2), g, 1/r, p (2), then soft-core: 1/r^2 (r with the
// core's radius), Tong-Lin: Y, Y1, e2, e4, e6;
// the stage stride puts lanes of neighbouring stages on different banks
constexpr int kFields = 12;
constexpr int kStage = kFields * kT + kT;
// matrix -> columns: A, B, C, D (4 entries each), the out-of-plane rows (a, b), (c, d) or
// (float bins) g of the stages, state, the action's integrand at the four stages
constexpr int kM = 16, kState = 20, kAct = 24, kN12 = 28;
// columns -> bins: state at grid point n, then (float bins) the action there, the columns
// after the step (4 x 4) and the out-of-plane block (4), or the action's four integrands,
// 8 det Z (2) and its branch at grid point n
constexpr int kDetF = 5, kDetD = 8, kN23 = 25;

// barrier bases of the three hand-offs; the last one has three slots, which the bins warp's
// longer grid points (those with a bin) need
constexpr int kHand0 = 1, kHand1 = 5, kHand2 = 9;

struct QShared {
    double s01[2][4 * kStage];
    double s12[2][kN12 * kT];
    double s23[3][kN23 * kT];
    double hess[4 * 3 * kT];   // stage Hessians (a, b, c), matrix warp only
    double phase[16][2];       // cos and -sin of Ip t at bin k in row k & 15 (float bins)
    int alive[kT];             // written by the bins warp, read late by the warps ahead
    long long last;            // the group's last grid point when it ends early, else -1 (GroupEnd)
};

struct QCommon {
    int64_t n_first, n_last;   // first and last grid point of the block
    int n_out;
    bool have;
    int64_t i, n0, k_cnt;
    bool alive0;
    int t, l;                  // trajectory in the block, lane of the trajectory
};

__device__ __forceinline__ double from_lane(double v, int lane) { return __shfl_sync(0xffffffffu, v, lane); }
__device__ __forceinline__ double xor_lane(double v, int m) { return __shfl_xor_sync(0xffffffffu, v, m); }

template <int POT>
__device__ __forceinline__ PotConst<double> pot_const(const TargetDev& tg) {
    PotConst<double> pc;
    pc.a2 = (POT == POT_SOFTCORE || POT == POT_HARMONIC) ? tg.pot_param[0] * tg.pot_param[0] : 0.0;
    pc.Zc = tg.pot_param[0]; pc.a1 = tg.pot_param[1]; pc.a2t = tg.pot_param[2];
    pc.a3 = tg.pot_param[3]; pc.a4 = tg.pot_param[4]; pc.a5 = tg.pot_param[5];
    pc.a6 = tg.pot_param[6];
    return pc;
}

// Ip t mod 2 pi at grid point n
__device__ __forceinline__ double bin_phase(const FieldDev& f, const TargetDev& tg, int64_t n) {
    return fmod_2pi(tg.ip * (f.t_start + (double)n * f.dt));
}

// dynamics: the state at grid point n and the stages of the step n -> n + 1.  The force
// does not depend on the momentum, so the RK4 positions are
//   Q1, Q2 = Q1 + h/2 P1, Q3 = Q1 + h/2 P2, Q4 = Q1 + h P3,
//   P2 = P1 + h/2 F(Q1), P3 = P1 + h/2 F(Q2), P4 = P1 + h F(Q3):
// the forces of stages 1 and 2 are formed side by side, then those of 3 and 4.  Lane
// (component c = l & 1, pair g = l >> 1) takes stages 1 and 3 (g = 0) or 2 and 4.
template <int POT, bool FB>
__device__ void quad_dynamics(const FieldDev& f, const TargetDev& tg, const TrajArgs& a, const QCommon& cm,
                              QShared& sm) {
    const PotConst<double> pc = pot_const<POT>(tg);
    const int t = cm.t, c = cm.l & 1, pair = cm.l >> 1;
    double q1, p1;   // this lane's component of the state
    {
        TrajP<double, POT> T;
        T.init(0.0, 0.0, cm.have ? a.qz[cm.i] : 0.0, cm.have ? a.px[cm.i] : 0.0, cm.have ? a.py[cm.i] : 0.0,
               cm.have ? a.pz[cm.i] : 0.0);
        q1 = c ? T.q[2] : T.q[0];
        p1 = c ? T.p[2] : T.p[0];
    }
    const StepK<double> hk = f.k64;
    const double* E = f.E64;
    auto e_at = [&](int64_t j) { return j < f.table_len ? __ldg(E + j) : 0.0; };
    double e0 = e_at(2 * cm.n_first), e1 = e_at(2 * cm.n_first + 1), e2 = e_at(2 * cm.n_first + 2);
    const volatile int* alive = sm.alive;
    // Tong-Lin: this lane's first exponent, and its constants of Y (c = 0) or Y' (c = 1)
    const double ea = c ? -pc.a4 : -pc.a2t, t_r = c ? -pc.a4 : 1.0, t_1 = c ? 1.0 : 0.0, t_0 = c ? 0.0 : pc.Zc,
                 t_2 = c ? -pc.a1 * pc.a2t : pc.a1, t_6 = c ? -(pc.a5 * pc.a6) : pc.a5;
    Producer<2> out(kHand0);
    // the force at a stage from this lane's component q of its position; the stage's
    // Hessian data into the slot at os
    auto force = [&](double q, double ek, double* os, double& g) {
        const double qo = xor_lane(q, kT);
        const double x = c ? qo : q, z = c ? q : qo;
        double aux = 0.0;
        if constexpr (POT == POT_SOFTCORE) {
            const double r2 = fma(x, x, fma(z, z, pc.a2));
            const double s = rsq(r2);
            const double s2 = s * s;
            g = s2 * s;
            aux = s;
            if (c == 0) os[6 * kT] = s2;
        } else if constexpr (POT == POT_TONGLIN) {
            const double r2 = fma(x, x, z * z);
            const double ir = rsq(r2);
            const double r = r2 * ir;
            const double ex_l = ex(ea * r), x6 = ex(-pc.a6 * r);
            const double ex_o = xor_lane(ex_l, kT);
            const double x2 = c ? ex_o : ex_l, x4 = c ? ex_l : ex_o;
            // Y in even and Y' in odd lanes, 5 instructions instead of 9
            const double t3 = pc.a3 * fma(t_r, r, t_1);
            const double v = fma(c ? t3 : t_2, c ? x4 : x2, t_0);
            const double yl = fma(t_6, x6, fma(c ? t_2 : t3, c ? x2 : x4, v));
            const double yo = xor_lane(yl, kT);
            g = tonglin_g(ir, c ? yo : yl, c ? yl : yo);
            aux = ir;
            os[(6 + c) * kT] = yl;
            os[(8 + c) * kT] = ex_l;
            if (c == 0) os[10 * kT] = x6;
        } else if constexpr (POT == POT_HARMONIC) {
            g = pc.a2;
        } else {
            g = 0.0;
        }
        os[c * kT] = q;                       // q_x', q_z
        os[(2 + c) * kT] = c ? aux : g;       // g, aux
        return -fma(g, q, c ? ek : 0.0);      // -g x' and -(g z + E)
    };
    int rem = (int)(cm.n_first % cm.n_out);
    int64_t k_bin = (cm.n_first + cm.n_out - 1) / cm.n_out;
    for (int64_t n = cm.n_first; n <= cm.n_last;) {
        int left = GroupEnd::stretch(n, cm.n_last);
        GroupEnd::decide(sm.last, n + left - 1, alive[t]);
        for (; left > 0; --left, ++n) {
            const int d = out.acquire();
            // float bins: e^{-i Ip t} of the bin at this grid point (this warp has the FP64
            // instructions to spare; the hand-offs keep the bins warp less than 16 grid points
            // behind, so a row is read before its next use even with a bin at every point)
            if (FB && rem == 0) {
                if (threadIdx.x % 32 == 0) {
                    double sn, cs;
                    sincos(bin_phase(f, tg, n), &sn, &cs);
                    sm.phase[k_bin & 15][0] = cs;
                    sm.phase[k_bin & 15][1] = -sn;
                }
                ++k_bin;
            }
            rem = (rem + 1 == cm.n_out) ? 0 : rem + 1;
            double* const o = sm.s01[d] + t;
            const double f0 = e_at(2 * n + 2), f1 = e_at(2 * n + 3), f2 = e_at(2 * n + 4);
            const bool step = cm.have && n >= cm.n0 && n < cm.n_last && alive[t];
            double g;
            const double qa = pair ? fma(hk.hh, p1, q1) : q1;                       // Q1, Q2
            const double ka = force(qa, pair ? e1 : e0, o + pair * kStage, g);      // F1, F2
            const double pn = fma(hk.hh, ka, p1);                                   // P2, P3
            const double qb = fma(pair ? hk.h : hk.hh, pn, q1);                     // Q3, Q4
            const double kb = force(qb, pair ? e2 : e1, o + (2 + pair) * kStage, g);   // F3, F4
            const double p4 = fma(hk.h, kb, p1);                                    // (P4 in the first pair)
            // stage momenta: P2 and P3, P1 and P4
            o[(1 + pair) * kStage + (4 + c) * kT] = pn;
            const double p4_o = xor_lane(p4, 2 * kT);
            o[(pair ? 3 * kStage : 0) + (4 + c) * kT] = pair ? p4_o : p1;
            out.publish(d);
            // the RK4 combination, q_c in the first pair and p_c in the second; the last term of
            // p_x' is -g x' unrounded (so nvcc contracts it in the other FP64 kernels: found by
            // comparing chaotic trajectories)
            const double pn_o = xor_lane(pn, 2 * kT), ka_o = xor_lane(ka, 2 * kT), kb_o = xor_lane(kb, 2 * kT);
            const double s3 = fma(2.0, (pair ? ka : pn) + (pair ? kb_o : pn_o), pair ? ka_o : p1);
            const bool px = pair && c == 0;
            const double s = fma(px ? -g : 1.0, px ? qb : (pair ? kb : p4), s3);
            const double nb = fma(hk.h6, s, pair ? p1 : q1);
            const double no = xor_lane(nb, 2 * kT);
            if (step) {
                q1 = pair ? no : nb;
                p1 = pair ? nb : no;
            }
            e0 = f0;
            e1 = f1;
            e2 = f2;
        }
        if (GroupEnd::here(sm.last, n - 1)) break;
    }
    out.drain();
}

// the out-of-plane rows: (a, b) in even lanes, (c, d) in odd lanes (TrajP::step_matrix)
__device__ __forceinline__ double2 out_of_plane(const StepK<double>& k, double g0, double g1, double g2, double g3,
                                                bool odd) {
    const double g23 = g1 + g2;
    const double ad = fma(k.c4, (odd ? g3 : g2) * (odd ? g1 : g0), -k.c2 * (g23 + (odd ? g3 : g0)));
    const double w = fma(g2, g0, g3 * g1), v = -k.h6 * (fma(2.0, g23, g0) + g3);
    const double bc = fma(odd ? k.c3 : -k.c3, odd ? w : g23, odd ? v : k.h);
    return odd ? make_double2(bc, ad) : make_double2(ad, bc);
}

// 8 det Z (of 2 Z: powers of two, exact) in every lane, from column l of the in-plane block
// and entry l of the out-of-plane one (TrajP::detc in parts); gz = -2 gamma, qz = 1/(2 gamma)
__device__ __forceinline__ Cx2<double> det8(double X0, double X1, double Y0, double Y1, double w, double gz, double qz,
                                            int t, bool odd) {
    const double X0p = xor_lane(X0, 2 * kT), X1p = xor_lane(X1, 2 * kT), Y0p = xor_lane(Y0, 2 * kT),
                 Y1p = xor_lane(Y1, 2 * kT);   // column l + 2 in lanes 0 and 1
    const double aq = from_lane(w, t), ap = from_lane(w, t + kT), bq = from_lane(w, t + 2 * kT),
                 bp = from_lane(w, t + 3 * kT);
    double zr0 = Y0p + X0, zr1 = Y1p + X1;
    double zi0 = fma(gz, X0p, qz * Y0), zi1 = fma(gz, X1p, qz * Y1);
    // column (l & 1) of Z in every lane, then both
    zr0 = from_lane(zr0, t + odd * kT);
    zr1 = from_lane(zr1, t + odd * kT);
    zi0 = from_lane(zi0, t + odd * kT);
    zi1 = from_lane(zi1, t + odd * kT);
    const double wr0 = xor_lane(zr0, kT), wr1 = xor_lane(zr1, kT), wi0 = xor_lane(zi0, kT), wi1 = xor_lane(zi1, kT);
    const double r00 = odd ? wr0 : zr0, r10 = odd ? wr1 : zr1, i00 = odd ? wi0 : zi0, i10 = odd ? wi1 : zi1;
    const double r01 = odd ? zr0 : wr0, r11 = odd ? zr1 : wr1, i01 = odd ? zi0 : wi0, i11 = odd ? zi1 : wi1;
    const double u1 = i00 * (odd ? r11 : i11), u2 = i01 * (odd ? r10 : i10);
    const double dd = fma(r00, odd ? i11 : r11, odd ? u1 : -u1) - fma(r01, odd ? i10 : r10, odd ? u2 : -u2);
    const double dx = xor_lane(dd, kT);
    const double ar = odd ? dx : dd, ai = odd ? dd : dx;
    // Z_yy: the real part in even and the imaginary part in odd lanes, then both
    double y = fma(odd ? qz : 1.0, odd ? ap : bp, odd ? 0.0 : aq);
    if (odd) y = fma(gz, bq, y);
    const double yx = xor_lane(y, kT);
    const double yr = odd ? yx : y, yi = odd ? y : yx;
    const double u3 = ai * (odd ? yr : yi);
    const double de = fma(ar, odd ? yi : yr, odd ? u3 : -u3);
    const double df = xor_lane(de, kT);
    return Cx2<double>{odd ? df : de, odd ? de : df};
}

// matrix: the step matrix of grid point n and the action's integrand at its stages
template <int POT, bool FB>
__device__ void quad_matrix(const FieldDev& f, const TargetDev& tg, const QCommon& cm, QShared& sm) {
    const PotConst<double> pc = pot_const<POT>(tg);
    const StepK<double> hk = f.k64;
    const int t = cm.t, l = cm.l, ei = l >> 1, ej = l & 1;
    const bool odd = l & 1;
    const double* E = f.E64;
    auto e_at = [&](int64_t j) { return j < f.table_len ? __ldg(E + j) : 0.0; };
    const int e_off = l == 0 ? 0 : (l == 3 ? 2 : 1);   // stage l reads E at t, t + h/2, t + h/2, t + h
    double e_cur = e_at(2 * cm.n_first + e_off);
    Consumer<2> in_q(kHand0);
    Producer<2> out(kHand1);
    const double h = hk.h, c2 = hk.c2, c4 = hk.c4, c3 = hk.c3, c1 = hk.h6;
    for (int64_t n = cm.n_first; n <= cm.n_last;) {
        int left = GroupEnd::stretch(n, cm.n_last);
        for (; left > 0; --left, ++n) {
            const double e_next = e_at(2 * n + 2 + e_off);
            const int di = in_q.wait();
            const double* const in = sm.s01[di] + t;
            // stage l: Hessian data and the action integrand
            const double* const st = in + l * kStage;
            const double x = st[0], z = st[kT], g = st[2 * kT], px = st[4 * kT], pz = st[5 * kT];
            double hs, V;
            if constexpr (POT == POT_SOFTCORE) {
                hs = -3.0 * g * st[6 * kT];
                V = -st[3 * kT];
            } else if constexpr (POT == POT_TONGLIN) {
                const double ir = st[3 * kT], Y = st[6 * kT], Y1 = st[7 * kT];
                const double r = fma(x, x, z * z) * ir;
                hs = tonglin_h(pc, r, ir, Y, Y1, st[8 * kT], st[9 * kT], st[10 * kT]);
                V = -Y * ir;
            } else if constexpr (POT == POT_HARMONIC) {
                hs = 0.0;
                V = 0.5 * pc.a2 * fma(x, x, z * z);
            } else {
                hs = 0.0;
                V = 0.0;
            }
            const double hx = hs * x;
            double* const H = sm.hess + t;
            H[(3 * l) * kT] = fma(hx, x, g);
            H[(3 * l + 1) * kT] = hx * z;
            H[(3 * l + 2) * kT] = fma(hs * z, z, g);
            const double kS = TrajP<double, POT>::action_term(px, pz, z, e_cur, V);
            const double g0 = in[2 * kT], g1 = in[kStage + 2 * kT], g2 = in[2 * kStage + 2 * kT],
                         g3 = in[3 * kStage + 2 * kT];
            const double state_l = in[(l < 2 ? l : l + 2) * kT];   // q_x', q_z, p_x', p_z at n
            in_q.release(di);
            __syncwarp();
            const int dq = out.acquire();
            double* const o = sm.s12[dq] + t;
            // entry (ei, ej) from row ei of H3, H4 and column ej of H1, H2
            auto He = [&](int s, int i, int j) { return H[(3 * s + i + j) * kT]; };
            const double h0e = He(0, ei, ej), h1e = He(1, ei, ej), h2e = He(2, ei, ej), h3e = He(3, ei, ej);
            const double p31 = fma(He(2, ei, 0), He(0, 0, ej), He(2, ei, 1) * He(0, 1, ej));
            const double p42 = fma(He(3, ei, 0), He(1, 0, ej), He(3, ei, 1) * He(1, 1, ej));
            __syncwarp();   // the Hessians are read before the next grid point writes them
            const double s23 = h1e + h2e;
            o[l * kT] = fma(c4, p31, -c2 * (s23 + h0e));
            o[(4 + l) * kT] = fma(-c3, s23, ei == ej ? h : 0.0);
            o[(8 + l) * kT] = fma(c3, p31 + p42, -c1 * (fma(2.0, s23, h0e) + h3e));
            o[(12 + l) * kT] = fma(c4, p42, -c2 * (s23 + h3e));
            if constexpr (FB) {
                o[(kM + l) * kT] = l == 0 ? g0 : (l == 1 ? g1 : (l == 2 ? g2 : g3));
            } else {
                const double2 r = out_of_plane(hk, g0, g1, g2, g3, odd);
                if (l < 2) {
                    o[(kM + 2 * l) * kT] = r.x;
                    o[(kM + 2 * l + 1) * kT] = r.y;
                }
            }
            o[(kState + l) * kT] = state_l;
            o[(kAct + l) * kT] = kS;
            out.publish(dq);
            e_cur = e_next;
        }
        if (GroupEnd::here(sm.last, n - 1)) break;
    }
    out.drain();
}

// columns: lane c advances column c of the in-plane block; lanes 0..3 hold
// dy/dy0, dpy/dy0, dy/dpy0, dpy/dpy0 of the out-of-plane block; with FP64 bins also det Z
// and its branch, with float bins (a light bins warp) the out-of-plane rows and the action
template <int POT, bool FB>
__device__ void quad_columns(const FieldDev& f, const TrajArgs& a, const QCommon& cm, QShared& sm) {
    const int t = cm.t, l = cm.l;
    const bool odd = l & 1;
    const StepK<double> hk = f.k64;
    const double gz = -2.0 * a.gamma, qz = 2.0 * a.qg64;
    double X0 = l == 0 ? 1.0 : 0.0, X1 = l == 1 ? 1.0 : 0.0, Y0 = l == 2 ? 1.0 : 0.0, Y1 = l == 3 ? 1.0 : 0.0;
    double w = (l == 0 || l == 3) ? 1.0 : 0.0;
    Cx2<double> Dp{8.0, 0.0};
    double sgn = 1.0;
    unsigned turned = 0;   // the step into this grid point moved arg det Z by more than pi/2
    double S = 0.0;        // the action at grid point n
    const volatile int* alive = sm.alive;
    Consumer<2> in_q(kHand1);
    Producer<3> out(kHand2);
    for (int64_t n = cm.n_first; n <= cm.n_last;) {
        int left = GroupEnd::stretch(n, cm.n_last);
        for (; left > 0; --left, ++n) {
            const int di = in_q.wait();
            const double* const in = sm.s12[di] + t;
            int dq = 0;
            if constexpr (!FB) {
                dq = out.acquire();
                double* const o = sm.s23[dq] + t;
                // 8 det Z at grid point n: re, im, the branch's sign (doubled after a turn)
                if (l < 3) o[(kDetD + l) * kT] = l == 0 ? Dp.re : (l == 1 ? Dp.im : (turned ? 2.0 * sgn : sgn));
                o[l * kT] = in[(kState + l) * kT];
                o[(4 + l) * kT] = in[(kAct + l) * kT];
                out.publish(dq);
            }
            const bool step = cm.have && n >= cm.n0 && n < cm.n_last && alive[t];
            const double wp = xor_lane(w, kT);   // the other entry of this out-of-plane column
            double m0, m1;
            if constexpr (FB) {
                const double2 r = out_of_plane(hk, in[kM * kT], in[(kM + 1) * kT], in[(kM + 2) * kT], in[(kM + 3) * kT], odd);
                m0 = r.x;
                m1 = r.y;
            } else {
                m0 = in[(kM + 2 * odd) * kT];
                m1 = in[(kM + 2 * odd + 1) * kT];
            }
            if (step) {
                const double x0 = X0, x1 = X1, y0 = Y0, y1 = Y1;
                X0 = fma(in[0], x0, fma(in[kT], x1, fma(in[4 * kT], y0, fma(in[5 * kT], y1, x0))));
                X1 = fma(in[2 * kT], x0, fma(in[3 * kT], x1, fma(in[5 * kT], y0, fma(in[7 * kT], y1, x1))));
                Y0 = fma(in[8 * kT], x0, fma(in[9 * kT], x1, fma(in[12 * kT], y0, fma(in[13 * kT], y1, y0))));
                Y1 = fma(in[10 * kT], x0, fma(in[11 * kT], x1, fma(in[14 * kT], y0, fma(in[15 * kT], y1, y1))));
                const double q = odd ? wp : w, p = odd ? w : wp;
                w = fma(m0, q, fma(m1, p, w));
            }
            if constexpr (FB) {
                const double state_l = in[(kState + l) * kT], s_n = S;
                if (cm.have && n >= cm.n0 && n < cm.n_last)
                    S += TrajP<double, POT>::action_sum(in[kAct * kT], in[(kAct + 1) * kT], in[(kAct + 2) * kT],
                                                        in[(kAct + 3) * kT], hk.h6);
                in_q.release(di);
                dq = out.acquire();
                double* const o = sm.s23[dq] + t;
                o[l * kT] = state_l;
                if (l == 0) o[4 * kT] = s_n;
                o[(kDetF + 4 * l) * kT] = X0;
                o[(kDetF + 4 * l + 1) * kT] = X1;
                o[(kDetF + 4 * l + 2) * kT] = Y0;
                o[(kDetF + 4 * l + 3) * kT] = Y1;
                o[(kDetF + 16 + l) * kT] = w;
                out.publish(dq);
            } else {
                in_q.release(di);
                const Cx2<double> D = det8(X0, X1, Y0, Y1, w, gz, qz, t, odd);
                turned = 0;
                if (step) follow_branch<double>(Dp, D, sgn, turned);
            }
        }
        if (GroupEnd::here(sm.last, n - 1)) break;
    }
    out.drain();
}

// bins: labels, removal, prefactor and the recombination sums
template <int POT, bool FB>
__device__ void quad_bins(const FieldDev& f, const TargetDev& tg, const GtoTerms& gt, const TrajArgs& a,
                          const QCommon& c, QShared& sm) {
    const int t = c.t, l = c.l;
    const Cx<double> amp{c.have ? a.amp_re[c.i] : 0.0, c.have ? a.amp_im[c.i] : 0.0};
    const float gamf = (float)a.gamma;
    bool alive = c.alive0;
    unsigned flags = (c.have && !alive) ? 8u : 0u;
    const bool pw = a.pw_mask != 0;
    const double pw_r2 = a.pw_radius * a.pw_radius;
    int pw_cls = -1;
    bool pw_in = false;
    unsigned long long all_steps = 0, steps = 0;
    double S = 0.0;   // the action at grid point n
    // float bins: 8 det Z and its branch
    const double gz = -2.0 * a.gamma, qz = 2.0 * a.qg64;
    Cx2<double> Dp{8.0, 0.0};
    double sgn = 1.0;
    int rem = (int)(c.n_first % c.n_out);
    int64_t k_bin = (c.n_first + c.n_out - 1) / c.n_out;   // bin index of the next output point
    volatile int* alive_out = sm.alive;
    Consumer<3> in_q(kHand2);
    for (int64_t n = c.n_first; n <= c.n_last;) {
        int left = GroupEnd::stretch(n, c.n_last);
        for (; left > 0; --left, ++n) {
            const int di = in_q.wait();
            const double* const in = sm.s23[di] + t;
            const double q0 = in[0], q2 = in[kT], p0 = in[2 * kT], p2 = in[3 * kT];
            double k1 = 0.0, k2 = 0.0, k3 = 0.0, k4 = 0.0;
            double X0 = 0.0, X1 = 0.0, Y0 = 0.0, Y1 = 0.0, w = 0.0;
            if constexpr (FB) {
                S = in[4 * kT];
                X0 = in[(kDetF + 4 * l) * kT];
                X1 = in[(kDetF + 4 * l + 1) * kT];
                Y0 = in[(kDetF + 4 * l + 2) * kT];
                Y1 = in[(kDetF + 4 * l + 3) * kT];
                w = in[(kDetF + 16 + l) * kT];
            } else {
                k1 = in[4 * kT];
                k2 = in[5 * kT];
                k3 = in[6 * kT];
                k4 = in[7 * kT];
                Dp = Cx2<double>{in[kDetD * kT], in[(kDetD + 1) * kT]};
                sgn = in[(kDetD + 2) * kT];
            }
            in_q.release(di);
            const bool on_bin = rem == 0;
            if (!FB && alive && (__double2hiint(sgn) & 0x7fffffff) == 0x40000000) flags |= 4u;   // |sgn| = 2
            // partial waves (Sec. III.A-B), as in redo.cu
            if (pw && alive && n >= c.n0) {
                const double qx = q0, qy = 0.0, qzz = q2;
                const bool inside = qx * qx + qy * qy + qzz * qzz < pw_r2;
                if (inside && !pw_in) {
                    const double px = p0, py = 0.0, pz = p2;
                    const double lx = qy * pz - qzz * py, ly = qzz * px - qx * pz, lz = qx * py - qy * px;
                    const double L2 = lx * lx + ly * ly + lz * lz;
                    pw_cls = L2 < 0.25 ? 0 : (L2 < 2.25 ? 1 : (L2 < 6.25 ? 2 : 3));
                }
                pw_in = inside;
            }
            const bool pw_ok = !pw || (pw_cls >= 0 && ((a.pw_mask >> pw_cls) & 1));
            if (on_bin) {
                bool valid = false;
                Cx<double> C{0.0, 0.0};
                if (alive && n >= c.n0) {
                    const cd D = 0.125 * cd{Dp.re, Dp.im};
                    const double fs = q0 + q2 + p0 + p2;
                    const bool ok = isfinite(fs) && isfinite(S);
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
                    }
                }
                if (__any_sync(0xffffffffu, valid)) {
                    double cl = 0.0, cv = 0.0;
                    if constexpr (FB) {
                        if (valid && l == 0) {
                            const FloatState fsn(q0, 0.0, q2, p0, 0.0, p2, S);
                            float fl, fv;
                            contribution<float>(fsn, gt, gamf, Cx<float>{(float)C.re, (float)C.im},
                                                Cx<float>{(float)amp.re, (float)amp.im},
                                                Cx<float>{(float)sm.phase[k_bin & 15][0], (float)sm.phase[k_bin & 15][1]}, fl, fv);
                            cl = (double)fl;
                            cv = (double)fv;
                        }
                    } else {
                        // e^{-i Ip t} in even lanes and e^{i S} in odd lanes
                        double sn, cs;
                        sincos((l & 1) ? S : bin_phase(f, tg, n), &sn, &cs);
                        const double sn_o = xor_lane(sn, kT), cs_o = xor_lane(cs, kT);   // lane 0: e^{i S}
                        // the GTO terms in four parts
                        const PView v(q0, q2, p0, p2, S);
                        double pp, qq, pq;
                        recomb_invariants<double>(v, pp, qq, pq);
                        const float ppf = (float)pp, qqf = (float)qq;
                        float most = -INFINITY;
                        for (int j = l; j < gt.n; j += 4) most = fmaxf(most, gto_size(gt, ppf, qqf, j));
                        most = fmaxf(most, __shfl_xor_sync(0xffffffffu, most, kT));
                        most = fmaxf(most, __shfl_xor_sync(0xffffffffu, most, 2 * kT));
                        GtoSums<double> g{};
                        for (int j = l; j < gt.n; j += 4)
                            if (valid && !(gto_size(gt, ppf, qqf, j) < most - kGtoNothing))
                                gto_terms<double>(gt, pp, qq, pq, j, j + 1, g);
                        auto fold = [](double& x) {
                            x += xor_lane(x, kT);
                            x += xor_lane(x, 2 * kT);
                        };
                        __syncwarp();
                        fold(g.s0.re);
                        fold(g.s0.im);
                        fold(g.s1.re);
                        fold(g.s1.im);
                        if (gt.l == 1) {
                            fold(g.s2.re);
                            fold(g.s2.im);
                            fold(g.s3.re);
                            fold(g.s3.im);
                        }
                        if (valid && l == 0)
                            contribution_closed<double>(v, gt, a.gamma, C, amp, Cx<double>{cs, -sn}, Cx<double>{cs_o, sn_o},
                                                        g, cl, cv);
                    }
                    __syncwarp();
#pragma unroll
                    for (int o = 4; o > 0; o >>= 1) {   // over the trajectories (lanes 0..7 hold them)
                        cl += xor_lane(cl, o);
                        cv += xor_lane(cv, o);
                    }
                    if ((threadIdx.x & 31) == 0 && k_bin < f.n_bins && (cl != 0.0 || cv != 0.0)) {
                        atomicAdd(&a.d_len[k_bin], cl);
                        atomicAdd(&a.d_vel[k_bin], cv);
                    }
                }
                ++k_bin;
            }
            alive_out[t] = alive ? 1 : 0;
            rem = (rem + 1 == c.n_out) ? 0 : rem + 1;
            if constexpr (FB) {
                // the step n -> n + 1: det Z of the advanced columns
                const Cx2<double> D = det8(X0, X1, Y0, Y1, w, gz, qz, t, l & 1);
                if (alive && n >= c.n0 && n < c.n_last) follow_branch<double>(Dp, D, sgn, flags);
            } else {
                if (c.have && n >= c.n0 && n < c.n_last) S += TrajP<double, POT>::action_sum(k1, k2, k3, k4, f.k64.h6);
            }
            if (alive && n >= c.n0 && n < c.n_last) {
                ++all_steps;
                if (n >= c.k_cnt) ++steps;
            }
        }
        if (GroupEnd::here(sm.last, n - 1)) break;
    }
    if (a.stats) {
        const bool one = l == 0;   // a trajectory is counted by its first lane
        unsigned rm = __reduce_add_sync(0xffffffffu, one && (flags & 1u) ? 1u : 0u);
        unsigned nf = __reduce_add_sync(0xffffffffu, one && (flags & 2u) ? 1u : 0u);
        unsigned bg = __reduce_add_sync(0xffffffffu, one && (flags & 4u) ? 1u : 0u);
        unsigned sk = __reduce_add_sync(0xffffffffu, one && (flags & 8u) ? 1u : 0u);
        unsigned long long st = one ? steps : 0, ast = one ? all_steps : 0;
#pragma unroll
        for (int o = 16; o > 0; o >>= 1) {
            st += __shfl_xor_sync(0xffffffffu, st, o);
            ast += __shfl_xor_sync(0xffffffffu, ast, o);
        }
        if ((threadIdx.x & 31) == 0) {
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

// One group of 8 list entries (list positions 8 g .. 8 g + 7).
template <int POT, bool FB>
__device__ void quad_group(const FieldDev& f, const TargetDev& tg, const GtoTerms& gt, const TrajArgs& a, int64_t g,
                           int64_t n_list, QShared& sm) {
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    QCommon c;
    c.t = lane & (kT - 1);
    c.l = lane / kT;
    c.n_out = (int)f.n_out;
    c.n_last = a.n_last;
    const int64_t j = g * kT + c.t;
    c.have = j < n_list;
    c.i = c.have ? (a.idx ? (int64_t)a.idx[j] : j) : 0;
    c.k_cnt = (c.have && a.k_from) ? (int64_t)a.k_from[j] * c.n_out : 0;
    c.n0 = c.have ? (int64_t)a.n0[c.i] : 0;
    const double ar = c.have ? a.amp_re[c.i] : 0.0, ai = c.have ? a.amp_im[c.i] : 0.0;
    c.alive0 = c.have && c.n0 <= a.n_last && c.n0 >= 0 && (ar != 0.0 || ai != 0.0);
    long long m = c.alive0 ? (long long)c.n0 : LLONG_MAX;   // first grid point of the block
#pragma unroll
    for (int o = 4; o > 0; o >>= 1) {
        const long long u = __shfl_xor_sync(0xffffffffu, m, o);
        m = u < m ? u : m;
    }
    if (m == LLONG_MAX) {
        // nothing to integrate; one warp still reports skipped births
        if (a.stats && warp == 0) {
            const unsigned sk = __reduce_add_sync(0xffffffffu, c.have && c.l == 0 ? 1u : 0u);
            if (lane == 0 && sk) atomicAdd(&a.stats->skipped, (unsigned long long)sk);
        }
        return;
    }
    c.n_first = m;
    if (warp == 0 && c.l == 0) sm.alive[c.t] = c.alive0 ? 1 : 0;
    if (threadIdx.x == 0) sm.last = -1;
    __syncthreads();
    const int role = (warp + (int)(g & 3)) & 3;
    if (role == 0) quad_dynamics<POT, FB>(f, tg, a, c, sm);
    else if (role == 1) quad_matrix<POT, FB>(f, tg, c, sm);
    else if (role == 2) quad_columns<POT, FB>(f, a, c, sm);
    else quad_bins<POT, FB>(f, tg, gt, a, c, sm);
}

// FB: recombination terms in float, as the float pass forms them (escalation lists)
template <int POT, bool FB>
__global__ void __launch_bounds__(kThreads, 3) quad_kernel(FieldDev f, TargetDev tg, GtoTerms gt, TrajArgs a) {
    __shared__ QShared sm;
    __shared__ long long s_g;
    const int64_t n_list = a.count ? (int64_t)*a.count : a.n;
    // an empty list (its blocks would otherwise look through every SM's list), or a long one,
    // which redo.cu takes
    if (a.count && (n_list == 0 || n_list > a.quad_limit)) return;
    GroupSource src(a, (n_list + kT - 1) / kT);
    for (;;) {
        const int64_t g = src.next(a, s_g);
        if (g < 0) break;
        quad_group<POT, FB>(f, tg, gt, a, g, n_list, sm);
        __syncthreads();   // every role has drained its hand-offs before the next group
    }
}

template <int POT>
cudaError_t launch_pot(const FieldDev& f, const TargetDev& t, const GtoTerms& gt, const TrajArgs& a, cudaStream_t s) {
    // with a plan: persistent, as many blocks as fit on every SM (3); without one: a block
    // per group
    const int64_t blocks = a.redo_ctr ? (int64_t)a.redo_lists * 3 : (a.n + kT - 1) / kT;
    if (a.float_bins) quad_kernel<POT, true><<<(unsigned)blocks, kThreads, 0, s>>>(f, t, gt, a);
    else quad_kernel<POT, false><<<(unsigned)blocks, kThreads, 0, s>>>(f, t, gt, a);
    return cudaGetLastError();
}

}  // namespace

cudaError_t launch_quad(const FieldDev& f, const TargetDev& t, const TrajArgs& a, cudaStream_t s) {
    const GtoTerms gt = make_gto_terms(t, a.gamma);
    switch (t.pot) {
        case POT_SOFTCORE: return launch_pot<POT_SOFTCORE>(f, t, gt, a, s);
        case POT_TONGLIN: return launch_pot<POT_TONGLIN>(f, t, gt, a, s);
        case POT_HARMONIC: return launch_pot<POT_HARMONIC>(f, t, gt, a, s);
        default: return launch_pot<POT_ZERO>(f, t, gt, a, s);
    }
}

}  // namespace sfhk
