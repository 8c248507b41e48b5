// SFA births on the GPU (App. A, Eq. SAPeq / Eq. SFAwf / Eq. Int / Eq. SFHKwf;
// App. B.1 tunnelling matrix elements; App. B.2 modified SPA; Sec. III.C ADK
// births renormalised to the SFA rate at the pulse's two sub-peaks).
//
// FP64, a thread for each birth's draw and bracket and for its amplitude, the roots in
// between from a queue.  The birth draws (grid or Philox) are integer
// exact; the saddle point is the smallest t_t > 0 with
// Im A(t0 + i t_t) = s kappa, s = -sign E(t0), found by a scan for the first grid
// cell with a sign change, then a Newton iteration kept inside the bracket
// (bisection whenever a step would leave it).
//
// Bound by FP64 instructions (64 cycles of a sub-partition each on GB300).  The scan
// (up to 1250 points; births in a weak field go to the end) only needs signs, so it runs
// in float with an error bound, 16 points at a time, skipping a run that a slope bound
// shows to be free of roots; a point whose sign the bound leaves open is evaluated in
// FP64.  Per-target constants and the sines and cosines at a birth's time are formed
// once.  The Newton iteration takes 4 steps for half of the births and up to 48 where it
// ends in bisection, so the lanes of a block take their problems from a queue over its
// births (4 per thread in a large call) instead of waiting for the slowest of 32.
// Measured at 1e6 births (H, 800 nm, 8 cycles): 30.0 ms with the scan in FP64, 9.2 ms
// with the scan in float, 6.0 ms with the queue.
#include "sfhk_device.cuh"

namespace sfhk {
namespace {

// Constants of a launch that every thread would form the same way, made once per block.
struct BirthConst {
    double gk[kMaxGto], gc[kMaxGto];         // -1/(4 a_j); prefactor of term j of the tunnelling element
    FieldConst fc;
    double part[128];                        // the ADK renormalisation's partial sums
};
__device__ void make_const(const FieldDev& f, const TargetDev& t, BirthConst& bc) {
    const double pi32 = 5.5683279968317078;          // pi^{3/2}
    for (int j = threadIdx.x; j < t.n_gto; j += blockDim.x) {
        const double a = t.alpha[j];
        bc.gk[j] = -0.25 / a;
        bc.gc[j] = t.gto_l == 0 ? t.c[j] * 0.5 * pi32 / (a * a * sqrt(a)) : t.c[j] * 0.25 * pi32 / (a * a * a * sqrt(a));
    }
    make_field_const(f, bc.fc);
    __syncthreads();
}

// Tunnelling element m(k) = (2pi)^{-3/2} int e^{-i k.r} z psi0 d^3r for complex k
// (GTO closed forms: s: -i pi^{3/2}/2 k_z a^{-5/2} e^{-k^2/4a};
//                    p: pi^{3/2}/4 a^{-7/2} (2a - k_z^2) e^{-k^2/4a}).
__device__ cd tunnel_element(const TargetDev& t, const BirthConst& bc, cd kx, cd ky, cd kz) {
    cd k2 = kx * kx + ky * ky + kz * kz;
    const double pw = 0.063493635934240969;          // (2 pi)^{-3/2}
    cd s = mk(0, 0);
    for (int j = 0; j < t.n_gto; ++j) {
        double a = t.alpha[j];
        cd g = c_exp(bc.gk[j] * k2);
        if (t.gto_l == 0) s = s + bc.gc[j] * (kz * g);
        else s = s + bc.gc[j] * ((mk(2.0 * a, 0) - kz * kz) * g);
    }
    if (t.gto_l == 0) s = mk(0, -1) * s;   // factor -i of the s-type element
    return pw * s;
}

// The saddle's equation f(tau) = sum_j c_j sinh(w_j tau) - target, c_j = a_j cos(w_j t0 +
// cep) (cs[j]: the cosines): the grid cell [(hit - 1) h, hit h] of its smallest root on
// (0, 25/w_max], h = 0.02/w_max; 0 when there is none.
__device__ __forceinline__ double scan_step(const FieldDev& f) {
    double wmax = 0.0;
    for (int j = 0; j < f.n_modes; ++j) wmax = fmax(wmax, fabs(f.w[j]));
    return wmax == 0.0 ? 0.0 : 0.02 / wmax;
}
__device__ int scan_root(const FieldDev& f, const double* cs, double target) {
    double c[3], w[3];
    double wmax = 0.0;
    for (int j = 0; j < f.n_modes; ++j) {
        c[j] = f.a[j] * cs[j];
        w[j] = f.w[j];
        wmax = fmax(wmax, fabs(w[j]));
    }
    if (wmax == 0.0) return 0;
    const double h = 0.02 / wmax, tmax = 25.0 / wmax;
    const int nscan = (int)(tmax / h);
    // The first grid point it h at which f has left the sign of f(0) = -target.  Float
    // values of e^{w tau}: a run's start from expf of a float argument of at most 25 (two
    // roundings: 3e-6), then up to 16 products with a factor good to 1e-7 (2.6e-6): below
    // 6e-6 in all, so 1e-5 of the terms' sizes at the run's end bounds the error of f at
    // every point.  (A negative w enters as -c sinh(-w tau).)
    const bool up0 = -target > 0.0;
    const float tf = (float)target;
    float cf[3], wh[3], q[3], iq[3], e0[3], e1[3];
#pragma unroll
    for (int j = 0; j < 3; ++j) {
        const bool on = j < f.n_modes;
        const bool neg = on && w[j] < 0.0;
        cf[j] = on ? 0.5f * (float)(neg ? -c[j] : c[j]) : 0.f;
        wh[j] = on ? (float)(fabs(w[j]) * h) : 0.f;
        q[j] = expf(wh[j]);
        iq[j] = expf(-wh[j]);
        e1[j] = 1.f;
    }
    constexpr int kRun = 16;
    int hit = 0;
    for (int b = 0; b < nscan && !hit; b += kRun) {
        float v = -tf, size = 0.f, slope = 0.f, ie[3];
#pragma unroll
        for (int j = 0; j < 3; ++j) {
            e0[j] = e1[j];
            ie[j] = __frcp_rn(e0[j]);
            e1[j] = expf((float)(b + kRun) * wh[j]);
            v = fmaf(cf[j], e0[j] - ie[j], v);
            const float ch = fabsf(cf[j]) * (e1[j] + 1.f);   // |c_j| cosh or more, up to the run's end
            size += ch;
            slope = fmaf(wh[j], ch, slope);
        }
        const float err = fmaf(1e-5f, size, 1e-6f * fabsf(tf));
        if (fabsf(v) > fmaf((float)kRun, slope, err)) continue;   // no sign change up to the run's end
        const int last = nscan - b < kRun ? nscan - b : kRun;
        for (int i = 1; i <= last; ++i) {
            v = -tf;
#pragma unroll
            for (int j = 0; j < 3; ++j) {
                e0[j] *= q[j];
                ie[j] *= iq[j];
                v = fmaf(cf[j], e0[j] - ie[j], v);
            }
            bool up = v > 0.f;
            if (!(fabsf(v) > err)) {
                const double tau = (b + i) * h;
                double d = -target;
                for (int j = 0; j < f.n_modes; ++j) d += c[j] * sinh(w[j] * tau);
                up = d > 0.0;
            }
            if (up != up0) {
                hit = b + i;
                break;
            }
        }
    }
    return hit;
}

// The root in that cell: safeguarded Newton inside the bracket (bisection when a step
// leaves it), one step at a time.
struct Newton {
    double c[3], target, lo, hi, x;
    int it;
    __device__ __forceinline__ void start(const FieldDev& f, const double cs[3], double goal, int hit, double h) {
#pragma unroll
        for (int j = 0; j < 3; ++j) c[j] = j < f.n_modes ? f.a[j] * cs[j] : 0.0;
        target = goal;
        const double tau = hit * h;
        lo = tau - h;
        hi = tau;
        x = 0.5 * (lo + hi);
        it = 0;
    }
    // true when done: the root is x
    __device__ __forceinline__ bool step(const FieldDev& f) {
        double v = -target, d = 0.0;
#pragma unroll
        for (int j = 0; j < 3; ++j) {
            if (j >= f.n_modes) break;
            const double e = exp(f.w[j] * x), ie = 1.0 / e;
            v += c[j] * 0.5 * (e - ie);            // sinh
            d += c[j] * f.w[j] * 0.5 * (e + ie);   // derivative: w cosh
        }
        if ((v > 0) == (-target > 0.0)) lo = x; else hi = x;   // f has the sign of f(0) at lo
        double xn = (d != 0.0) ? x - v / d : 0.5 * (lo + hi);
        if (!(xn > lo && xn < hi)) xn = 0.5 * (lo + hi);
        const bool done = fabs(xn - x) <= 1e-15 * fabs(xn) || hi - lo <= 1e-15 * hi;
        x = xn;
        return done || ++it == 100;
    }
};

// ADK rate per unit time (Z_c = 1, m = 0, l = gto_l; the tail constant C_l^2 left out):
//   w(F) = (2l+1)/2 kappa^{1-2/kappa} (2 kappa^3/F)^{2/kappa-1} exp(-2 kappa^3/(3F)),
// and per d^2 k_perp: rho = w(F) (kappa/(pi F)) exp(-kappa k_perp^2/F).
__device__ double adk_rate(const TargetDev& t, double F) {
    if (!(F > 0.0)) return 0.0;
    const double kappa = sqrt(2.0 * t.ip), k3 = kappa * kappa * kappa;
    return 0.5 * (2.0 * t.gto_l + 1.0) * pow(kappa, 1.0 - 2.0 / kappa) * pow(2.0 * k3 / F, 2.0 / kappa - 1.0) *
           exp(-2.0 * k3 / (3.0 * F));
}
__device__ double adk_density(const TargetDev& t, double F, double kperp2) {
    if (!(F > 0.0)) return 0.0;
    const double kappa = sqrt(2.0 * t.ip);
    return adk_rate(t, F) * kappa / (kPi * F) * exp(-kappa * kperp2 / F);
}

// A birth at (t0, kx, ky) with the mode phases sn0, cs0: its side of the saddle's equation
// (0 where the field vanishes and there is no saddle).
__device__ __forceinline__ double saddle_target(const FieldDev& f, const TargetDev& t, const double cs0[3], double kx,
                                                double ky) {
    double Et0 = 0.0;
    for (int j = 0; j < f.n_modes; ++j) Et0 = Et0 + (-f.a[j] * f.w[j]) * cs0[j];
    if (Et0 == 0.0) return 0.0;
    const double kp2 = kx * kx + ky * ky;
    const double kappa = sqrt(2.0 * t.ip + kp2);
    const double s = Et0 > 0 ? -1.0 : 1.0;
    return s * kappa;
}

// The saddle of a birth at t0 + i tt and its amplitude without the Monte Carlo measure:
// kind 0 standard SPA, 1 modified SPA, 2 ADK (modulus sqrt(adk_n2 rho), phase Re S, exit
// q0 = -Ip/E(t0), kz = 0).
__device__ void birth_amp(const FieldDev& f, const TargetDev& t, const BirthConst& bc, double t0, double tt,
                          const double sn0[3], const double cs0[3], double kx, double ky, int kind, double adk_n2,
                          double* kz_out, double* qz_out, cd* amp_out) {
    const FieldAt0 at0 = field_at_real(f, t0, sn0, cs0, bc.fc);
    const double Et0 = at0.E;
    const double kp2 = kx * kx + ky * ky;
    const cd ts = mk(t0, tt);
    const FieldAt ats = field_at(f, ts, sn0, cs0, bc.fc);
    const double A0 = at0.A;
    const cd Ats = ats.A;
    double kz = A0 - Ats.re;
    const cd F0 = mk(at0.F, 0.0), Fs = ats.F;
    double qz = (F0 - Fs).re;
    const double cc = kz - A0;
    const cd G0 = mk(at0.G, 0.0), Gs = ats.G;
    // int_{ts}^{t0} v^2/2 with v = k + A - A(t0): constant, linear and quadratic parts
    const cd dt0 = mk(0.0, -tt);  // t0 - ts
    cd integ = 0.5 * ((kp2 + cc * cc) * dt0 + 2.0 * cc * (F0 - Fs) + (G0 - Gs));
    const cd S = t.ip * ts - integ;
    cd amp;
    if (kind == 2) {
        // ADK (Sec. III.C): quasi-static exit, ADK modulus, the saddle's real action
        kz = 0.0;
        qz = -t.ip / Et0;
        amp = sqrt(adk_n2 * adk_density(t, fabs(Et0), kp2)) * c_exp(mk(0.0, S.re));
    } else {
        const cd vz = mk(kz - A0, 0.0) + Ats;
        const cd Ets = ats.E;
        const cd EdotV = Ets * vz;
        const cd ph = c_exp(mk(-S.im, S.re + kz * qz));   // e^{i(S + p0.q0)}
        if (kind == 0) {
            cd m = tunnel_element(t, bc, mk(kx, 0), mk(ky, 0), vz);
            amp = cdiv(Ets * m, c_sqrt(EdotV)) * ph;
        } else {
            amp = cdiv(ph, EdotV);
        }
    }
    if (!isfinite(amp.re) || !isfinite(amp.im)) amp = mk(0, 0);
    *kz_out = kz;
    *qz_out = qz;
    *amp_out = amp;
}

// ADK renormalisation N^2 (Sec. III.C), evaluated by every block of 128 threads
// (the same sum in the same order, so every block gets the same value): the SFA
// rate over the ADK rate summed over the two sub-peaks t_j = ((k* + j) pi - phi)/w,
// j = -1, +1, k* = floor(phi/pi + 1/2); the SFA rate by composite Simpson over
// k_perp in [0, 6 sqrt(F/kappa)], 128 intervals: thread (j, m) takes the nodes
// i = 2m + 1 and 2m + 2 of sub-peak j.
__device__ double adk_norm2_block(const FieldDev& f, const TargetDev& t, BirthConst& bc) {
    double* const s_part = bc.part;
    const int tid = threadIdx.x, j = tid >> 6, m = tid & 63;
    const double ks = floor(f.cep / kPi + 0.5);
    const double tj = ((ks + (j == 0 ? -1.0 : 1.0)) * kPi - f.cep) / f.omega;
    const double F = fabs(field_E(f, mk(tj, 0)).re);
    const double kappa = sqrt(2.0 * t.ip);
    const double h = 6.0 * sqrt(F / kappa) / 128.0;
    double part = 0.0;
    if (F > 0.0) {
        for (int q = 0; q < 2; ++q) {
            const int i = 2 * m + 1 + q;
            const double k = (double)i * h;
            const double c = (i == 128) ? 1.0 : ((i & 1) ? 4.0 : 2.0);
            double sn[3], cs[3], kz, qz;
            mode_phases(f, tj, sn, cs);
            const double goal = saddle_target(f, t, cs, k, 0.0);
            const int hit = goal != 0.0 ? scan_root(f, cs, goal) : 0;
            if (hit == 0) continue;
            Newton nw;
            nw.start(f, cs, goal, hit, scan_step(f));
            while (!nw.step(f)) {
            }
            cd a;
            birth_amp(f, t, bc, tj, nw.x, sn, cs, k, 0.0, 0, 0.0, &kz, &qz, &a);
            part += c * k * (a.re * a.re + a.im * a.im);
        }
    }
    s_part[tid] = part;
    __syncthreads();
    double num = 0.0, den = 0.0;
    for (int jj = 0; jj < 2; ++jj) {
        const double tq = ((ks + (jj == 0 ? -1.0 : 1.0)) * kPi - f.cep) / f.omega;
        const double Fq = fabs(field_E(f, mk(tq, 0)).re);
        if (!(Fq > 0.0)) continue;
        double R = 0.0;
        for (int q = 0; q < 64; ++q) R += s_part[64 * jj + q];
        num += 2.0 * kPi * ((6.0 * sqrt(Fq / kappa) / 128.0) / 3.0) * R;
        den += adk_rate(t, Fq);
    }
    const double n2 = num / den;
    return (den > 0.0 && isfinite(n2)) ? n2 : 0.0;
}

// The draws of birth o of the produced range (output index): its step and transverse
// momentum, and its Monte Carlo measure.
__device__ void draw_birth(const FieldDev& f, const BirthArgs& a, int64_t o, int64_t& nb, double& kx, double& ky,
                           double& w) {
    const int64_t i = a.first + o;                                       // birth index
    const int64_t M = f.n_steps - 1;
    if (a.mode == 0) {
        int64_t it = i / a.n_k, ik = i % a.n_k;
        nb = (int64_t)floor(((double)it + 0.5) * (double)f.n_steps / (double)a.n_t);
        nb = nb < 1 ? 1 : (nb > M ? M : nb);
        double dk = a.kmax / a.n_k;
        kx = ((double)ik + 0.5) * dk;
        ky = 0.0;
        w = 2.0 * kPi * kx * dk * ((double)f.n_steps * f.dt / (double)a.n_t);
    } else {
        uint64_t x[4] = {(uint64_t)i, 0, 0, 0};
        philox4x64_10(x, a.seed, 0);
        unsigned __int128 num = (((unsigned __int128)(uint64_t)i) << 32) + (unsigned __int128)(x[0] >> 32);
        num *= (unsigned __int128)(uint64_t)M;
        unsigned __int128 den = ((unsigned __int128)(uint64_t)a.n) << 32;
        nb = 1 + (int64_t)(num / den);
        double u1 = (double)((x[1] >> 11) + 1) * 0x1.0p-53;
        double u2 = (double)(x[2] >> 11) * 0x1.0p-53;
        double rad = a.sigma * sqrt(-2.0 * log(u1));
        double sn, cs;
        sincospi(2.0 * u2, &sn, &cs);
        kx = rad * cs;
        ky = rad * sn;
        double s2 = a.sigma * a.sigma;
        // w = 1/(n pdf),  pdf = e^{-k^2/2s^2}/(2 pi s^2) * 1/(M dt)
        w = 2.0 * kPi * s2 * exp((kx * kx + ky * ky) / (2.0 * s2)) * ((double)M * f.dt) / (double)a.n;
    }
}

constexpr int kThreads = 128;   // the ADK renormalisation spreads its 2 x 64 Simpson pairs over 128 threads

// R births per thread and tile, between the draws and the amplitudes in shared memory
template <int R>
struct BirthTile {
    double sn[3][R * kThreads], cs[3][R * kThreads];
    double root[R * kThreads];   // the equation's target, then its root
    double w[R * kThreads];
    int hit[R * kThreads];
    int next;
};

template <int R>
__global__ void __launch_bounds__(kThreads, 2) births_kernel(FieldDev f, TargetDev t, BirthArgs a) {
    __shared__ BirthConst bc;
    __shared__ BirthTile<R> tl;
    make_const(f, t, bc);
    const double adk_n2 = t.amp == 2 ? adk_norm2_block(f, t, bc) : 0.0;   // every thread takes part
    const double h = scan_step(f);
    constexpr int kTile = R * kThreads;
    for (int64_t o0 = (int64_t)blockIdx.x * kTile; o0 < a.count; o0 += (int64_t)gridDim.x * kTile) {
        const int nt = (int)(a.count - o0 < kTile ? a.count - o0 : kTile);
        // draws and brackets
        for (int u = threadIdx.x; u < nt; u += kThreads) {
            const int64_t o = o0 + u;
            int64_t nb;
            double kx, ky, w, sn[3], cs[3];
            draw_birth(f, a, o, nb, kx, ky, w);
            const double t0 = f.t_start + (double)nb * f.dt;
            mode_phases(f, t0, sn, cs);
            const double goal = saddle_target(f, t, cs, kx, ky);
            tl.hit[u] = goal != 0.0 ? scan_root(f, cs, goal) : 0;
            tl.root[u] = goal;
            tl.w[u] = w;
            for (int j = 0; j < f.n_modes; ++j) {
                tl.sn[j][u] = sn[j];
                tl.cs[j][u] = cs[j];
            }
            a.n0[o] = (int32_t)nb;
            a.t0[o] = t0;
            a.px[o] = kx;
            a.py[o] = ky;
        }
        if (threadIdx.x == 0) tl.next = 0;
        __syncthreads();
        // roots: every lane iterates on one birth and then takes the next
        {
            Newton nw;
            int u = -1;
            for (;;) {
                while (u < 0) {
                    u = atomicAdd(&tl.next, 1);
                    if (u >= nt) break;
                    if (tl.hit[u] == 0) {
                        u = -1;
                        continue;
                    }
                    const double cs[3] = {tl.cs[0][u], tl.cs[1][u], tl.cs[2][u]};
                    nw.start(f, cs, tl.root[u], tl.hit[u], h);
                }
                if (u >= nt) break;
                if (nw.step(f)) {
                    tl.root[u] = nw.x;
                    u = -1;
                }
            }
        }
        __syncthreads();
        // amplitudes
        for (int u = threadIdx.x; u < nt; u += kThreads) {
            const int64_t o = o0 + u;
            double kz = 0.0, qz = 0.0;
            cd amp = mk(0, 0);
            if (tl.hit[u]) {
                double sn[3], cs[3];
                for (int j = 0; j < f.n_modes; ++j) {
                    sn[j] = tl.sn[j][u];
                    cs[j] = tl.cs[j][u];
                }
                birth_amp(f, t, bc, a.t0[o], tl.root[u], sn, cs, a.px[o], a.py[o], t.amp, adk_n2, &kz, &qz, &amp);
            }
            const double w = tl.w[u];
            a.pz[o] = kz;
            a.qz[o] = qz;
            a.amp_re[o] = w * amp.re;
            a.amp_im[o] = w * amp.im;
        }
        __syncthreads();   // the tile is free
    }
}

}  // namespace

cudaError_t launch_births(const FieldDev& f, const TargetDev& t, const BirthArgs& a, cudaStream_t s) {
    if (a.count == 0) return cudaSuccess;
    // four births per thread where that still fills the chip (2 blocks on each of 152 SMs);
    // ADK: every block evaluates the renormalisation (two births a thread), so no more
    // blocks than are resident at once, each on several tiles
    const bool large = a.count >= (int64_t)4 * kThreads * 304;
    const int64_t tile = large ? 4 * kThreads : kThreads;
    int64_t grid = (a.count + tile - 1) / tile;
    if (t.amp == 2 && grid > 304) grid = 304;
    if (large) births_kernel<4><<<(unsigned)grid, kThreads, 0, s>>>(f, t, a);
    else births_kernel<1><<<(unsigned)grid, kThreads, 0, s>>>(f, t, a);
    return cudaGetLastError();
}

}  // namespace sfhk
