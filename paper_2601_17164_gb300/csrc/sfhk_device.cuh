// Device helpers of the SFHK library: complex double arithmetic, the
// Philox4x64-10 counter-based generator, and the analytic laser field for
// complex times.
#pragma once

#include <cuda_runtime.h>
#include <stdint.h>

#include "sfhk_internal.cuh"

namespace sfhk {

struct cd {
    double re, im;
};
__device__ __forceinline__ cd mk(double r, double i) { return cd{r, i}; }
__device__ __forceinline__ cd operator+(cd a, cd b) { return cd{a.re + b.re, a.im + b.im}; }
__device__ __forceinline__ cd operator-(cd a, cd b) { return cd{a.re - b.re, a.im - b.im}; }
__device__ __forceinline__ cd operator-(cd a) { return cd{-a.re, -a.im}; }
__device__ __forceinline__ cd operator*(cd a, cd b) {
    return cd{a.re * b.re - a.im * b.im, a.re * b.im + a.im * b.re};
}
__device__ __forceinline__ cd operator*(double s, cd a) { return cd{s * a.re, s * a.im}; }
__device__ __forceinline__ cd cdiv(cd a, cd b) {
    double d = b.re * b.re + b.im * b.im;
    return cd{(a.re * b.re + a.im * b.im) / d, (a.im * b.re - a.re * b.im) / d};
}
__device__ __forceinline__ cd c_exp(cd z) {
    double s, c;
    sincos(z.im, &s, &c);
    double e = exp(z.re);
    return cd{e * c, e * s};
}
// cos(x + i y) = cos x cosh y - i sin x sinh y
__device__ __forceinline__ cd c_cos(cd z) {
    double s, c;
    sincos(z.re, &s, &c);
    return cd{c * cosh(z.im), -s * sinh(z.im)};
}
// principal square root
__device__ __forceinline__ cd c_sqrt(cd z) {
    double r = hypot(z.re, z.im);
    if (r == 0.0) return cd{0.0, 0.0};
    if (z.re >= 0.0) {
        double t = sqrt(0.5 * (r + z.re));
        return cd{t, z.im / (2.0 * t)};
    }
    double t = sqrt(0.5 * (r - z.re));
    return cd{fabs(z.im) / (2.0 * t), copysign(t, z.im)};
}

// ---- Philox4x64-10 (Salmon et al., SC'11) ----------------------------------
__device__ __forceinline__ void philox4x64_10(uint64_t c[4], uint64_t k0, uint64_t k1) {
    const uint64_t M0 = 0xD2E7470EE14C6C93ULL, M1 = 0xCA5A826395121157ULL;
    const uint64_t W0 = 0x9E3779B97F4A7C15ULL, W1 = 0xBB67AE8584CAA73BULL;
#pragma unroll
    for (int r = 0; r < 10; ++r) {
        uint64_t lo0 = M0 * c[0], hi0 = __umul64hi(M0, c[0]);
        uint64_t lo1 = M1 * c[2], hi1 = __umul64hi(M1, c[2]);
        uint64_t n0 = hi1 ^ c[1] ^ k0, n2 = hi0 ^ c[3] ^ k1;
        c[0] = n0;
        c[1] = lo1;
        c[2] = n2;
        c[3] = lo0;
        k0 += W0;
        k1 += W1;
    }
}

// ---- analytic field on complex time ----------------------------------------
// A(t) = sum_j a_j sin(w_j t + cep), E = -dA/dt, F = int_0^t A, G = int_0^t A^2.
__device__ __forceinline__ cd field_E(const FieldDev& f, cd t) {
    cd s = mk(0, 0);
    for (int j = 0; j < f.n_modes; ++j)
        s = s + (-f.a[j] * f.w[j]) * c_cos(mk(f.w[j] * t.re + f.cep, f.w[j] * t.im));
    return s;
}
// All four at one time from the sines and cosines of the mode phases
// a_j = w_j t + cep, each computed once: A and E are sums over them, F a sum over
// the cosines, and G's terms sin((w_j -+ w_k) t + ...) = sin(a_j -+ a_k) follow by
// the angle-sum identities (no further transcendental calls).
struct FieldAt {
    cd A, E, F, G;
};
// The field's constants that every evaluation at a time would form the same way: sines and
// cosines of cep and 2 cep, a_j/w_j and 1/(w_j -+ w_k) (0 where the divisor is below 1e-14).
struct FieldConst {
    double s_cep, c_cep, s_2cep, c_2cep;
    double aw[3], im[3][3], ip[3][3];
};
// by the threads of a block (64 or more); the caller synchronises
__device__ __forceinline__ void make_field_const(const FieldDev& f, FieldConst& c) {
    const int v = threadIdx.x;
    if (v == 0) sincos(f.cep, &c.s_cep, &c.c_cep);
    if (v == 32) sincos(2.0 * f.cep, &c.s_2cep, &c.c_2cep);
    if (v < 9) {
        const int j = v / 3, k = v % 3;
        const double wm = f.w[j] - f.w[k], wp = f.w[j] + f.w[k];
        c.im[j][k] = fabs(wm) < 1e-14 ? 0.0 : 1.0 / wm;
        c.ip[j][k] = fabs(wp) < 1e-14 ? 0.0 : 1.0 / wp;
        if (k == 0) c.aw[j] = fabs(f.w[j]) < 1e-14 ? 0.0 : f.a[j] / f.w[j];
    }
}
// sine and cosine of the mode phases w_j t + cep at a real time
__device__ __forceinline__ void mode_phases(const FieldDev& f, double t, double sn[3], double cs[3]) {
    const int nm = f.n_modes < 3 ? f.n_modes : 3;
    for (int j = 0; j < nm; ++j) sincos(f.w[j] * t + f.cep, &sn[j], &cs[j]);
}
// at a complex t, whose real part has the mode phases sn, cs
__device__ __forceinline__ FieldAt field_at(const FieldDev& f, cd t, const double sn[3], const double cs[3],
                                            const FieldConst& fc) {
    cd s[3], c[3];
    const int nm = f.n_modes < 3 ? f.n_modes : 3;
    FieldAt r{mk(0, 0), mk(0, 0), mk(0, 0), mk(0, 0)};
    for (int j = 0; j < nm; ++j) {
        const double y = f.w[j] * t.im, ch = cosh(y), sh = sinh(y);
        s[j] = mk(sn[j] * ch, cs[j] * sh);     // sin(x + i y)
        c[j] = mk(cs[j] * ch, -sn[j] * sh);    // cos(x + i y)
    }
    for (int j = 0; j < nm; ++j) {
        const double a = f.a[j], w = f.w[j];
        r.A = r.A + a * s[j];
        r.E = r.E + (-a * w) * c[j];
        if (fc.aw[j] == 0.0) r.F = r.F + (a * fc.s_cep) * t;
        else r.F = r.F + fc.aw[j] * (mk(fc.c_cep, 0.0) - c[j]);
    }
    for (int j = 0; j < nm; ++j)
        for (int k = 0; k < nm; ++k) {
            const double cf = 0.5 * f.a[j] * f.a[k];
            const cd sc = s[j] * c[k], cc = c[j] * s[k];
            const cd im = fc.im[j][k] == 0.0 ? t : fc.im[j][k] * (sc - cc);                              // int cos(wm s) ds
            const cd ip = fc.ip[j][k] == 0.0 ? fc.c_2cep * t : fc.ip[j][k] * ((sc + cc) - mk(fc.s_2cep, 0.0));  // int cos(wp s + 2 cep)
            r.G = r.G + cf * (im - ip);
        }
    return r;
}
// the same at a real t: the real parts by the same operations (the imaginary ones are 0)
struct FieldAt0 {
    double A, E, F, G;
};
__device__ __forceinline__ FieldAt0 field_at_real(const FieldDev& f, double t, const double s[3], const double c[3],
                                                  const FieldConst& fc) {
    const int nm = f.n_modes < 3 ? f.n_modes : 3;
    FieldAt0 r{0.0, 0.0, 0.0, 0.0};
    for (int j = 0; j < nm; ++j) {
        const double a = f.a[j], w = f.w[j];
        r.A = r.A + a * s[j];
        r.E = r.E + (-a * w) * c[j];
        if (fc.aw[j] == 0.0) r.F = r.F + (a * fc.s_cep) * t;
        else r.F = r.F + fc.aw[j] * (fc.c_cep - c[j]);
    }
    for (int j = 0; j < nm; ++j)
        for (int k = 0; k < nm; ++k) {
            const double cf = 0.5 * f.a[j] * f.a[k];
            const double sc = __dmul_rn(s[j], c[k]), cc = __dmul_rn(c[j], s[k]);
            const double im = fc.im[j][k] == 0.0 ? t : fc.im[j][k] * (sc - cc);
            const double ip = fc.ip[j][k] == 0.0 ? fc.c_2cep * t : fc.ip[j][k] * ((sc + cc) - fc.s_2cep);
            r.G = r.G + cf * (im - ip);
        }
    return r;
}

// sr + i si += sum over u < n of y[u] e^{i w t_{k0 + u}}, t_k = t0 + k dt, by a rotation per
// bin (rc + i rs = e^{i w dt}) that an exact sincos re-anchors every 64 bins: the sum of the
// transforms' short forms (spectrum.cu, gabor.cu)
__device__ __forceinline__ void direct_sum(const double* y, int n, double w, double t0, double dt, int64_t k0,
                                           double rc, double rs, double& sr, double& si) {
    double er = 0.0, ei = 0.0;
    for (int u = 0; u < n; ++u) {
        if ((u & 63) == 0) sincos(w * (t0 + (double)(k0 + u) * dt), &ei, &er);
        const double v = y[u];
        sr = fma(v, er, sr);
        si = fma(v, ei, si);
        const double nr = fma(er, rc, -ei * rs);
        ei = fma(er, rs, ei * rc);
        er = nr;
    }
}

}  // namespace sfhk
