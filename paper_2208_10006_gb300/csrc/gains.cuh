// Complex path gain g_n(f) of one path at one frequency (Eq. 1, 3, 6-10).
//
// Per reflection k:
//   eta = eps_r - j sigma / (2 pi f eps0)                         (lossy dielectric)
//   G_TE = (cos - sqrt(eta - sin^2)) / (cos + sqrt(eta - sin^2))
//   G_TM = (eta cos - sqrt(eta - sin^2)) / (eta cos + sqrt(eta - sin^2))
//   rho  = exp(-g/2), g = (4 pi sigma_h cos f / c)^2                (Eq. 6-8)
// applied to the field in the (s, p) basis of that reflection, followed by the
// real 2x2 change to the next reflection's basis; then the Rx projection, the
// Friis amplitude c / (4 pi f L) (Eq. 3), absorption 10^(-gamma L / 20000)
// (Eq. 9) and the dispersion phase -phi (pi/180) L / 1000 (Eq. 10).
//
// Computed in double-float: the co-polar projection of a multi-bounce field can
// cancel to 1e-5 of the field, so FP32 is too coarse, and an FP64 operation
// takes as long as 71 FP32 ones (1.68 against 120 lanes per clock and SM) where
// its double-float form takes 7 to 22. The real exponents (roughness of every
// reflection, absorption) are added up and exponentiated once. The gains are
// rounded to FP32: the error against 64 bits is that rounding (2.5e-8 in the
// 2-norm) in both forms. Inputs outside the FP32 range, where products of
// squares would leave it, take the FP64 form.
#pragma once
#include "dfloat.cuh"
#include "sbr_internal.cuh"

namespace sbr {
namespace {

struct cd {
    double re, im;
};
__device__ __forceinline__ cd cmul(cd a, cd b) { return cd{a.re * b.re - a.im * b.im, a.re * b.im + a.im * b.re}; }
__device__ __forceinline__ cd cadd(cd a, cd b) { return cd{a.re + b.re, a.im + b.im}; }
__device__ __forceinline__ cd csub(cd a, cd b) { return cd{a.re - b.re, a.im - b.im}; }
__device__ __forceinline__ cd cscale(cd a, double s) { return cd{a.re * s, a.im * s}; }
// a / b as a conj(b) / |b|^2: one FP64 division (FP64 is a narrow pipe on this
// GPU). The denominators here are cos + sqrt(eta - sin^2) and its TM form:
// |b|^2 stays far inside the FP64 range for any physical permittivity,
// conductivity and incidence angle.
__device__ __forceinline__ cd cdiv(cd a, cd b) {
    const double inv = 1.0 / (b.re * b.re + b.im * b.im);
    return cd{(a.re * b.re + a.im * b.im) * inv, (a.im * b.re - a.re * b.im) * inv};
}
// principal square root; the larger part is sqrt((|z| + |re|) / 2) and the
// other im / (2 that), so neither cancels
__device__ __forceinline__ cd csqrt_(cd z) {
    const double r = sqrt(z.re * z.re + z.im * z.im);
    if (r == 0.0) return cd{0.0, 0.0};
    const double u = sqrt(0.5 * (r + fabs(z.re)));
    const double v = 0.5 * fabs(z.im) / u;
    if (z.re >= 0.0) return cd{u, z.im < 0.0 ? -v : v};
    return cd{v, z.im < 0.0 ? -u : u};
}

// Fresnel coefficients (TE, TM) of reflection k and its roughness factor rho
// at frequency f; cosine of incidence c from the polarimetric record
struct Refl {
    cd te, tm;
    double rho;
};
__device__ __forceinline__ Refl reflection(const sbr_material& mt, double c, double f) {
    const double eps2_scale = 1.0 / (2.0 * kPi * f * kEps0);
    const double kr = 4.0 * kPi * f / kC0;
    double s2 = 1.0 - c * c;
    cd eta{mt.eps_r, -mt.sigma_s_per_m * eps2_scale};
    cd root = csqrt_(cd{eta.re - s2, eta.im});
    cd cc{c, 0.0};
    Refl r;
    r.te = cdiv(csub(cc, root), cadd(cc, root));
    cd ec = cscale(eta, c);
    r.tm = cdiv(csub(ec, root), cadd(ec, root));
    double gk = kr * mt.rough_m * c;
    r.rho = exp(-0.5 * gk * gk);
    return r;
}

// the field (b0, b1) through reflection k (coefficients rf), then the change to
// the next reflection's basis (k + 1 < m)
__device__ __forceinline__ void reflect_field(cd& b0, cd& b1, const Refl& rf, const double* __restrict__ J,
                                              int k, int m) {
    b0 = cscale(cmul(rf.te, b0), rf.rho);
    b1 = cscale(cmul(rf.tm, b1), rf.rho);
    if (k + 1 < m) {
        const double* M = J + 4 + 4 * k;
        cd n0 = cadd(cscale(b0, M[0]), cscale(b1, M[1]));
        cd n1 = cadd(cscale(b0, M[2]), cscale(b1, M[3]));
        b0 = n0;
        b1 = n1;
    }
}

// Rx projection, Friis amplitude, absorption and dispersion phase of the field
__device__ __forceinline__ float2 finish_gain(cd b0, cd b1, const double* __restrict__ J, int pb, double Lp,
                                              double f, const float* gamma, const float* disp) {
    const double* cv = J + 32 + pb;
    cd proj = cadd(cscale(b0, cv[0]), cscale(b1, cv[1]));
    double amp = kC0 / (4.0 * kPi * f * Lp);
    double att = gamma ? exp10(-(double)*gamma * Lp / 20000.0) : 1.0;
    double ph = disp ? -(double)*disp * (kPi / 180.0) * Lp / 1000.0 : 0.0;
    double sn, cs;
    sincos(ph, &sn, &cs);
    cd v = cmul(cscale(cd{cs, sn}, amp * att), proj);
    return make_float2((float)v.re, (float)v.im);
}

// the gain in FP64 (inputs beyond the range of the double-float form)
__device__ __noinline__ float2 path_gain_f64(int m, const int32_t* __restrict__ surf, double Lp,
                                            const double* __restrict__ J, const sbr_material* __restrict__ mats,
                                            int32_t S, double f, const float* gamma, const float* disp, int pol) {
    const int pb = pol == SBR_POL_V ? 0 : 2;
    cd b0{J[pb], 0.0}, b1{J[pb + 1], 0.0};
    for (int k = 0; k < m; ++k) {
        int s = surf[k];
        if (s < 0 || s >= S) return make_float2(NAN, NAN);  // not reachable: S is checked on the host
        reflect_field(b0, b1, reflection(mats[s], J[36 + k], f), J, k, m);
    }
    return finish_gain(b0, b1, J, pb, Lp, f, gamma, disp);
}

// complex double-float
struct cdf {
    df re, im;
};
__device__ __forceinline__ cdf cdf_mul(cdf a, cdf b) {
    return cdf{df_dot2(a.re, b.re, df_neg(a.im), b.im), df_dot2(a.re, b.im, a.im, b.re)};
}
__device__ __forceinline__ cdf cdf_inv(cdf a) {
    const df d = df_rcp(df_dot2(a.re, a.re, a.im, a.im));
    return cdf{df_mul(a.re, d), df_neg(df_mul(a.im, d))};
}
__device__ __forceinline__ df df_scale2(df a, float s) { return df{a.hi * s, a.lo * s}; }   // s a power of two

// e^x = m 2^n with m in [0.7, 1.42]: Cody-Waite reduction by ln 2 (double-float)
// and the Taylor series on |r| <= 0.35, through r^5 in double-float; the terms from
// r^6 on are below 3e-6 of the sum, so that FP32 carries them to 2^-42 of it.
// |x| beyond 400 saturates n.
__device__ __forceinline__ df df_exp_parts(df x, int& n) {
    const float xh = fminf(fmaxf(x.hi, -400.f), 400.f);
    const float k = rintf(__fmul_rn(xh, 1.44269504f));
    const df p = two_prod(k, 0.693147182f);               // ln 2 = 0.693147182 - 1.9046543e-9
    const float lo = xh == x.hi ? x.lo : 0.f;
    const df r = two_sum(__fsub_rn(xh, p.hi), __fadd_rn(__fsub_rn(lo, p.lo), __fmul_rn(k, 1.9046543e-9f)));
    float q = 1.f / 479001600.f;
    q = __fmaf_rn(q, r.hi, 1.f / 39916800.f);
    q = __fmaf_rn(q, r.hi, 1.f / 3628800.f);
    q = __fmaf_rn(q, r.hi, 1.f / 362880.f);
    q = __fmaf_rn(q, r.hi, 1.f / 40320.f);
    q = __fmaf_rn(q, r.hi, 1.f / 5040.f);
    q = __fmaf_rn(q, r.hi, 1.f / 720.f);
    constexpr double c5 = 1.0 / 120.0, c4 = 1.0 / 24.0, c3 = 1.0 / 6.0;
    df t = df_fma(df{(float)c5, (float)(c5 - (double)(float)c5)}, r, df{q, 0.f});
    t = df_fma(df{(float)c4, (float)(c4 - (double)(float)c4)}, r, t);
    t = df_fma(df{(float)c3, (float)(c3 - (double)(float)c3)}, r, t);
    t = df_fma(df{0.5f, 0.f}, r, t);
    n = (int)k;
    return df_add(df{1.f, 0.f}, df_fma(r, r, df_mul(r, t)));
}

// m reflections off surfaces surf[0..m), unfolded length Lp, polarimetric
// record J (kJones doubles); gamma / disp may be null (no absorption / phase)
__device__ __forceinline__ float2 path_gain(int m, const int32_t* __restrict__ surf, double Lp,
                                            const double* __restrict__ J, const sbr_material* __restrict__ mats,
                                            int32_t S, double f, const float* gamma, const float* disp, int pol) {
    const int pb = pol == SBR_POL_V ? 0 : 2;
    const df fd = df_split(f), Ld = df_split(Lp);
    // FP32 carries the squares below for f in [1, 1e18] Hz, L in [1e-9, 1e15] m, |eta| < 1e15,
    // |eta - sin^2| > 1e-15
    bool wide = !(fd.hi >= 1.f && fd.hi <= 1e18f && Ld.hi >= 1e-9f && Ld.hi <= 1e15f) ||
                (gamma && !(fabsf(*gamma) < 1e15f));
    const df fi = df_rcp(fd);
    constexpr double kEta = 1.0 / (2.0 * kPi * kEps0), kRough = 4.0 * kPi / kC0, kAmp = kC0 / (4.0 * kPi);
    const df kr = df_mul(fd, df{(float)kRough, (float)(kRough - (double)(float)kRough)});
    const df ef = df_mul(fi, df{(float)kEta, (float)(kEta - (double)(float)kEta)});
    cdf b0{df_split(J[pb]), df{0.f, 0.f}}, b1{df_split(J[pb + 1]), df{0.f, 0.f}};
    df x{0.f, 0.f};   // exponent of the roughness factors and of the absorption
    for (int k = 0; k < m && !wide; ++k) {
        const int s = surf[k];
        if (s < 0 || s >= S) return make_float2(NAN, NAN);  // not reachable: S is checked on the host
        const df c = df_split(J[36 + k]);
        const df er = df_split(mats[s].eps_r), ei = df_neg(df_mul(df_split(mats[s].sigma_s_per_m), ef));
        const df gk = df_mul(df_mul(kr, df_split(mats[s].rough_m)), c);
        wide = !(fabsf(er.hi) < 1e15f && fabsf(ei.hi) < 1e15f && fabsf(gk.hi) < 1e18f);
        x = df_sub(x, df_scale2(df_mul(gk, gk), 0.5f));
        // root = sqrt(eta - sin^2): the larger part from |z| + |Re z|, the other by division
        const df c2 = df_mul(c, c);
        const df zr = df_add(er, df_sub(c2, df{1.f, 0.f}));
        const df z2 = df_dot2(zr, zr, ei, ei);
        wide |= !(z2.hi >= 1e-30f);   // |z| < 1e-15: grazing incidence on eta = 1
        const df r = df_sqrt(z2);
        const bool neg = zr.hi < 0.f;
        const df u = df_sqrt(df_scale2(df_add(r, neg ? df_neg(zr) : zr), 0.5f));
        const df v = df_mul(df_scale2(ei, 0.5f), df_rcp(u));   // signed as Im z
        const df um = ei.hi < 0.f ? df_neg(u) : u;
        const df ur = neg ? (v.hi < 0.f ? df_neg(v) : v) : u, ui = neg ? um : v;
        // (a - root) / (a + root) = (a^2 - root^2) / (a + root)^2 with the numerator in
        // factors free of cancellation: 1 - eta for a = cos (TE), (eta - 1)(cos^2 (1 + eta) - 1)
        // for a = eta cos (TM)
        const df one{1.f, 0.f};
        const cdf et{df_sub(er, one), ei};
        const cdf te_w = cdf_inv(cdf{df_add(c, ur), ui});
        const cdf te = cdf_mul(cdf_mul(cdf{df_neg(et.re), df_neg(ei)}, te_w), te_w);
        const cdf tm_w = cdf_inv(cdf{df_add(df_mul(er, c), ur), df_add(df_mul(ei, c), ui)});
        const cdf brewster{df_sub(df_mul(c2, df_add(er, one)), one), df_mul(c2, ei)};
        const cdf tm = cdf_mul(cdf_mul(et, tm_w), cdf_mul(brewster, tm_w));
        b0 = cdf_mul(te, b0);
        b1 = cdf_mul(tm, b1);
        if (k + 1 < m) {   // to the basis of the next reflection
            const double* M = J + 4 + 4 * k;
            const df m0 = df_split(M[0]), m1 = df_split(M[1]), m2 = df_split(M[2]), m3 = df_split(M[3]);
            const cdf n0{df_dot2(b0.re, m0, b1.re, m1), df_dot2(b0.im, m0, b1.im, m1)};
            b1 = cdf{df_dot2(b0.re, m2, b1.re, m3), df_dot2(b0.im, m2, b1.im, m3)};
            b0 = n0;
        }
    }
    if (wide) return path_gain_f64(m, surf, Lp, J, mats, S, f, gamma, disp, pol);
    const df c0 = df_split(J[32 + pb]), c1 = df_split(J[33 + pb]);
    cdf v{df_dot2(b0.re, c0, b1.re, c1), df_dot2(b0.im, c0, b1.im, c1)};   // Rx projection
    if (gamma) {
        constexpr double kAtt = -2.302585092994045684 / 20000.0;   // ln 10 / 20000
        x = df_add(x, df_mul(df_mul_f(Ld, *gamma), df{(float)kAtt, (float)(kAtt - (double)(float)kAtt)}));
    }
    if (disp) {   // FP64: an unreduced phase of any size
        double sn, cs;
        sincos(-(double)*disp * (kPi / 180.0) * Lp / 1000.0, &sn, &cs);
        v = cdf_mul(cdf{df_split(cs), df_split(sn)}, v);
    }
    int n;
    df a = df_exp_parts(x, n);
    a = df_mul(a, df_mul(df_mul(fi, df_rcp(Ld)), df{(float)kAmp, (float)(kAmp - (double)(float)kAmp)}));
    return make_float2(ldexpf(df_mul(v.re, a).hi, n), ldexpf(df_mul(v.im, a).hi, n));
}

}  // namespace
}  // namespace sbr
