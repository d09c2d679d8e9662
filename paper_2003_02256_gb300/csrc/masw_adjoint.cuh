// masw_adjoint.cuh -- derivatives of the element stiffness's quadratic form for
// the null-vector adjoint of the refined root.
//
// At a simple root C* of det K(c; theta) = 0, Jacobi's formula with the
// rank-one adjugate adj K = kappa u u^T (u the null vector of the symmetric K)
// gives the implicit-function derivative
//   dC*/dtheta = - (u^T dK/dtheta u) / (u^T dK/dc u).
// The paper has no gradient ("no backpropagation", Section 2.1); this is the
// differentiation extension of the same stiffness matrix. u^T dK/dtheta u
// of a 4x4 element comes from a reverse pass through its closed form
// (elem_quad_grad), in three directions: c, the layer's beta (Poisson ratio
// held, so alpha moves with beta) and the layer's thickness h; the
// half-space's 2x2 block from dual numbers in c and beta. Intervals without a
// simple root (poles) take the element in dual numbers too (layer_element_d).
#pragma once

#include "masw_device.cuh"

namespace masw {

struct D4 { double v, d0, d1, d2; };

__device__ __forceinline__ D4 mk(double v) { return {v, 0.0, 0.0, 0.0}; }
__device__ __forceinline__ D4 operator+(D4 a, D4 b) { return {a.v + b.v, a.d0 + b.d0, a.d1 + b.d1, a.d2 + b.d2}; }
__device__ __forceinline__ D4 operator-(D4 a, D4 b) { return {a.v - b.v, a.d0 - b.d0, a.d1 - b.d1, a.d2 - b.d2}; }
__device__ __forceinline__ D4 operator-(D4 a) { return {-a.v, -a.d0, -a.d1, -a.d2}; }
__device__ __forceinline__ D4 operator*(D4 a, D4 b) {
    return {a.v * b.v, a.d0 * b.v + a.v * b.d0, a.d1 * b.v + a.v * b.d1, a.d2 * b.v + a.v * b.d2};
}
__device__ __forceinline__ D4 operator*(double s, D4 a) { return {s * a.v, s * a.d0, s * a.d1, s * a.d2}; }
__device__ __forceinline__ D4 operator+(double s, D4 a) { return {s + a.v, a.d0, a.d1, a.d2}; }
__device__ __forceinline__ D4 operator/(D4 a, D4 b) {
    double iv = 1.0 / b.v;
    double q = a.v * iv;
    return {q, (a.d0 - q * b.d0) * iv, (a.d1 - q * b.d1) * iv, (a.d2 - q * b.d2) * iv};
}
__device__ __forceinline__ D4 chain(D4 a, double f, double df) {
    return {f, df * a.d0, df * a.d1, df * a.d2};
}
__device__ __forceinline__ D4 dexp(D4 a) { double e = exp(a.v); return chain(a, e, e); }
__device__ __forceinline__ D4 drsqrt(D4 a) {
    double r = rsqrt(a.v);
    return chain(a, r, -0.5 * r * r * r);
}
__device__ __forceinline__ void dsincos(D4 a, D4* s, D4* c) {
    double sn, cs;
    sincos(a.v, &sn, &cs);
    *s = chain(a, sn, cs);
    *c = chain(a, cs, -sn);
}

__device__ __forceinline__ D4 dsqrt(D4 a) { double s = sqrt(a.v); return chain(a, s, 0.5 / s); }

// The even functions of one wave (wave_fns) and, for the derivative with
// respect to w^2, H = d(Sd)/d(w^2) = (x C - Sd) / (2 w^2) at x = k h (E, C, Sd,
// Sm scaled alike, E held: see elem_quad_grad); from its series where C and
// Sd are, d(sinh(x w)/w)/d(w^2) = x^3 sum_n n u^(n-1) / (2n+1)!, u = (x w)^2.
struct WaveH { double E, C, Sd, Sm, H; };
__device__ __forceinline__ WaveH wave_fns_h(double x, double w2) {
    const double x2 = x * x;
    const Wave f = wave_fns(x, x2, w2);
    const double u = x2 * w2;
    WaveH o{f.E, f.C, f.Sd, f.Sm, 0.0};
    if (abs_lt(u, SERIES_U)) {
        double p = 8.0 * inv_fact(17);
        p = fma(p, u, 7.0 * inv_fact(15));
        p = fma(p, u, 6.0 * inv_fact(13));
        p = fma(p, u, 5.0 * inv_fact(11));
        p = fma(p, u, 4.0 * inv_fact(9));
        p = fma(p, u, 3.0 * inv_fact(7));
        p = fma(p, u, 2.0 * inv_fact(5));
        p = fma(p, u, inv_fact(3));
        o.H = x * x2 * p;
    } else {
        o.H = fma(x, f.C, -f.Sd) / (2.0 * w2);
    }
    return o;
}

// The derivatives of q = u^T K u of one finite layer, u = (x0, z0, x1, z1), with
// respect to c, beta (Poisson ratio held) and h: K = mu Phi(c^2/beta^2, k h) has
// two independent directions only. With q / mu = Nn / D (D the element's
// denominator, Nn the quadratic form of its numerators) and phi = q / mu,
// d q = (mu / D) d L, L = Nn - phi D, phi held; the reverse pass takes L's
// derivatives with respect to the two waves' C, Sd, Sm, then those with respect
// to kh and w^2:
//   d(C, Sd, Sm)/d(kh) = (Sm, C, w^2 C),
//   d(C, Sd, Sm)/d(w^2) = (kh Sd / 2, H, (Sd + kh C) / 2).
// L is zero and homogeneous in each wave's (E, C, Sd, Sm), so their common
// scale e^-x is held: its derivative drops out.
__device__ __forceinline__ void elem_quad_grad(const double* __restrict__ L, double k, double c,
                                               double c2, double x0, double z0, double x1,
                                               double z1, double* qc, double* qb, double* qh) {
    const double h = L[L_H], ib2 = L[L_IB2], mu = L[L_MU];
    const double X = k * h;
    const double xi2 = c2 * ib2, pp = c2 * L[L_IA2];
    const double r2 = 1.0 - pp, s2 = 1.0 - xi2;
    const WaveH R = wave_fns_h(X, r2), S = wave_fns_h(X, s2);
    const double xx = fma(x0, x0, x1 * x1), zz = fma(z0, z0, z1 * z1);
    const double b = 2.0 * fma(x0, z0, -x1 * z1), e = 2.0 * x0 * x1;
    const double f = 2.0 * fma(x0, z1, -z0 * x1), g = 2.0 * z0 * z1;
    const double u = fma(R.E, S.E, -R.C * S.C), SdSd = R.Sd * S.Sd;
    const double D = fma(2.0, u, fma(R.Sm, S.Sm, SdSd));
    const double iD = 1.0 / D;
    const double A1 = fma(R.C, S.Sd, -S.C * R.Sm), D1 = fma(S.C, R.Sd, -R.C * S.Sm);
    const double E1 = fma(R.Sm, S.E, -R.E * S.Sd), G1 = fma(S.Sm, R.E, -S.E * R.Sd);
    const double F1 = fma(R.E, S.C, -R.C * S.E);
    const double B1 = fma(s2 + 3.0, -u, -fma(S.Sm, fma(2.0, R.Sm, R.Sd), SdSd));
    const double n1 = fma(xx, A1, fma(zz, D1, fma(e, E1, fma(f, F1, g * G1))));
    const double phi = fma(xi2, n1, b * B1) * iD;
    const double ax = xi2 * xx, az = xi2 * zz, ae = xi2 * e, af = xi2 * f, ag = xi2 * g;
    const double bc = fma(b, s2 + 3.0, 2.0 * phi);  // of C_r C_s in L
    const double bs = b + phi;
    // L's derivatives with respect to the waves' functions
    const double Cr = fma(ax, S.Sd, fma(-az, S.Sm, fma(-af, S.E, bc * S.C)));
    const double Cs = fma(-ax, R.Sm, fma(az, R.Sd, fma(af, R.E, bc * R.C)));
    const double Sdr = fma(az, S.C, fma(-ag, S.E, fma(-b, S.Sm, -bs * S.Sd)));
    const double Sds = fma(ax, R.C, fma(-ae, R.E, -bs * R.Sd));
    const double Smr = fma(-ax, S.C, fma(ae, S.E, -fma(2.0, b, phi) * S.Sm));
    const double Sms = fma(-az, R.C, fma(ag, R.E, -fma(fma(2.0, b, phi), R.Sm, b * R.Sd)));
    // ... to kh and to the two w^2
    const double LX = fma(Cr, R.Sm, R.C * fma(Smr, r2, Sdr)) +
                      fma(Cs, S.Sm, S.C * fma(Sms, s2, Sds));
    const double hx = 0.5 * X;
    const double Lr = fma(Cr, hx * R.Sd, fma(Sdr, R.H, Smr * fma(hx, R.C, 0.5 * R.Sd)));
    const double Ls = fma(Cs, hx * S.Sd, fma(Sds, S.H, Sms * fma(hx, S.C, 0.5 * S.Sd))) - b * u;
    // r2 = 1 - xi2 (beta/alpha)^2, s2 = 1 - xi2: xi2 d/d(xi2) of L
    const double Lxi = fma(xi2, n1 - Ls, -pp * Lr);
    const double mD = mu * iD;
    const double gc = 2.0 * mD * Lxi;  // c d q / d c
    const double beta = L[L_BETA];
    *qc = gc / c;
    *qb = fma(2.0 * mu, phi, -gc) / beta;
    *qh = mD * LX * k;
}

struct WaveD { D4 E, C, Sd, Sm; };

// Dual version of wave_fns (same branches, same scaling).
__device__ inline WaveD wave_fns_d(D4 kh, D4 w2) {
    D4 u = kh * kh * w2;
    WaveD o;
    if (fabs(u.v) < SERIES_U) {
        D4 pc = mk(inv_fact(18));
        const double cc[9] = {inv_fact(16), inv_fact(14), inv_fact(12), inv_fact(10), inv_fact(8),
                              inv_fact(6), inv_fact(4), inv_fact(2), 1.0};
        for (int i = 0; i < 9; ++i) pc = cc[i] + pc * u;
        D4 ps = mk(inv_fact(17));
        const double cs[8] = {inv_fact(15), inv_fact(13), inv_fact(11), inv_fact(9), inv_fact(7),
                              inv_fact(5), inv_fact(3), 1.0};
        for (int i = 0; i < 8; ++i) ps = cs[i] + ps * u;
        D4 khps = kh * ps;
        o.E = mk(1.0);
        o.C = pc;
        o.Sd = khps;
        o.Sm = w2 * khps;
    } else if (w2.v > 0.0) {
        D4 rw = drsqrt(w2);
        D4 w = w2 * rw;
        D4 E = dexp(-(kh * w));
        D4 E2 = E * E;
        D4 t = 0.5 + (-0.5) * E2;
        o.E = E;
        o.C = 0.5 + 0.5 * E2;
        o.Sd = t * rw;
        o.Sm = t * w;
    } else {
        D4 rw = drsqrt(-w2);
        D4 w = (-w2) * rw;
        D4 sn, cs;
        dsincos(kh * w, &sn, &cs);
        o.E = mk(1.0);
        o.C = cs;
        o.Sd = sn * rw;
        o.Sm = -(w * sn);
    }
    return o;
}

// Element stiffness entries (k dropped) of one finite layer as duals in the
// directions (c, beta, h): K = [[A, B, E, F], [B, Dd, -F, G],
// [E, -F, A, -B], [F, G, -B, Dd]].
struct ElemD { D4 A, B, Dd, E, F, G; };

__device__ inline ElemD layer_element_d(const double* __restrict__ L, double k, double c) {
    D4 cc = {c, 1.0, 0.0, 0.0};
    D4 be = {L[L_BETA], 0.0, 1.0, 0.0};
    D4 hh = {L[L_H], 0.0, 0.0, 1.0};
    double rho = L[L_RHO], ratio = L[L_RATIO];
    D4 c2 = cc * cc;
    D4 b2 = be * be;
    D4 mu = rho * b2;
    D4 q = c2 / b2;
    D4 r2 = 1.0 + (-1.0) * (c2 / ((ratio * ratio) * b2));
    D4 s2 = 1.0 + (-1.0) * q;
    D4 kh = k * hh;
    WaveD R = wave_fns_d(kh, r2);
    WaveD S = wave_fns_d(kh, s2);
    D4 ErEs = R.E * S.E;
    D4 CrCs = R.C * S.C;
    D4 Dh = 2.0 * (ErEs - CrCs) + R.Sd * S.Sd + R.Sm * S.Sm;
    D4 A1 = R.C * S.Sd - S.C * R.Sm;
    D4 D1 = S.C * R.Sd - R.C * S.Sm;
    D4 B1 = (s2 + mk(3.0)) * (CrCs - ErEs) - S.Sm * (2.0 * R.Sm + R.Sd) - R.Sd * S.Sd;
    D4 E1 = R.Sm * S.E - R.E * S.Sd;
    D4 F1 = R.E * S.C - R.C * S.E;
    D4 G1 = S.Sm * R.E - S.E * R.Sd;
    D4 rc2 = rho * c2;
    ElemD o;
    o.A = rc2 * A1 / Dh;
    o.B = mu * B1 / Dh;
    o.Dd = rc2 * D1 / Dh;
    o.E = rc2 * E1 / Dh;
    o.F = rc2 * F1 / Dh;
    o.G = rc2 * G1 / Dh;
    return o;
}

// Quadratic form u_e^T K u_e of an element and its three directional
// derivatives; u = (x0, z0, x1, z1).
__device__ __forceinline__ D4 elem_quad(const ElemD& K, double x0, double z0, double x1, double z1) {
    double xx = x0 * x0 + x1 * x1, zz = z0 * z0 + z1 * z1;
    double b = 2.0 * (x0 * z0 - x1 * z1), e = 2.0 * x0 * x1, f = 2.0 * (x0 * z1 - z0 * x1),
           g = 2.0 * z0 * z1;
    return xx * K.A + zz * K.Dd + b * K.B + e * K.E + f * K.F + g * K.G;
}

// Half-space 2x2 (k dropped) as duals in (c, beta_hs, unused).
struct HalfD { D4 H00, H01, H11; };

__device__ inline HalfD halfspace_d(const double* __restrict__ L, double c) {
    D4 cc = {c, 1.0, 0.0, 0.0};
    D4 be = {L[L_BETA], 0.0, 1.0, 0.0};
    double rho = L[L_RHO], ratio = L[L_RATIO];
    D4 c2 = cc * cc;
    D4 b2 = be * be;
    D4 mu = rho * b2;
    D4 q = c2 / b2;
    D4 p = c2 / ((ratio * ratio) * b2);
    D4 r = dsqrt(1.0 + (-1.0) * p);
    D4 s = dsqrt(1.0 + (-1.0) * q);
    D4 g = 1.0 + r * s;
    D4 den = (p + q - p * q) / g;  // 1 - r s
    D4 rc2 = rho * c2;
    HalfD o;
    o.H00 = rc2 * r / den;
    o.H01 = mu * (q - 2.0 * den) / den;
    o.H11 = rc2 * s / den;
    return o;
}

__device__ __forceinline__ D4 half_quad(const HalfD& H, double x, double z) {
    return (x * x) * H.H00 + (2.0 * x * z) * H.H01 + (z * z) * H.H11;
}

}  // namespace masw
