// masw_bound.cuh -- FP32 count of K's negative eigenvalues with a running
// error bound: the count and whether it is proven.
//
// The certificate of the counting search needs the count at V[n-1] and V[n].
// Its double-float recurrence takes about 1,640 thread instructions a
// layer-evaluation, this one about 280, and the root lies anywhere between
// the two points: a relative distance of u dc / c from the nearer one, u
// uniform, against FP32 errors of 1e-7 .. 1e-5 of the pivots. So most counts
// are already decided here, with a floating-point filter: the recurrence
// carries a bound E of the error of its 2x2 state P (-E <= error <= E, a
// symmetric matrix), a pivot S = P + K11 whose bound keeps every perturbed S
// nonsingular has the inertia of the exact one, and when every pivot does, the
// count is the exact count of K (Sylvester). Otherwise the point goes to the
// double-float recurrence (masw_df.cuh), which also decides whatever this
// filter cannot.
//
// The recurrence. A layer thin next to the wavelength has K11, K12 of order
// 1/(kh) and P' - P of order kh, so P' = K22 - K21 S^-1 K12 loses (kh)^-2 in
// relative accuracy. With W = P + K11 + K12 (= S + K12) the same P' is
//   P' = P + 2 diag(A + E, D + G) - W^T S^-1 W
// (K11 = [[A, B], [B, D]], K12 = [[E, F], [-F, G]], K22 = [[A, -B], [-B, D]]),
// whose terms are of order kh where A + E and D + G are formed without
// cancellation: A + E from e^-x cosh x - e^-x = (1 - e^-x)^2 / 2. For a thick
// layer K12 is the small one and the first form has no cancellation; the
// smaller of W and K12 picks the form.
//
// The bound (first order, with the second-order factor of S^-1; eps = 2^-24).
// With T = S^-1 K12 and R = S^-1 W = T + I, an error E of P reaches P' as
// T^T E T, which keeps its direction: next to a pivot that is nearly singular
// P' is large along one vector and its error with it, while the other vector's
// stays small (a bound by norms alone proved 67 % instead of 89 % of the counts
// at random velocities of the uniform batch). The computed element differs
// from the exact one in three ways:
//  * its common denominator (relative error th: the sum of the magnitudes of
//    D's terms over |D|) scales K11, K12, K22 together, which changes the
//    element's energy, at most 2 q1 + 2 (q1 + q2) R + R^T K11 R with
//    q1 = max(|A + E|, |D + G|), q2 = |B| + |F|, by th;
//  * its numerators (the sums of the magnitudes of their terms over |D|): an
//    error dn of K11 enters as dn R^T R, dd of A + E and D + G as
//    2 dd (1 + R), dO of B and F as 2 dO R (2 x R <= x (I + R^T R));
//  * the rounded inputs (k, h, c, moduli), in effect another layer within a
//    few eps: the kinetic energy's kin = rho c^2 min(kh, 1) (I + T^T T), and,
//    for the phases x = k h |w|, whose error grows with k h q / |w| (an
//    error of q moves w^2 = 1 - q by as much), a factor `amp` on all of these.
// The Schur step's own rounding adds eps (||X|| ||S^-1 X|| cond(S) + ||Q||) for
// P' = Q - X^T S^-1 X. Every S + error is nonsingular when the eigenvalues of
// E^(1/2) S^-1 E^(1/2) stay below 1 in magnitude; 1/2 is asked.
// The constants in front of eps were set by measuring the error of P against
// the double-float recurrence, layer by layer: the largest eigenvalue of
// E^-1 error was 0.35 over 1.9 million evaluations of the uniform and
// ragged workloads (around the root and at random velocities) and 0.64
// over 0.39 million of models far outside them (thicknesses 0.05..50 m at
// wavelengths 0.5..500 m). No proven count differed
// from the double-float one. The bound proves both counts of 95 % (uniform)
// and 92 % (ragged) of the items and one of the two for nearly all others.
//
// The element is the screen's (masw_screen.cuh), with 1 - E_r E_s from the
// e^-x - 1 it is made of.
#pragma once

#include "masw_screen.cuh"

namespace masw {

constexpr float BOUND_EPS = 5.9604645e-8f;        // 2^-24
constexpr float BOUND_EL = 4.0f * BOUND_EPS;     // element and inputs
constexpr float BOUND_STEP = 2.0f * BOUND_EPS;    // Schur step

__device__ __forceinline__ float sqrt_approx(float x) {
    float r;
    asm("sqrt.approx.ftz.f32 %0, %1;" : "=f"(r) : "f"(x));
    return r;
}

// An element so near its pole that its denominator's relative error could
// exceed this is left to the double-float recurrence (the bound is of first
// order in that error).
constexpr float BOUND_SCALE = 1.0f / 64.0f;

// max-norm sum of a symmetric 2x2 block, an upper bound of its 2-norm
__device__ __forceinline__ float norm_2x2(float a, float b, float d) {
    return fmaxf(fabsf(a), fabsf(d)) + fabsf(b);
}

// An element's denominator and numerators (D, A, D, B, F of det_core_f; AE and
// DG of A + E and D + G), the sums of the magnitudes of their terms (tD of the
// denominator, t1 the larger of A and D, tB, tF, t2 the larger of AE and DG)
// and the phase factor times the element constant.
struct ElemBound { float Dh, A1, D1, B1, F1, AE, DG, tD, t1, tB, tF, t2, ca; };

// wave_fns_f with V = C - E: cosh - 1 (or cos - 1) where E = 1, and
// e^-x cosh x - e^-x = (1 - E)^2 / 2 where E = e^-x.
// mC, mSd, mSm, mV: their magnitudes for the sums of terms; in the
// trigonometric branch the amplitudes (1, 1/|w|, |w|, 1), since an error of the
// phase moves a sine near its zero by the amplitude.
struct WaveV { float E, C, Sd, Sm, V, mC, mSd, mSm, mV; };
__device__ __forceinline__ WaveV wave_fns_v(float kh, float w2) {
    const float u = kh * kh * w2;
    WaveV o;
    if (fabsf(u) < 1.0f) {
        float pc = fmaf(u, 1.0f / 3628800.0f, 1.0f / 40320.0f);
        pc = fmaf(pc, u, 1.0f / 720.0f);
        pc = fmaf(pc, u, 1.0f / 24.0f);
        pc = fmaf(pc, u, 0.5f);
        float ps = fmaf(u, 1.0f / 39916800.0f, 1.0f / 362880.0f);
        ps = fmaf(ps, u, 1.0f / 5040.0f);
        ps = fmaf(ps, u, 1.0f / 120.0f);
        ps = fmaf(ps, u, 1.0f / 6.0f);
        ps = fmaf(ps, u, 1.0f);
        o.E = 1.0f;
        o.V = pc * u;
        o.C = 1.0f + o.V;
        o.Sd = kh * ps;
        o.Sm = w2 * o.Sd;
        o.mC = o.C;
        o.mSd = o.Sd;
        o.mSm = fabsf(o.Sm);
        o.mV = fabsf(o.V);
    } else {
        const WaveF f = wave_fns_f(kh, w2);
        o.E = f.E;
        o.C = f.C;
        o.Sd = f.Sd;
        o.Sm = f.Sm;
        const float m = 1.0f - f.E;
        o.V = w2 > 0.0f ? 0.5f * m * m : f.C - 1.0f;
        const float rw = rsqrtf(fabsf(w2));
        o.mC = w2 > 0.0f ? f.C : 1.0f;
        o.mSd = w2 > 0.0f ? f.Sd : rw;
        o.mSm = w2 > 0.0f ? f.Sm : -w2 * rw;
        o.mV = w2 > 0.0f ? o.V : fmaxf(-o.V, 1.0f);
    }
    return o;
}

// The element above the layer's shear speed (s2 <= 0), every difference of
// products of E and C written with V:
//   E_r E_s - C_r C_s = -(V_r E_s + V_s E_r + V_r V_s),  F = E_r V_s - V_r E_s,
//   A + E = Sd_s V_r - Sm_r V_s,  D + G = Sd_r V_s - Sm_s V_r.
// Out of line: fewer layers take it, and the hot branch below the shear speed
// stays compact.
static __device__ __noinline__ ElemBound elem_bound_trig(float kh, float pp, float q) {
    const float r2 = 1.0f - pp, s2 = 1.0f - q;
    const WaveV R = wave_fns_v(kh, r2), S = wave_fns_v(kh, s2);
    ElemBound o;
    const float u1 = R.V * S.E, u2 = S.V * R.E, u3 = R.V * S.V;
    const float m1 = R.mV * S.E, m2 = S.mV * R.E, tU = fmaf(R.mV, S.mV, m1 + m2);
    const float SdSd = R.Sd * S.Sd, u = -(u1 + u2 + u3), mSS = R.mSd * S.mSd;
    o.Dh = fmaf(2.0f, u, fmaf(R.Sm, S.Sm, SdSd));
    o.tD = fmaf(2.0f, tU, fmaf(R.mSm, S.mSm, mSS));
    o.A1 = fmaf(R.C, S.Sd, -S.C * R.Sm);
    o.D1 = fmaf(S.C, R.Sd, -R.C * S.Sm);
    o.t1 = fmaxf(fmaf(R.mC, S.mSd, S.mC * R.mSm), fmaf(S.mC, R.mSd, R.mC * S.mSm));
    o.B1 = -fmaf(s2 + 3.0f, u, fmaf(S.Sm, fmaf(2.0f, R.Sm, R.Sd), SdSd));
    o.tB = fmaf(fabsf(s2) + 3.0f, tU, fmaf(S.mSm, fmaf(2.0f, R.mSm, R.mSd), mSS));
    o.F1 = u2 - u1;
    o.tF = m1 + m2;
    o.AE = fmaf(S.Sd, R.V, -R.Sm * S.V);
    o.DG = fmaf(R.Sd, S.V, -S.Sm * R.V);
    o.t2 = fmaxf(fmaf(S.mSd, R.mV, R.mSm * S.mV), fmaf(R.mSd, S.mV, S.mSm * R.mV));
    const float amp = fmaf(0.5f * kh * q, fminf(kh, rsqrtf(fabsf(s2))), 1.0f) +
                      0.5f * kh * pp * R.E * fminf(kh, rsqrtf(fabsf(r2)));
    o.ca = BOUND_EL * amp;
    return o;
}

// The state of the recurrence: P and the bound E of its error, -E <= error <= E.
struct BoundState { float p00, p01, p11, e00, e01, e11; };

// Eliminates one layer's top node: the number of negative eigenvalues of its
// pivot; *sure is cleared when the pivot's inertia is not proven. BOUND false:
// the recurrence alone.
template <bool BOUND>
__device__ __forceinline__ int bound_layer(BoundState& st, const float* __restrict__ L, float k,
                                           float c2, bool* sure) {
    const float4 LA = *reinterpret_cast<const float4*>(L);
    const float2 LB = *reinterpret_cast<const float2*>(L + 4);
    const float kh = k * LA.x, q = c2 * LB.x, pp = c2 * LA.w;
    const float r2 = 1.0f - pp, s2 = 1.0f - q;
    ElemBound o;
    if (s2 > 0.0f) {
        const float rwr = rsqrtf(r2), rws = rsqrtf(s2);
        const float r = r2 * rwr, s = s2 * rws;
        const float emr1 = expm1_neg(-kh * r), ems1 = expm1_neg(-kh * s);
        const float Er = 1.0f + emr1, Es = 1.0f + ems1;
        const float hr = -0.5f * emr1 * (1.0f + Er), hs = -0.5f * ems1 * (1.0f + Es);
        const float cr = 1.0f - hr, cs = 1.0f - hs;
        const float rs = r * s;
        const float dE = -Es * expm1_neg(-kh * c2 * LB.y * rcp_approx(r + s));
        const float omP = -fmaf(emr1, ems1, emr1 + ems1);  // 1 - E_r E_s
        const float om = fmaf(-pp, q, pp + q) * rcp_approx(1.0f + rs);
        const float shd = 0.5f * dE * (Es + Er);
        const float dE2 = dE * dE, x1 = om * om * (hr * rwr) * (hs * rws);
        o.Dh = x1 - dE2;
        o.tD = x1 + dE2;
        const float xa = om * cs * hr;
        o.A1 = (xa - shd) * rws;
        o.D1 = fmaf(om * cr, hs, shd) * rwr;
        const float K2 = fmaf(4.0f - q, rs, fmaf(2.0f * rs, rs, s2 + 1.0f));
        const float xb = dE2 * K2, xc = omP * omP * om, w4 = 0.25f * rwr * rws;
        o.B1 = fmaf(xc, fmaf(-2.0f, om, q), xb) * w4;
        o.tB = fmaf(xc, fmaf(2.0f, om, q), xb) * w4;
        o.tF = 0.5f * dE * omP;
        o.F1 = -o.tF;
        // A + E and D + G, with cosh - e^-x = (1 - e^-x)^2 / 2 (scaled)
        o.AE = 0.5f * ems1 * fmaf(om * hr, ems1, dE * emr1) * rws;
        const float g1 = om * hs * emr1, g2 = dE * ems1, wg = 0.5f * emr1 * rwr;
        o.DG = wg * (g1 - g2);
        o.t2 = fmaxf(o.AE, wg * (g1 + g2));
        o.t1 = fmaxf((xa + shd) * rws, o.D1);
        o.ca = BOUND_EL * fmaf(0.5f * kh * q * Es, fminf(kh, rws), 1.0f);
    } else {
        o = elem_bound_trig(kh, pp, q);
    }
    const float iD = rcp_approx(o.Dh), rc2 = LA.z * c2;
    const float fr = rc2 * iD, fm = LA.y * iD;
    const float n00 = fr * o.A1, n01 = fm * o.B1, n11 = fr * o.D1;
    const float cf = fr * o.F1, aE = fr * o.AE, dG = fr * o.DG;
    const float s00 = st.p00 + n00, s01 = st.p01 + n01, s11 = st.p11 + n11;
    const float det = fmaf(s00, s11, -s01 * s01);
    const float idet = rcp_approx(det);
    const float ai = fabsf(idet), afr = fabsf(fr);
    // P' = Q - X^T Y, Y = S^-1 X: X = W = P + K11 + K12, Q = P + 2 diag(A + E, D + G)
    // for a thin layer, X = K12, Q = K22 for a thick one, whichever X is smaller
    const float ce = aE - n00, cg = dG - n11;
    const float q1 = fmaxf(fabsf(aE), fabsf(dG)), pn = norm_2x2(st.p00, st.p01, st.p11);
    const float q2 = fabsf(n01) + fabsf(cf);
    const float mW = pn + q1 + q2, m12 = norm_2x2(ce, cf, cg);
    const bool thin = mW < m12;
    const float w00 = thin ? st.p00 + aE : ce, w11 = thin ? st.p11 + dG : cg;
    const float w01 = thin ? s01 + cf : cf, w10 = thin ? s01 - cf : -cf;
    const float y00 = idet * fmaf(s11, w00, -s01 * w10), y01 = idet * fmaf(s11, w01, -s01 * w11);
    const float y10 = idet * fmaf(s00, w10, -s01 * w00), y11 = idet * fmaf(s00, w11, -s01 * w01);
    st.p00 = (thin ? fmaf(2.0f, aE, st.p00) : n00) - fmaf(w00, y00, w10 * y10);
    st.p01 = (thin ? st.p01 : -n01) - fmaf(w00, y01, w10 * y11);
    st.p11 = (thin ? fmaf(2.0f, dG, st.p11) : n11) - fmaf(w01, y01, w11 * y11);
    if (!BOUND) return neg_eigs_2x2(det, s00);
    // the bound
    const float M = norm_2x2(n00, n01, n11);
    const float dO = o.ca * fmaf(fabsf(fm), o.tB, afr * o.tF);
    const float dn = fmaf(o.ca * afr, o.t1, dO), dd = o.ca * afr * o.t2;
    const float th = o.ca * fmaf(o.tD, fabsf(iD), 1.0f);
    const float mS = norm_2x2(s00, s01, s11), cond = mS * mS * ai;
    const float loc = fmaf(th, M, fmaf(BOUND_EPS, mS, dn));
    const float f00 = st.e00 + loc, f11 = st.e11 + loc;
    // the largest eigenvalue of E^(1/2) S^-1 E^(1/2), at most |trace| + sqrt|det|
    const float tr = idet * fmaf(s11, f00, fmaf(s00, f11, -2.0f * s01 * st.e01));
    const float dt = ai * fabsf(fmaf(f00, f11, -st.e01 * st.e01));
    const float rho = fabsf(tr) + sqrt_approx(dt);
    // (a NaN or infinity anywhere leaves the comparisons false)
    *sure = *sure && (fmaf(4.0f * BOUND_EPS, cond, rho) < 0.5f) && th < BOUND_SCALE;
    const float kin = o.ca * fabsf(rc2) * fminf(kh, 1.0f);
    const float cross = fmaf(th, q1 + q2, dd + dO);
    // R = S^-1 W, T = S^-1 K12 = R - I
    const float one = thin ? 1.0f : 0.0f;
    const float x00 = y00 - one, x11 = y11 - one, r00 = x00 + 1.0f, r11 = x11 + 1.0f;
    const float y2 = fmaxf(fabsf(y00), fabsf(y11)) + fmaxf(fabsf(y01), fabsf(y10));  // >= ||Y||
    const float mX = thin ? mW : m12, mQ = thin ? fmaf(2.0f, q1, pn) : M;
    const float al = fmaf(2.0f, fmaf(th, q1, dd), cross) + kin +
                     fmaf(BOUND_STEP, fmaf(mX * y2, cond, mQ), 4.0f * BOUND_EPS * (st.e00 + st.e11));
    const float be = fmaf(th, M, dn) + cross;
    // E' = (1 + 2 rho) T^T (E + kin) T + al + be R^T R
    const float g = fmaf(2.0f, rho, 1.0f), k00 = st.e00 + kin, k11 = st.e11 + kin, k01 = st.e01;
    const float v00 = fmaf(k00, x00, k01 * y10), v01 = fmaf(k00, y01, k01 * x11);
    const float v10 = fmaf(k01, x00, k11 * y10), v11 = fmaf(k01, y01, k11 * x11);
    st.e00 = fmaf(g, fmaf(x00, v00, y10 * v10), fmaf(be, fmaf(r00, r00, y10 * y10), al));
    st.e01 = fmaf(g, fmaf(x00, v01, y10 * v11), be * fmaf(r00, y01, y10 * r11));
    st.e11 = fmaf(g, fmaf(y01, v01, x11 * v11), fmaf(be, fmaf(y01, y01, r11 * r11), al));
    return neg_eigs_2x2(det, s00);
}

// Negative eigenvalues of K(k, c) (inertia_f) with the running bound: *sure
// is true when the count is proven (BOUND false: not touched). Requires
// c < beta_halfspace.
template <bool BOUND = true>
__device__ __forceinline__ int inertia_bound_f(const float* __restrict__ lay, int N, float k,
                                               float c, bool* sure) {
    const float c2 = c * c;
    BoundState st{0.0f, 0.0f, 0.0f, 0.0f, 0.0f, 0.0f};
    bool ok = true;
    int cnt = 0;
    for (int j = 0; j < N; ++j) cnt += bound_layer<BOUND>(st, lay + j * LAYER_STRIDE32, k, c2, &ok);
    const float4 LA = *reinterpret_cast<const float4*>(lay + N * LAYER_STRIDE32);
    const float q = c2 * lay[N * LAYER_STRIDE32 + 4], p = c2 * LA.w;
    const float s2 = 1.0f - q, r = sqrtf(1.0f - p), s = sqrtf(s2);
    const float g = fmaf(r, s, 1.0f), den = fmaf(-p, q, p + q);
    const float iden = rcp_approx(den);
    const float rc2g = LA.z * c2 * g * iden;
    const float h00 = rc2g * r, h11 = rc2g * s;
    const float h01 = LA.y * iden * fmaf(g, q, -2.0f * den);
    const float s00 = st.p00 + h00, s01 = st.p01 + h01, s11 = st.p11 + h11;
    const float det = fmaf(s00, s11, -s01 * s01);
    if (!BOUND) return cnt + neg_eigs_2x2(det, s00);
    const float mS = norm_2x2(s00, s01, s11);
    // the half-space block: its terms, and s = sqrt(1 - q), whose error is that of q over s
    const float mH = fmaxf(h00, h11) + LA.y * iden * fmaf(g, q, 2.0f * den) + rc2g * rsqrtf(s2);
    const float loc = BOUND_EL * mH + BOUND_EPS * mS;
    const float f00 = st.e00 + loc, f11 = st.e11 + loc, idet = rcp_approx(det);
    const float tr = idet * fmaf(s11, f00, fmaf(s00, f11, -2.0f * s01 * st.e01));
    const float dt = fabsf(idet * fmaf(f00, f11, -st.e01 * st.e01));
    *sure = ok && (fmaf(4.0f * BOUND_EPS * mS * mS, fabsf(idet), fabsf(tr) + sqrt_approx(dt)) < 0.5f);
    return cnt + neg_eigs_2x2(det, s00);
}

// clamped_modes_f (masw_screen.cuh) with *sure cleared when one of the signs it
// rests on is not proven: a numerator or denominator within its error, the
// element's constant times the amplitudes of its terms, the phase's part (amp
// at that level's thickness) and the doublings' (2 per level) included, and a
// further factor of four. The level is taken from a slightly larger x: any
// level whose pieces lie under the pole-free bound gives the count.
__device__ __forceinline__ int clamped_modes_bound_f(const float* __restrict__ L, float k, float c2,
                                                     bool* sure) {
    const float q = c2 * L[F_IB2];
    if (!(q > 1.0f - 1.0e-5f)) return 0;
    const float kh = k * L[F_H], q1 = fmaxf(q - 1.0f, 0.0f);
    const float x = 1.001f * fmaf(kh, sqrtf(q1) * 0.318309886f, 1.0e-3f);  // kh sqrt(q - 1) / pi
    if (!(x >= 1.0f)) return 0;
    if (!(x < 1.0e30f)) {
        *sure = false;
        return 0;
    }
    const int lv = ((__float_as_int(x) >> 23) & 0xff) - 126;  // 2^lv > x >= 2^(lv-1)
    float khj = kh * __int_as_float((127 - lv) << 23);        // kh 2^-lv, exact
    const float r2 = fmaf(-c2, L[F_IA2], 1.0f), s2 = 1.0f - q;
    WaveF R = wave_fns_f(khj, r2), S = wave_fns_f(khj, s2);
    const float ar = fmaxf(sqrt_approx(fabsf(r2)), 1.0e-3f), as = fmaxf(sqrt_approx(fabsf(s2)), 1.0e-3f);
    const float ir = rcp_approx(ar), is = rcp_approx(as);
    float grow = 1.0f;
    int J = 0;
    for (int j = lv; j >= 1; --j) {
        if (j < lv) {
            R = WaveF{R.E * R.E, fmaf(2.0f * R.C, R.C, -R.E * R.E), 2.0f * R.Sd * R.C,
                      2.0f * R.Sm * R.C};
            S = WaveF{S.E * S.E, fmaf(2.0f * S.C, S.C, -S.E * S.E), 2.0f * S.Sd * S.C,
                      2.0f * S.Sm * S.C};
            khj *= 2.0f;
            grow *= 2.0f;
        }
        const float D = fmaf(2.0f, fmaf(R.E, S.E, -R.C * S.C), fmaf(R.Sd, S.Sd, R.Sm * S.Sm));
        const float an = fmaf(R.C, S.Sd, -S.C * R.Sm);
        const float dn = fmaf(S.C, R.Sd, -R.C * S.Sm);
        const float amp = 0.5f * khj * (q * fminf(khj, is) + c2 * L[F_IA2] * fminf(khj, ir));
        const float tol = 4.0f * BOUND_EL * (grow + amp);
        // amplitudes: C <= 1, Sd <= min(1/w, kh), Sm <= w (each times at most 1)
        const float mr = fminf(ir, khj), ms = fminf(is, khj);
        if (!(fabsf(D) > tol * fmaf(mr, ms, fmaf(ar, as, 4.0f)) && fabsf(an) > tol * (ms + ar) &&
              fabsf(dn) > tol * (mr + as)))
            *sure = false;
        J = 2 * J + (int)((an < 0.0f) != (D < 0.0f)) + (int)((dn < 0.0f) != (D < 0.0f));
    }
    return J;
}

// The mode count T = s + 2 J0 with its proof (inertia_bound_f,
// clamped_modes_bound_f).
__device__ __forceinline__ int mode_count_bound_f(const float* __restrict__ lay, int N, float k,
                                                  float c, int* s_out, bool* sure) {
    const int s = inertia_bound_f(lay, N, k, c, sure);
    const float c2 = c * c;
    int j0 = 0;
    for (int j = 0; j < N; ++j) j0 += clamped_modes_bound_f(lay + j * LAYER_STRIDE32, k, c2, sure);
    *s_out = s;
    return s + 2 * j0;
}

}  // namespace masw
