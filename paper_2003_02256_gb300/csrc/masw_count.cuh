// masw_count.cuh -- counting search with its FP64 certificate for one
// (model, wavenumber) item (plan precision 2 of the batch path and the
// serving tick).
//
//  * Search (FP32). Inside the pole-free range [0, npf) of pole_free_points_f
//    the negative-eigenvalue count of K (inertia_f) is a non-decreasing step
//    function of the grid index, 0 at c = 0 (Wittrick-Williams below the
//    lowest clamped-layer mode). One thread bisects it (count_search_single,
//    or count_search_guess from a guess interpolated between the indices of
//    neighbouring wavelengths), or G lanes split the bracket in G + 1 per step
//    (the _group forms): about log2(npf), or log_{G+1}(npf) steps, instead of
//    Algorithm 1's linear walk.
//  * Certificate. The count is 0 at V[n-1] (so 0, and V[0]'s sign, at every
//    point below) and odd at V[n] (the sign differs). The search evaluates
//    these two counts with their FP32 error bound (masw_bound.cuh); the ones
//    it does not prove are evaluated in double-float (det_inertia_dd in
//    masw_df.cuh, the half-space's step in FP64). When the FP32 count was off
//    next to the change (count 0 at both points: the change is higher;
//    nonzero at V[n-1]: lower), a few double-float points in that direction,
//    inside the range, settle it. An even count (two or more) after count 0
//    means no sign change there: a second search looks for the first odd count
//    above it, certified the same way. Items left without a certificate take
//    the sign scan (batch path) or the linear screen (serving tick) from the
//    last point known to have an even count.
#pragma once

#include "masw_bound.cuh"
#include "masw_device.cuh"
#include "masw_df.cuh"
#include "masw_screen.cuh"

namespace masw {

struct PairCount {
    int cert;   // certified first change (>= 1), or -1
    int n;      // the search's index when the certificate failed (>= 1), or -1
    int start;  // cert and n < 1: a linear scan's start (npf when the range holds no
                // change, the located point after an even FP64 count, else 0)
    int counts; // cert inside the pole-free range: the certificate's FP64 counts,
                // s(V[cert]) << 16 | s(V[cert-1]) (there J0 = 0, so T = s); else -1
};

__device__ __forceinline__ int pack_counts(int s_lo, int s_hi) {
    return (s_lo >= 0 && s_hi >= s_lo && s_hi < 32768) ? (s_hi << 16) | s_lo : -1;
}

// First grid index in (lo, top] whose FP32 negative-eigenvalue count is at
// least `target`, the count being non-decreasing there and below `target` at
// lo; -1 when the count at `top` is below `target`. The pair evaluates `top`
// and the bracket's midpoint, then splits the bracket in three per step (one
// point per lane). Both lanes return the same index.
static __device__ __noinline__ int pair_search(const float* __restrict__ lay32, int N, float kf,
                                           float c0f, float dcf, int lo, int top, int target,
                                           int half, unsigned pair) {
    int hi = top;
    const int mid = lo + ((hi - lo) >> 1);
    const int pt = half ? mid : hi;
    const int cnt = pt > lo ? inertia_f(lay32, N, kf, fmaf((float)pt, dcf, c0f)) : 0;
    const int oth = __shfl_xor_sync(pair, cnt, 1);
    const int c_top = half ? oth : cnt, c_mid = half ? cnt : oth;
    if (c_top < target) return -1;
    if (mid > lo) {
        if (c_mid >= target) hi = mid;
        else lo = mid;
    }
    while (hi - lo > 1) {
        const int len = hi - lo;
        const int a = lo + (len + 1) / 3, bq = lo + (2 * len + 1) / 3;  // lo < a <= bq < hi
        const int q = half ? bq : a;
        const int c = inertia_f(lay32, N, kf, fmaf((float)q, dcf, c0f));
        const int co = __shfl_xor_sync(pair, c, 1);
        const int ca = half ? co : c, cb = half ? c : co;
        if (ca >= target) {
            hi = a;
        } else if (cb >= target) {
            lo = a;
            hi = bq;
        } else {
            lo = bq;
        }
    }
    return hi;
}

// What the split search knows of an item: its index n (the first grid point
// in [0, npf) with a nonzero FP32 count, or -1) and which of the counts at
// V[n-1] and V[n] the FP32 error bound proves (masw_bound.cuh).
enum { PROOF_LO = 1, PROOF_HI = 2 };  // count 0 at V[n-1]; an odd count at V[n]
struct Located {
    int n;
    int proof;  // PROOF_LO | PROOF_HI
    int count;  // PROOF_HI: the count at V[n]
};

// FP32 count at grid point n with its error bound (the test velocity rounded
// once from its FP64 value).
__device__ __forceinline__ int count_bound_at(const float* __restrict__ lay32, int N, float kf,
                                              double c0, double dc, int n, bool* sure) {
    return inertia_bound_f(lay32, N, kf, (float)grid_c(c0, dc, n), sure);
}

// The search stage by one thread (the split search kernel on large batches):
// the first grid point in [0, npf) with a nonzero FP32 count, or -1, by
// bisection. One point per step is one bit per evaluation, the fewest; lane
// groups take fewer steps where latency counts. The bisection's
// points take the plain count and the two points of the result the bounded
// one: about 10 + 2 evaluations, the bounded one costing 1.5 plain ones.
__device__ __forceinline__ Located count_search_single(const float* __restrict__ lay32, int N,
                                                       double k, double c0, double dc, int npf) {
    Located r{-1, 0, 0};
    if (npf < 1) return r;
    const float kf = (float)k, c0f = (float)c0, dcf = (float)dc;
    // count 0 at lo (c = 0 when lo = -1), nonzero at hi; the top is taken as
    // nonzero and evaluated only when the bisection ends there (the change
    // lies inside the range for nearly every item: one evaluation fewer)
    int lo = -1, hi = npf - 1;
    while (hi - lo > 1) {
        const int mid = lo + ((hi - lo) >> 1);
        if (inertia_f(lay32, N, kf, fmaf((float)mid, dcf, c0f)) >= 1) hi = mid;
        else lo = mid;
    }
    // the bounded counts, and where they disagree with the plain ones (thin
    // layers) a step towards them
#pragma unroll 1
    for (int tries = 0;; ++tries) {
        bool s_hi, s_lo = false;
        const int c_hi = count_bound_at(lay32, N, kf, c0, dc, hi, &s_hi);
        if (c_hi < 1 && hi == npf - 1) return r;  // no change inside the range
        int c_lo = 0;
        if (c_hi < 1 && tries < 4) {
            lo = hi++;
            continue;
        }
        if (lo >= 0) c_lo = count_bound_at(lay32, N, kf, c0, dc, lo, &s_lo);
        if (c_lo >= 1 && tries < 4) {
            hi = lo--;
            continue;
        }
        r.proof = (s_lo && c_lo == 0 ? PROOF_LO : 0) | (s_hi && (c_hi & 1) ? PROOF_HI : 0);
        r.count = c_hi;
        break;
    }
    r.n = hi;
    return r;
}

// The guess for an item between two searched wavelengths of its model
// (indices na, nb >= 1, d items apart; the item x after the first): the line
// through them, rounded down from a quarter point below it. A fundamental
// mode's phase velocity is smooth and convex in the wavelength's place on a
// log-spaced set, so the line overestimates: on a ragged batch of 8192 models
// this guess was the change or the point below it (two evaluations) for 85 %
// of the items, the rounded line for 65 % (a parabola through a third
// neighbour, 86 %, cost more in loads and divisions than it saved).
__device__ __forceinline__ int search_guess(int na, int nb, int x, int d) {
    // (a guess: a fast division, any rounding of it gives the same result)
    return __float2int_rd(
        fmaf(__fdividef((float)(nb - na), (float)d), (float)x, (float)na - 0.25f));
}

// The search stage for an item between two searched wavelengths of its
// model, from a guess g (search_guess). The count at g says on which
// side the change lies; steps of 1, 2, 4, ... from g away in that direction
// bracket it, and bisection closes the bracket: 2 evaluations when g is the
// change or the point below it, about 2 log2(e) + 2 for an error of e
// points. The result is the same first nonzero point of a non-decreasing
// count in [0, npf), or -1. Every point takes the bounded count, so that the
// two points of the result carry their proof with them (the plain count and
// two bounded ones after it took 25 % longer). One place evaluates, so the
// lanes of a warp stay together and the code compact.
__device__ __forceinline__ Located count_search_guess(const float* __restrict__ lay32, int N,
                                                      double k, double c0, double dc, int npf,
                                                      int guess) {
    Located r{-1, 0, 0};
    if (npf < 1) return r;
    const float kf = (float)k;
    int lo = -1, hi = npf;  // count 0 at lo (c = 0 when lo = -1), nonzero at hi (not seen: npf)
    int p = min(guess, npf - 1), step = 1;
    bool down = false;
    for (bool first = true;; first = false) {
        bool sure;
        const int c = count_bound_at(lay32, N, kf, c0, dc, p, &sure);
        if (c >= 1) {
            hi = p;
            r.count = c;
            r.proof = (r.proof & PROOF_LO) | ((sure && (c & 1)) ? PROOF_HI : 0);
        } else {
            lo = p;
            r.proof = (r.proof & PROOF_HI) | (sure ? PROOF_LO : 0);
        }
        if (first) down = c >= 1;
        if (hi - lo <= 1) break;
        if (down && lo < 0) {  // no lower end yet
            p = max(hi - step, 0);
            step *= 2;
        } else if (!down && hi == npf) {  // no upper end yet
            p = min(lo + step, npf - 1);
            step *= 2;
        } else {
            p = lo + ((hi - lo) >> 1);
        }
    }
    if (hi < npf) r.n = hi;  // else no change inside the range
    return r;
}

// The two searches by a group of G lanes per item, for batches too small to
// fill the GPU with a thread each: G points per step, so log_(G+1) instead of
// log_2 steps of one evaluation's latency. All lanes of a group (`gmask`, lane
// `gl`, first lane `g0` of the warp) call them together and get the same
// result.

// Lane i's point of G that split (lo, hi), hi - lo > 1; the step's points are
// lo + 1 .. hi - 1, and hi for lanes left over, once G reaches them all.
template <int G>
__device__ __forceinline__ int section_point(int lo, int hi, int i) {
    const int len = hi - lo;
    return len - 1 <= G ? min(lo + 1 + i, hi) : lo + (int)(((long long)len * (i + 1)) / (G + 1));
}

// count_search_single by a group.
template <int G>
__device__ __forceinline__ Located count_search_group(const float* __restrict__ lay32, int N,
                                                      double k, double c0, double dc, int npf,
                                                      int gl, int g0, unsigned gmask) {
    Located r{-1, 0, 0};
    if (npf < 1) return r;
    const float kf = (float)k, c0f = (float)c0, dcf = (float)dc;
    int lo = -1, hi = npf - 1;  // (the top is taken as nonzero until the end)
    while (hi - lo > 1) {
        const int p = section_point<G>(lo, hi, gl);
        const int c = p < hi ? inertia_f(lay32, N, kf, fmaf((float)p, dcf, c0f)) : 1;
        const unsigned m = (__ballot_sync(gmask, c >= 1) >> g0) & (G == 32 ? ~0u : (1u << G) - 1u);
        const int f = m ? __ffs(m) - 1 : G;  // first lane at or above the change
        const int top = __shfl_sync(gmask, p, g0 + min(f, G - 1)), below = __shfl_sync(gmask, p, g0 + max(f - 1, 0));
        if (f < G) hi = top;
        if (f > 0) lo = below;
    }
    // the bounded counts, even lanes V[lo], odd lanes V[hi], and where they
    // disagree with the plain ones (thin layers) a step towards them
    for (int tries = 0;; ++tries) {
        const int p = (gl & 1) ? hi : lo;
        bool sure = false;
        const int c = p >= 0 ? count_bound_at(lay32, N, kf, c0, dc, p, &sure) : 0;
        const int c_lo = __shfl_sync(gmask, c, g0), c_hi = __shfl_sync(gmask, c, g0 + 1);
        const bool s_lo = __shfl_sync(gmask, (int)sure, g0), s_hi = __shfl_sync(gmask, (int)sure, g0 + 1);
        if (c_hi < 1 && hi == npf - 1) return r;  // no change inside the range
        if (tries < 4 && c_hi < 1) {
            lo = hi++;
        } else if (tries < 4 && c_lo >= 1) {
            hi = lo--;
        } else {
            r.n = hi;
            r.proof = (s_lo && c_lo == 0 ? PROOF_LO : 0) | (s_hi && (c_hi & 1) ? PROOF_HI : 0);
            r.count = c_hi;
            return r;
        }
    }
}

// count_search_guess by a group of G lanes: first the points guess - 1 ..
// guess + G - 2 (the change lies among them for most items: one evaluation's
// latency), then steps of 4^i away on the side where it lies, then splits.
template <int G>
__device__ __forceinline__ Located count_search_guess_group(const float* __restrict__ lay32, int N,
                                                            double k, double c0, double dc, int npf,
                                                            int guess, int gl, int g0,
                                                            unsigned gmask) {
    Located r{-1, 0, 0};
    if (npf < 1) return r;
    const float kf = (float)k;
    int lo = -1, hi = npf, step = 4;  // hi = npf: not seen; lo = -1: c = 0
    bool s_lo = false, s_hi = false, first = true, up = false;
    for (;;) {
        int p;
        if (first) p = min(max(guess - 1 + gl, 0), npf - 1);
        else if (!up && lo < 0) p = max(hi - (step << (2 * (G - 1 - gl))), 0);
        else if (up && hi == npf) p = min(lo + (step << (2 * gl)), npf - 1);
        else p = section_point<G>(lo, hi, gl);
        bool sure = true;
        const int c = p < hi ? count_bound_at(lay32, N, kf, c0, dc, p, &sure) : 1;
        const unsigned m = (__ballot_sync(gmask, c >= 1) >> g0) & (G == 32 ? ~0u : (1u << G) - 1u);
        const int f = m ? __ffs(m) - 1 : G;
        const int a = g0 + min(f, G - 1), z = g0 + max(f - 1, 0);
        const int p_hi = __shfl_sync(gmask, p, a), p_lo = __shfl_sync(gmask, p, z);
        const int c_hi = __shfl_sync(gmask, c, a);
        const bool t_hi = __shfl_sync(gmask, (int)sure, a), t_lo = __shfl_sync(gmask, (int)sure, z);
        if (f < G && p_hi < hi) {
            hi = p_hi;
            s_hi = t_hi && (c_hi & 1);
            r.count = c_hi;
        }
        if (f > 0 && p_lo > lo && p_lo < hi) {
            lo = p_lo;
            s_lo = t_lo;
        }
        if (first) up = f == G;
        else step <<= 2 * G;
        if (step > (1 << 20)) step = 1 << 20;
        first = false;
        if (hi - lo <= 1) break;
    }
    if (hi < npf) r.n = hi;
    r.proof = (s_lo ? PROOF_LO : 0) | (s_hi ? PROOF_HI : 0);
    return r;
}

// The certificate stage for the search's index n (count_search_guess or
// count_search_single) in the
// pole-free range [0, npf). Both lanes of the pair (lane bit 0 = half, `pair`
// = their shuffle mask) call it with the same item and get the same result.
// Requires nlim >= 2.
__device__ __forceinline__ PairCount certify_pair(const float* __restrict__ lay32,
                                                  const float* __restrict__ laydf,
                                                  const double* __restrict__ lay, int N, double k,
                                                  double c0, double dc, int nlim, int npf, int n,
                                                  int half, unsigned pair) {
    const float kf = (float)k;
    const float c0f = (float)c0, dcf = (float)dc;
    PairCount out{-1, -1, 0, -1};
    if (npf < 1) return out;
    // the FP64 certificate decides the parity at the first nonzero point
    if (n < 0) {
        out.start = npf;  // no mode below the bound: scan linearly above it
        return out;
    }
    if (n < 1) return out;  // a mode below V[0]: Algorithm 1 from V[0]
    const int v = det_inertia_dd(laydf, lay, N, k, grid_c(c0, dc, n - 1 + half));
    const int vo = __shfl_xor_sync(pair, v, 1);
    const int va = half ? vo : v;  // V[n-1]
    const int vb = half ? v : vo;  // V[n]
    int cert = (va == 0 && vb > 0 && (vb & 1)) ? n : -1;
    int s_lo = va, s_hi = vb;  // the FP64 counts at cert - 1 and cert
    if (cert < 0 && va >= 0 && vb >= 0) {
        const bool up = va == 0 && vb == 0;
        const bool down = va > 0 && n >= 3;
        if (up || down) {
            const int p = (up ? n + 1 : n - 3) + half;
            // inside the pole-free range the Schur step in double-float, above it in FP64
            const int w = p >= nlim ? -1
                          : p < npf ? det_inertia_dd(laydf, lay, N, k, grid_c(c0, dc, p))
                                    : det_inertia_df(laydf, lay, N, k, grid_c(c0, dc, p));
            const int wo = __shfl_xor_sync(pair, w, 1);
            const int c_lo = half ? wo : w, c_hi = half ? w : wo;
            if (up) {
                // count 0 at n; first nonzero at n+1, or at n+2 with n+1 inside the range
                if (c_lo > 0) {
                    if (c_lo & 1) {
                        cert = n + 1;
                        s_lo = vb;
                        s_hi = c_lo;
                    }
                } else if (c_lo == 0 && c_hi > 0 && (c_hi & 1) && n + 1 < npf) {
                    cert = n + 2;
                    s_lo = c_lo;
                    s_hi = c_hi;
                }
            } else {
                // count nonzero at n-1; first nonzero at n-1 or n-2
                if (c_hi == 0) {
                    if (va & 1) {
                        cert = n - 1;
                        s_lo = c_hi;
                        s_hi = va;
                    }
                } else if (c_hi > 0 && c_lo == 0 && (c_hi & 1)) {
                    cert = n - 2;
                    s_lo = c_lo;
                    s_hi = c_hi;
                }
            }
        }
    }
    if (cert < 0 && va == 0 && vb >= 2 && !(vb & 1)) {
        // FP64: count 0 below n and even at n (two modes inside one interval,
        // no sign change there). The first change is the first point above n
        // whose count is odd: search for the first count above vb and certify
        // count vb one point below it (so vb, an even count, all the way from
        // n) and an odd count at it; otherwise the item falls back with start n.
        const int m = pair_search(lay32, N, kf, c0f, dcf, n, npf - 1, vb + 1, half, pair);
        if (m > n) {
            const int u = det_inertia_dd(laydf, lay, N, k, grid_c(c0, dc, m - 1 + half));
            const int uo = __shfl_xor_sync(pair, u, 1);
            const int ua = half ? uo : u, ub = half ? u : uo;
            if (ua == vb && ub > vb && (ub & 1)) {
                cert = m;
                s_lo = ua;
                s_hi = ub;
            }
        }
        if (cert < 0) {
            out.start = n;
            return out;
        }
    }
    out.cert = cert;
    out.n = cert >= 1 ? -1 : n;
    if (cert >= 1 && cert < npf) out.counts = pack_counts(s_lo, s_hi);
    return out;
}

}  // namespace masw
