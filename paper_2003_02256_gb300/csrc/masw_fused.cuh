// masw_fused.cuh -- the counting search and its certificate for many items in
// one kernel, block by block: the batch path's fused plan and the serving tick.
//
// Src gives an item's data by its position t and takes its outcome:
//   CountItem get(t); double c0(), dc(); int route() (test routing level);
//   none(t)             fewer than two points below the scan limit
//   fallback(t, start)  the linear FP32 scan from V[start]
//   done(t, n, s_lo, s_hi)  the first change n and the counts at V[n-1], V[n]
//   missed(t, n, from)  not certified; from: the count is even up to V[n]
#pragma once

#include "masw_count.cuh"

namespace masw {

constexpr unsigned FULL = 0xffffffffu;

struct CountItem {
    const float* lay32;
    const float* laydf;
    const double* lay;
    int N, nlim;
    double k;
};

// One warp, a group of DD_GROUP lanes per item (`on`): items whose counts va at
// V[n-1] and vb at V[n] are not the certificate's because the FP32 index is off
// by a point or two. Count 0 at both: the change is higher, the points above
// in turn; nonzero at V[n-1]: lower, the points below; inside the pole-free
// range, four points at most, each by det_inertia_dd_group; an even count at
// V[n]: the first odd one above. Otherwise the
// item is handed on (src.missed; from the last point known to have an even
// count, where V[n-1] has count 0). A few items in 100,000: the sign scan
// after the kernel would cost them, and the whole batch, about 90 us.
template <class Src>
static __device__ __noinline__ void certify_near(const Src& src, bool on, int t, int n, int va, int vb,
                                                 float* sh) {
    const CountItem it = src.get(t);
    const int N = it.N;
    const double k = it.k, c0 = src.c0(), dc = src.dc();
    const int npf = on ? pole_free_points_f(it.lay32, N, (float)k, (float)c0, (float)dc, it.nlim) : 0;
    const bool up = va == 0 && vb == 0, down = va > 0;
    // the point in hand and its count: 0 going up, nonzero going down
    int at = up ? n : n - 1, cnt = up ? 0 : va;
    int cert = -1, s_lo = 0, s_hi = 0;
    bool go = on && (up || down);
    for (int tries = 0; tries < 4; ++tries) {
        const int p = up ? at + 1 : at - 1;
        go = go && p >= 0 && p < npf;
        if (!__any_sync(FULL, go)) break;
        const int v = det_inertia_dd_group(it.laydf, it.lay, go ? N : 0, k,
                                           grid_c(c0, dc, max(p, 0)), sh);
        if (!go) continue;
        if (v < 0) {
            go = false;
        } else if (up) {
            if (v > 0) {
                if (v & 1) {
                    cert = p;
                    s_hi = v;
                }
                go = false;
            }
            if (v == 0 || !(v & 1)) at = p;  // an even count up to here
        } else if (v == 0) {
            if (cnt & 1) {
                cert = at;
                s_hi = cnt;
            }
            go = false;
        } else {
            at = p;
            cnt = v;
        }
    }
    // Two modes inside one interval (count 0, then even): the first odd count
    // above, located on the FP32 count by the group's lanes, with the even
    // count one point below it.
    bool even = on && va == 0 && vb >= 2 && !(vb & 1);
    if (__any_sync(FULL, even)) {
        const int gl = threadIdx.x & (DD_GROUP - 1), g0 = (threadIdx.x & 31) - gl;
        int lo = n, hi = npf - 1;
        even = even && hi > lo;
        for (;;) {
            const bool act = even && hi - lo > 1;
            if (!__any_sync(FULL, act)) break;
            const int p = act ? section_point<DD_GROUP>(lo, hi, gl) : 0;
            const int c = act && p < hi
                              ? inertia_f(it.lay32, N, (float)k, fmaf((float)p, (float)dc, (float)c0))
                              : vb + 1;
            const unsigned mk = (__ballot_sync(FULL, c > vb) >> g0) & ((1u << DD_GROUP) - 1u);
            const int f = mk ? __ffs(mk) - 1 : DD_GROUP;
            const int p_up = __shfl_sync(FULL, p, g0 + min(f, DD_GROUP - 1));
            const int p_dn = __shfl_sync(FULL, p, g0 + max(f - 1, 0));
            if (act && f < DD_GROUP) hi = p_up;
            if (act && f > 0) lo = p_dn;
        }
        const int ua = det_inertia_dd_group(it.laydf, it.lay, even && hi - 1 > n ? N : 0, k,
                                            grid_c(c0, dc, max(hi - 1, 0)), sh);
        const int ub = det_inertia_dd_group(it.laydf, it.lay, even ? N : 0, k, grid_c(c0, dc, max(hi, 0)), sh);
        if (even && (hi - 1 == n || ua == vb) && ub > vb && (ub & 1)) {
            cert = hi;
            s_lo = vb;
            s_hi = ub;
        }
    }
    if (!on || (threadIdx.x & (DD_GROUP - 1))) return;
    if (cert >= 1) {
        src.done(t, cert, s_lo, s_hi);
    } else {
        // an even count at V[n], or going up at `at`, else at V[n-1]
        src.missed(t, up ? at : (vb >= 0 && !(vb & 1)) ? n : n - 1, va == 0);
    }
}

// Items [begin, end), G lanes each: the search (count_search_group) with the
// FP32 bound's proofs; the points that the bound leaves open, a twentieth of
// them, are collected in shared memory and take the double-float count, 8
// lanes of the block each (det_inertia_dd_group): in the items' own lanes
// nearly every warp would hold one and run the double-float code for it. An
// item whose counts are not the certificate's takes certify_near; items the
// search cannot place go to src.fallback. Bound by latency: G splits the range
// in G + 1 per step. (A lane pair per item with a double-float count on each
// lane: one curve of 60 items 45 us, here 20; 9,600 items of 8 layers 94, here
// 57; 64,000 of 8 layers 175, here 125; 76,800 of 12 layers 300, here 190.)
// Launch bounds: 768 threads per SM for pairs (85 registers, 64,000 items 125
// us against 140 at 512), 512 for the wider groups, whose latency counts.
template <int B, int G, class Src>
__device__ __forceinline__ void count_fused_block(const Src& src, int begin, int end) {
    constexpr int ITEMS = B / G;
    __shared__ int s_n, s_open[2 * ITEMS], s_at[2 * ITEMS], s_count[2 * ITEMS];
    __shared__ __align__(8) float s_dd[B / DD_GROUP][DD_GROUP_FLOATS];
    const int tid = threadIdx.x;
    const int slot = tid / G, gl = tid & (G - 1), g0 = (tid & 31) - gl;
    const unsigned gmask = G == 32 ? FULL : ((1u << G) - 1u) << g0;
    const int t0 = begin + blockIdx.x * ITEMS, t = t0 + slot;
    const double c0 = src.c0(), dc = src.dc();
    if (tid == 0) s_n = 0;
    __syncthreads();
    Located r{-1, 0, 0};
    bool open = false;  // leader lane: counts still wanted
    if (t < end) {
        const CountItem it = src.get(t);
        int npf = 0;
        if (it.nlim >= 2) {
            npf = pole_free_points_f(it.lay32, it.N, (float)it.k, (float)c0, (float)dc, it.nlim);
            r = count_search_group<G>(it.lay32, it.N, it.k, c0, dc, npf, gl, g0, gmask);
        }
        if (gl == 0) {
            if (it.nlim < 2) {
                src.none(t);
            } else if (r.n < 1 || src.route() >= 1) {
                // the start of the linear FP32 scan: the end of the range when
                // it holds no change, else (test routing too) V[0]
                src.fallback(t, (src.route() < 1 && npf >= 1 && r.n < 0) ? npf : 0);
            } else {
                open = true;
                s_count[2 * slot] = 0;
                s_count[2 * slot + 1] = r.count;
                for (int side = 0; side < 2; ++side)
                    if (!(r.proof & (side ? PROOF_HI : PROOF_LO))) {
                        const int q = atomicAdd(&s_n, 1);
                        s_open[q] = 2 * slot + side;
                        s_at[q] = r.n - 1 + side;
                    }
            }
        }
    }
    __syncthreads();
    for (int q0 = 4 * (tid >> 5); q0 < s_n; q0 += B / DD_GROUP) {  // a warp's four groups
        const int q = q0 + ((tid & 31) / DD_GROUP);
        const bool mine = q < s_n;
        const int e = s_open[mine ? q : q0];
        const CountItem it = src.get(t0 + (e >> 1));
        const int v = det_inertia_dd_group(it.laydf, it.lay, mine ? it.N : 0, it.k,
                                           grid_c(c0, dc, s_at[mine ? q : q0]), s_dd[tid / DD_GROUP]);
        if (mine && (tid & (DD_GROUP - 1)) == 0) s_count[e] = v;
    }
    __syncthreads();
    if (tid == 0) s_n = 0;
    __syncthreads();
    if (open) {
        const int va = s_count[2 * slot], vb = s_count[2 * slot + 1];
        if (va == 0 && vb > 0 && (vb & 1)) {
            src.done(t, r.n, va, vb);
        } else {
            const int q = atomicAdd(&s_n, 1);
            s_open[q] = slot;
            s_at[q] = r.n;
        }
    }
    __syncthreads();
    for (int q0 = 4 * (tid >> 5); q0 < s_n; q0 += B / DD_GROUP) {
        const int q = q0 + ((tid & 31) / DD_GROUP);
        const bool mine = q < s_n;
        const int e = s_open[mine ? q : q0];
        certify_near(src, mine, t0 + e, s_at[mine ? q : q0], s_count[2 * e], s_count[2 * e + 1],
                     s_dd[tid / DD_GROUP]);
    }
}

}  // namespace masw
