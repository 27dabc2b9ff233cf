// Device parts shared by the two forms of the Gram–Schmidt step: group sums over
// a warp and the last step once the coefficients and the norm are known.
//
// A warp's FP64 instruction holds its scheduler's pipe for 64 clocks on this GPU
// whatever the number of active lanes, so sums over lanes are made for several
// values at a time and scalar code goes through as few FP64 operations as it can.
#pragma once

#include "fp64.cuh"
#include "gs.h"

namespace sim {

// Warp sums of G complex values at once: at each of log2(G) stages a lane keeps
// half of its values and trades the other half with its partner, so that G
// values take 2 (G - 1 + 5 - log2 G) additions instead of 10 G.  Afterwards lane
// l holds the sum of value l / (32 / G).
template <int G> __device__ __forceinline__ double2 warp_sum_group(double2 (&v)[G]) {
    const int lane = threadIdx.x & 31;
#pragma unroll
    for (int width = G, mask = 16; width > 1; width >>= 1, mask >>= 1) {
        const bool upper = (lane & mask) != 0;
        const int half = width >> 1;
#pragma unroll
        for (int i = 0; i < half; ++i) {
            const double2 send = upper ? v[i] : v[i + half];
            const double2 keep = upper ? v[i + half] : v[i];
            v[i].x = keep.x + __shfl_xor_sync(0xffffffffu, send.x, mask);
            v[i].y = keep.y + __shfl_xor_sync(0xffffffffu, send.y, mask);
        }
    }
#pragma unroll
    for (int mask = 16 / G; mask > 0; mask >>= 1) {
        v[0].x += __shfl_xor_sync(0xffffffffu, v[0].x, mask);
        v[0].y += __shfl_xor_sync(0xffffffffu, v[0].y, mask);
    }
    return v[0];
}

// c += conj(q) w
__device__ __forceinline__ void conj_mac(double2& c, double2 q, double2 w) {
    c.x = fma(q.x, w.x, c.x);
    c.x = fma(q.y, w.y, c.x);
    c.y = fma(q.x, w.y, c.y);
    c.y = fma(-q.y, w.x, c.y);
}

// v -= q h
__device__ __forceinline__ void sub_mac(double2& v, double2 q, double2 h) {
    v.x = fma(-q.x, h.x, v.x);
    v.x = fma(q.y, h.y, v.x);
    v.y = fma(-q.x, h.y, v.y);
    v.y = fma(-q.y, h.x, v.y);
}

// Calls f(group size tag, first index) over cnt vectors in groups of 8, 4, 2, 1.
template <int G> struct GroupTag {
    static constexpr int value = G;
};
template <class F> __device__ __forceinline__ void for_groups(int cnt, F f) {
    int i = 0;
    for (; i + 8 <= cnt; i += 8) f(GroupTag<8>{}, i);
    if (cnt - i >= 4) {
        f(GroupTag<4>{}, i);
        i += 4;
    }
    if (cnt - i >= 2) {
        f(GroupTag<2>{}, i);
        i += 2;
    }
    if (cnt - i >= 1) f(GroupTag<1>{}, i);
}

// The last step, by one whole warp: h[0..cnt) the coefficients (shared memory),
// hn the norm, broken whether it counts as a breakdown.
__device__ __forceinline__ void gs_finish(const GSArgs& a, int job, const double2* h, double hn, bool broken) {
    const int lane = threadIdx.x & 31;
    const GmArgs& gm = a.gm;
    if (gm.mode != GmArgs::STEP && a.hcol) {
        double2* hc = a.hcol + (size_t)job * a.hstride;
        for (int i = lane; i < a.cnt; i += 32) hc[i] = h[i];
        if (lane == 0) hc[a.cnt] = make_double2((broken && a.Hfull) ? 0.0 : hn, 0.0);
    }
    if (lane == 0 && broken) {
        if (a.meff) a.meff[job] = a.j + 1;
        if (a.istat) {
            a.istat[job * IS_N + IS_BROKEN] = 1;
            if (a.h_istat) a.h_istat[job * IS_N + IS_BROKEN] = 1;
        }
    }
    if (gm.mode == GmArgs::NONE) return;
    const int k = gm.k;
    double2* g = gm.g + (size_t)job * (k + 1);
    double* sc = gm.scal + (size_t)job * SC_N;
    int* is = gm.istat + (size_t)job * IS_N;
    if (gm.mode == GmArgs::START) {
        for (int i = lane; i <= k; i += 32) g[i] = make_double2(i == 0 ? hn : 0.0, 0.0);
        if (lane == 0) {
            if (gm.first) {
                sc[SC_RNORM0] = hn;
                is[IS_ITERS] = 0;
                is[IS_DONE] = 0;
                is[IS_STALL] = 0;
                is[IS_LOOSE] = 0;
            }
            sc[SC_GAMMA] = hn;
            sc[SC_RES] = hn;
            is[IS_STEPS] = 0;
            const int conv = !(hn > gm.tol * sc[SC_RNORM0]);
            is[IS_CYCLE_DONE] = conv;
            a.h_istat[job * IS_N + IS_CYCLE_DONE] = conv;
            if (conv) is[IS_DONE] = 1;
        }
        return;
    }
    // STEP: a job whose cycle has ended takes no further columns
    if (is[IS_CYCLE_DONE]) return;
    const int i = gm.i;
    double2* R = gm.Hg + (size_t)job * (k + 1) * k;
    double2* col = R + (size_t)i * (k + 1);
    double2* cs = gm.cs + (size_t)job * k;
    double2* sn = gm.sn + (size_t)job * k;
    // the earlier rotations, every lane the same
    double2 cur = h[0];
    for (int q = 0; q < i; ++q) {
        const double c = cs[q].x;
        const double2 s = sn[q], b = h[q + 1];
        const double2 up = make_double2(fma(-s.y, b.y, fma(s.x, b.x, c * cur.x)), fma(s.y, b.x, fma(s.x, b.y, c * cur.y)));
        cur = make_double2(fma(-s.y, cur.y, fma(-s.x, cur.x, c * b.x)), fma(s.y, cur.x, fma(-s.x, cur.y, c * b.y)));
        if (lane == 0) col[q] = up;
    }
    // the new one: c = |a| / nu, s = a hn / (|a| nu), nu^2 = |a|^2 + hn^2
    const double na2 = fma(cur.x, cur.x, cur.y * cur.y), nu2 = fma(hn, hn, na2);
    double c;
    double2 s;
    if (na2 > 1e-280 && nu2 < 1e280) {
        const double pr = rsqrt_nr(na2) * rsqrt_nr(nu2);
        c = na2 * pr;
        s = cscale(cur, hn * pr);
    } else {
        const double na = cabsd(cur);
        if (na == 0.0) {
            c = 0.0;
            s = make_double2(1.0, 0.0);
        } else {
            const double nu = hypot(na, hn);
            c = na / nu;
            s = cscale(cscale(cur, 1.0 / na), hn / nu);
        }
    }
    const double2 gi = g[i];
    const double2 diag = make_double2(fma(s.x, hn, cur.x * c), fma(s.y, hn, cur.y * c));
    const double2 gn = make_double2(-fma(s.x, gi.x, s.y * gi.y), -fma(s.x, gi.y, -(s.y * gi.x)));
    const double r2 = fma(gn.x, gn.x, gn.y * gn.y);
    const double res = r2 > 1e-280 && r2 < 1e280 ? r2 * rsqrt_nr(r2) : cabsd(gn);
    const int iters = is[IS_ITERS] + 1;
    const int done = (res <= gm.tol * sc[SC_RNORM0]) || !(hn > 0.0) || (i + 1 == k) || (iters >= gm.max_iter);
    __syncwarp();
    if (lane == 0) {
        col[i] = diag;
        col[i + 1] = make_double2(0.0, 0.0);
        cs[i] = make_double2(c, 0.0);
        sn[i] = s;
        g[i] = cscale(gi, c);
        g[i + 1] = gn;
        sc[SC_RES] = res;
        is[IS_STEPS] = i + 1;
        is[IS_ITERS] = iters;
        is[IS_CYCLE_DONE] = done;
        a.h_istat[job * IS_N + IS_CYCLE_DONE] = done;
    }
    if (!done) return;
    // R y = g, a row per lane, the diagonal's reciprocals first
    __syncwarp();
    const int steps = i + 1;
    double2 acc = make_double2(0.0, 0.0), inv = make_double2(0.0, 0.0);
    if (lane < steps) {
        acc = g[lane];
        const double2 d = R[(size_t)lane * (k + 1) + lane];
        if (d.x != 0.0 || d.y != 0.0) inv = cdiv(make_double2(1.0, 0.0), d);
    }
    for (int q = steps - 1; q >= 0; --q) {
        const double2 t = cmul(acc, inv);
        const double2 yq = make_double2(__shfl_sync(0xffffffffu, t.x, q), __shfl_sync(0xffffffffu, t.y, q));
        if (lane == q) gm.y[(size_t)job * k + q] = yq;
        if (lane < q) acc = csub(acc, cmul(R[(size_t)q * (k + 1) + lane], yq));
    }
}

// Breakdown test: hn <= btol ||H(0:j, 0:j)||_F, column j being h.  `sum` adds a
// value over the CTA.
template <class F>
__device__ __forceinline__ double hess_frobenius2(const GSArgs& a, int job, const double2* h, F sum) {
    const double2* H = a.Hfull + (size_t)job * a.Hstride;
    const int jj = a.j, rows = a.j + 1;
    double f = 0.0;
    for (int idx = threadIdx.x; idx < jj * rows; idx += blockDim.x)
        f += cabs2(H[(size_t)(idx / rows) * a.Hld + idx % rows]);
    for (int r = threadIdx.x; r < rows; r += blockDim.x) f += cabs2(h[r]);
    return sum(f);
}

}  // namespace sim
