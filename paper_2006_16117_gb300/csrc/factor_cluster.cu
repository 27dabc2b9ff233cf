// Block-tridiagonal factorisation of K = A - σB on thread-block clusters.
//
// Same factors as k_factor (krylov.cu): the blocks are eliminated from both ends
// to the middle block mid, Dinv_k = D_k^{-1} with
//   D_k = K_kk - K_{k,outer(k)} E_{outer(k)}   (mid: minus both neighbours' terms),
//   E_k = Dinv_k K_{k,inner(k)},
// plus the shifted values of the outer couplings.  The blocks of a side form a
// serial chain and every block is T pivots long, so the time of a pivot bounds
// the factorisation, and two sides halve it: one launch factors the sides, one
// cluster each, and a second one the middle block of every shift.
//
// A cluster of Cf CTAs factors one side of one shift.  CTA q keeps Tc columns of D_k (all
// T rows) in shared memory, so a pivot search never leaves its CTA.  The
// in-place Gauss-Jordan inversion runs in panels of B columns:
//   panel   the owner's threads hold one row of the panel each, in registers;
//           a pivot (the largest |re|+|im| of the rows not used yet, ties to the
//           lower row) costs one warp reduction per 32 rows and one barrier of
//           the panel's warps (none with one warp; two in FP64 with more than four,
//           where only the winner's warp divides: an FP64 warp instruction holds its
//           scheduler's pipe for 64 clocks).  The
//           panel becomes G: column j is what the panel's pivots make of unit
//           vector e_{r_j}, r_j the row of pivot j.
//   update  every CTA, its other columns: R = the pivot rows' old values,
//           S[r][c] = (r a pivot row ? 0 : S[r][c]) + Σ_j G[r][j] R[j][c],
//           one row and CT columns per lane.
// The owner of the next panel updates that panel's columns first and factors it
// with its panel warps while its other warps (and the other CTAs) do the rest of
// the update: the chain of a panel is its pivots, not the update.  G reaches the
// other CTAs through global memory (L2; it uses the block's own E, which is
// written later), the pivot rows through distributed shared memory, and one
// cluster barrier per panel, split into arrive and wait around the update,
// publishes both.  No rows are swapped: the inverse comes out with its rows and
// columns permuted, Dinv[p][r_j] = S[r_p][j], and is stored that way round.
//
// Panels of 16 columns in complex64 (8 where shared memory is short) and 4 in
// complex128: the panel's own multiply-adds, T·B·B of them on one SM, are cheap
// in FP32 and as dear as the whole update in FP64.
//
// Measured for one shift, T = 200, nb = 200 complex64: 138 ms with rows over the
// cluster and two cluster barriers a pivot, 39.7 with the panels (2,050 clocks a
// pivot, about 1,000 of them the pivot itself), 20.1 from both ends, 16.3 on 13 CTAs
// a side; T = 98, nb = 97 complex128: 106, 31.6, 16.0, 12.7 ms; T = 30, nb = 30
// complex128: 5.6, 2.2, 1.2, 0.97 ms.  56 shifts of T = 200 complex64: 372 -> 53 ms.
#include <cooperative_groups.h>

#include <algorithm>
#include <map>
#include <mutex>
#include <tuple>

#include "internal.h"
#include "factor_cluster.h"
#include "fp64.cuh"

namespace cg = cooperative_groups;

namespace sim {

namespace {

template <class C> __device__ __forceinline__ C zc();
template <> __device__ __forceinline__ double2 zc<double2>() { return make_double2(0.0, 0.0); }
template <> __device__ __forceinline__ float2 zc<float2>() { return make_float2(0.f, 0.f); }

__device__ __forceinline__ double2 sval(const Pencil& P, int64_t e, double2 sg) {
    const double2 a = P.Ka[e], b = P.Kb[e];
    return make_double2(a.x - (sg.x * b.x - sg.y * b.y), a.y - (sg.x * b.y + sg.y * b.x));
}

// pivot magnitude |re| + |im| in the factor's own precision
template <class C> __device__ __forceinline__ auto m1(C a) -> decltype(a.x) { return fabs(a.x) + fabs(a.y); }

__device__ __forceinline__ void cluster_arrive() { asm volatile("barrier.cluster.arrive.release;" ::: "memory"); }
__device__ __forceinline__ void cluster_wait() { asm volatile("barrier.cluster.wait.acquire;" ::: "memory"); }
__device__ __forceinline__ void bar_panel(int threads) {
    asm volatile("bar.sync 1, %0;" ::"r"(threads) : "memory");
}

// one row of B values from shared memory, every lane the same (16-byte loads)
template <int B> __device__ __forceinline__ void load_row(const float2* p, float2 (&v)[B]) {
#pragma unroll
    for (int j = 0; j < B; j += 2) {
        const float4 t = *reinterpret_cast<const float4*>(p + j);
        v[j] = make_float2(t.x, t.y);
        v[j + 1] = make_float2(t.z, t.w);
    }
}
template <int B> __device__ __forceinline__ void load_row(const double2* p, double2 (&v)[B]) {
#pragma unroll
    for (int j = 0; j < B; ++j) v[j] = p[j];
}
template <int B> __device__ __forceinline__ void store_row(float2* p, const float2 (&v)[B]) {
#pragma unroll
    for (int j = 0; j < B; j += 2) *reinterpret_cast<float4*>(p + j) = make_float4(v[j].x, v[j].y, v[j + 1].x, v[j + 1].y);
}
template <int B> __device__ __forceinline__ void store_row(double2* p, const double2 (&v)[B]) {
#pragma unroll
    for (int j = 0; j < B; ++j) p[j] = v[j];
}
__device__ __forceinline__ float2 neg(float2 a) { return make_float2(-a.x, -a.y); }
// in complex128 by integer operations: negations and comparisons go through the FP64 pipe
__device__ __forceinline__ double neg(double a) {
    return __hiloint2double(__double2hiint(a) ^ (int)0x80000000, __double2loint(a));
}
__device__ __forceinline__ double2 neg(double2 a) { return make_double2(neg(a.x), neg(a.y)); }
__device__ __forceinline__ bool is_zero(float2 a) { return a.x == 0.f && a.y == 0.f; }
__device__ __forceinline__ bool is_zero(double2 a) {
    return (((uint32_t)(__double2hiint(a.x) | __double2hiint(a.y)) << 1) | (uint32_t)__double2loint(a.x) |
            (uint32_t)__double2loint(a.y)) == 0u;
}

constexpr int FC_MAXW = 16;  // panel warps: T <= 512 rows

// Sums over j of G[j][r] R[j][c] for RT rows (32 apart) and CT columns of a lane:
// packed FP32 pairs in complex64 (pa = Σ (g.x, g.x)·r, pb = Σ (g.y, g.y)·r,
// g r = (pa.x - pb.y, pa.y + pb.x)).  Two rows per lane halve the loads of R.
template <int RT, int CT>
__device__ __forceinline__ void gr_product(const float2* const (&G)[RT], const float2* R, int bw, int T, int ldr,
                                           float2 (&v)[RT][CT]) {
    float2 pa[RT][CT], pb[RT][CT];
#pragma unroll
    for (int r = 0; r < RT; ++r)
#pragma unroll
        for (int c = 0; c < CT; ++c) pa[r][c] = pb[r][c] = make_float2(0.f, 0.f);
#pragma unroll 2
    for (int j = 0; j < bw; ++j) {
        float2 gx[RT], gy[RT];
#pragma unroll
        for (int r = 0; r < RT; ++r) {
            const float2 g = G[r][(size_t)j * T];
            gx[r] = make_float2(g.x, g.x);
            gy[r] = make_float2(g.y, g.y);
        }
        const float4* Rj = reinterpret_cast<const float4*>(R + (size_t)j * ldr);
#pragma unroll
        for (int c = 0; c < CT; c += 2) {
            const float4 q = Rj[c / 2];
            const float2 q0 = make_float2(q.x, q.y), q1 = make_float2(q.z, q.w);
#pragma unroll
            for (int r = 0; r < RT; ++r) {
                pa[r][c] = __ffma2_rn(gx[r], q0, pa[r][c]);
                pb[r][c] = __ffma2_rn(gy[r], q0, pb[r][c]);
                pa[r][c + 1] = __ffma2_rn(gx[r], q1, pa[r][c + 1]);
                pb[r][c + 1] = __ffma2_rn(gy[r], q1, pb[r][c + 1]);
            }
        }
    }
#pragma unroll
    for (int r = 0; r < RT; ++r)
#pragma unroll
        for (int c = 0; c < CT; ++c) v[r][c] = make_float2(pa[r][c].x - pb[r][c].y, pa[r][c].y + pb[r][c].x);
}
template <int RT, int CT>
__device__ __forceinline__ void gr_product(const double2* const (&G)[RT], const double2* R, int bw, int T, int ldr,
                                           double2 (&v)[RT][CT]) {
#pragma unroll
    for (int r = 0; r < RT; ++r)
#pragma unroll
        for (int c = 0; c < CT; ++c) v[r][c] = make_double2(0.0, 0.0);
    for (int j = 0; j < bw; ++j) {
        double2 g[RT];
#pragma unroll
        for (int r = 0; r < RT; ++r) g[r] = G[r][(size_t)j * T];
#pragma unroll
        for (int c = 0; c < CT; ++c) {
            const double2 q = R[(size_t)j * ldr + c];
#pragma unroll
            for (int r = 0; r < RT; ++r) v[r][c] = cfma(g[r], q, v[r][c]);
        }
    }
}

// Runs f.load(i, c) and f.use(i, c, loaded) for every element (i, c) of a rows ×
// cols array, the block's threads over consecutive elements, 8 loads of a thread
// in flight before their first use.
template <class F> __device__ __forceinline__ void for_elements(int rows, int cols, F f) {
    constexpr int U = 8;
    const int nt = blockDim.x;
    const int di = nt / cols, dc = nt - di * cols;
    int i = threadIdx.x / cols, c = threadIdx.x - i * cols;
    while (i < rows) {
        typename F::Value v[U];
        int ii[U], cc[U];
#pragma unroll
        for (int u = 0; u < U; ++u) {
            ii[u] = i;
            cc[u] = c;
            if (i < rows) v[u] = f.load(i, c);
            i += di;
            c += dc;
            if (c >= cols) {
                c -= cols;
                ++i;
            }
        }
#pragma unroll
        for (int u = 0; u < U; ++u)
            if (ii[u] < rows) f.use(ii[u], cc[u], v[u]);
    }
}

// S -= K_{k,outer} E_outer, my columns (Ep and for mid's second neighbour Ep2 at my
// first column); each row's first coupling is staged
template <class C> struct SubCouplings {
    using Value = C;
    C* S;
    int ld, T;
    const C *Ep, *Ep2;
    const C* l0v;
    const int *l0c, *llo, *lhi;
    const C* Lval;
    const int32_t* Lcol;
    __device__ __forceinline__ C at(int col, int c) const {
        return col < T ? Ep[(size_t)col * T + c] : Ep2[(size_t)(col - T) * T + c];
    }
    __device__ __forceinline__ C load(int i, int c) const { return at(l0c[i], c); }
    __device__ __forceinline__ void use(int i, int c, C v) const {
        C acc = cmul(l0v[i], v);
        for (int e = llo[i]; e < lhi[i]; ++e) acc = cfma(Lval[e], at(Lcol[e], c), acc);
        S[(size_t)i * ld + c] = csub(S[(size_t)i * ld + c], acc);
    }
};

// E_k = Dinv_k K_{k,inner}, my columns; each column's first coupling is staged
template <class C> struct FormE {
    using Value = C;
    const Pencil& P;
    double2 sg;
    int T;
    const C* Dk;
    C* Ek;
    const C* l0v;
    const int *l0c, *llo, *lhi;
    __device__ __forceinline__ C load(int p, int c) const { return __ldcg(Dk + (size_t)p * T + l0c[c]); }
    __device__ __forceinline__ void use(int p, int c, C v) const {
        C acc = cmul(v, l0v[c]);
        for (int e = llo[c]; e < lhi[c]; ++e)
            acc = cfma(__ldcg(Dk + (size_t)p * T + P.up_row[e]), from_c128<C>(sval(P, P.up_idx[e], sg)), acc);
        Ek[(size_t)p * T + c] = acc;
    }
};

}  // namespace

template <class C, int B, int CT, int NT>
__global__ void __launch_bounds__(NT, 1) k_factor_cl(Pencil P, const int* shift_list, const double2* sigma,
                                                      void* const* fptrs, int* err, int Tc, int phase) {
    cg::cluster_group cl = cg::this_cluster();
    const int Cf = (int)cl.num_blocks();
    const int q = (int)cl.block_rank();
    const int T = P.T, nb = P.nb, mid = P.mid;
    // phase 0: blocks 0 .. mid-1 (side 0) or nb-1 .. mid+1 (side 1, launched if there
    // are any); phase 1: block mid
    const int sides = phase == 0 && mid + 1 < nb ? 2 : 1, side = (int)(blockIdx.x / Cf) % sides;
    const int len = phase ? 1 : (side ? nb - 1 - mid : mid);
    const int kfirst = phase ? mid : (side ? nb - 1 : 0), kstep = side ? -1 : 1;
    const int s = shift_list[blockIdx.x / Cf / sides];
    C* Dinv = reinterpret_cast<C*>(fptrs[s]);
    C* E = Dinv + (size_t)nb * T * T;
    C* Lval = Dinv + factor_lval_offset(P);
    const double2 sg = sigma[s];
    const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5, nw = blockDim.x >> 5, nt = blockDim.x;
    const int c0 = q * Tc, myc = max(0, min(Tc, T - c0)), ld = Tc + 1;
    const int np = (T + B - 1) / B, PW = (T + 31) / 32, ncg = Tc / CT;

    extern __shared__ __align__(16) unsigned char raw[];
    C* R = reinterpret_cast<C*>(raw);          // [B][Tc] pivot rows, old values
    C* cand = R + (size_t)B * Tc;              // [2][FC_MAXW][B] candidate pivot rows
    uint4* ckey = reinterpret_cast<uint4*>(cand + (size_t)2 * FC_MAXW * B);  // [2][FC_MAXW] their keys and rows
    C* Gs = reinterpret_cast<C*>(ckey + 2 * FC_MAXW);  // [2][B][T]
    C* l0v = Gs + (size_t)2 * B * T;           // [T] first coupling's value of a row of L
    C* u0v = l0v + T;                          // [Tc] first coupling's value of a column of U
    C* s_inv = u0v + Tc;                       // [1] (+1)
    C* S = s_inv + 2;                          // [T][ld], ld odd: lanes on rows or on columns without conflicts
    int* piv_row = reinterpret_cast<int*>(S + (size_t)T * ld + ((size_t)T * ld & 1));  // [T] row of pivot p
    int* l0c = piv_row + T;                    // [T]
    int* llo = l0c + T;                        // [T] further couplings [llo, lhi)
    int* lhi = llo + T;                        // [T]
    int* used = lhi + T;                       // [T]
    int* u0c = used + T;                       // [Tc], and of a column of U
    int* ulo = u0c + Tc;                       // [Tc]
    int* uhi = ulo + Tc;                       // [Tc]
    int* pnew = uhi + Tc;                      // [B] pivot rows of the panel being factored
    int* ctr = pnew + B;

    {
        // the couplings of my rows
        const int klo = side ? kfirst - (len - 1) : kfirst;
        const int64_t g_lo = (int64_t)klo * T, g_hi = min(P.n, (int64_t)(klo + len) * T);
        const int64_t e_hi = P.Lptr[g_hi];
        for (int64_t e = P.Lptr[g_lo] + tid + (int64_t)q * nt; e < e_hi; e += (int64_t)nt * Cf)
            Lval[e] = from_c128<C>(sval(P, P.Lidx[e], sg));
    }
    if (Cf > 1) {
        cluster_arrive();
        cluster_wait();
    }
    __syncthreads();

    // Gauss-Jordan on panel i in the registers of the first PW warps (row tid).
    // The pivot's column is always a[0]: a pivot turns the columns round by one (the
    // new column goes last), so the loop's body is short enough to stay in the
    // instruction cache; unrolled over the pivots it was bound by instruction fetch
    // (2,270 clocks a pivot of 16 columns).
    auto panel = [&](int i, C* scr) {
        const int p0 = i * B, bw = min(B, T - p0), lc = p0 - c0;
        const int r = tid;
        C a[B];
#pragma unroll
        for (int j = 0; j < B; ++j) a[j] = (r < T && j < bw) ? S[(size_t)r * ld + lc + j] : zc<C>();
        bool avail = r < T && used[min(r, T - 1)] == 0;
        // the warp's largest |re|+|im| of the rows not used yet, as an ordered key
        bool win;
        uint32_t mh, ml = 0;
        auto search = [&](C v) {
            if constexpr (sizeof(C) == 8) {
                const uint32_t key = avail ? max(__float_as_uint(m1(v)), 1u) : 0u;
                mh = __reduce_max_sync(0xffffffffu, key);
                win = avail && key == mh;
            } else {
                const long long w = __double_as_longlong(m1(v));
                const uint32_t hi = avail ? (uint32_t)(w >> 32) + 1u : 0u, lo = (uint32_t)w;
                mh = __reduce_max_sync(0xffffffffu, hi);
                ml = __reduce_max_sync(0xffffffffu, avail && hi == mh ? lo : 0u);
                win = avail && hi == mh && lo == ml;
            }
        };
        search(a[0]);
#pragma unroll 1
        for (int jj = 0; jj < bw; ++jj) {
            const int bo = (jj & 1) * FC_MAXW;
            const uint32_t ball = __ballot_sync(0xffffffffu, win);
            const int wl = ball == 0u ? 0 : __ffs(ball) - 1;
            if (lane == wl) {
                if (PW > 1) ckey[bo + warp] = make_uint4(ball ? mh : 0u, ml, (uint32_t)r, 0u);
                store_row<B>(cand + (size_t)(bo + warp) * B, a);
            }
            int ws = 0, row = wl;
            if (PW == 1) {
                __syncwarp();
            } else {
                bar_panel(PW * 32);
                // the winner among the warps' candidates: largest key, lowest warp (lowest row)
                const uint4 ck = ckey[bo + (lane < PW ? lane : 0)];
                const uint32_t wh = __reduce_max_sync(0xffffffffu, ck.x);
                bool wm = ck.x == wh;
                if constexpr (sizeof(C) == 16) {
                    const uint32_t wl = __reduce_max_sync(0xffffffffu, wm ? ck.y : 0u);
                    wm = wm && ck.y == wl;
                }
                ws = __ffs(__ballot_sync(0xffffffffu, wm)) - 1;
                row = (int)__shfl_sync(0xffffffffu, ck.z, ws);
            }
            C pr[B];
            load_row<B>(cand + (size_t)(bo + ws) * B, pr);
            if (is_zero(pr[0])) {  // singular Schur complement
                pr[0].x = (decltype(pr[0].x))1e-30;
                if (tid == 0) atomicExch(err, 1);
            }
            C inv;
            if (sizeof(C) == 8 || PW <= 4) {  // (four: a warp per scheduler)
                inv = crecip(pr[0]);
            } else {
                if (warp == ws) {
                    inv = crecip(pr[0]);
                    if (lane == 0) *s_inv = inv;
                }
                bar_panel(PW * 32);
                inv = *s_inv;
            }
            if (tid == 0) pnew[jj] = row;
            // row - g (pivot row), or for the pivot row itself 0 - (-1/pivot)(pivot row)
            const bool mine = r == row;
            if (mine) {
                avail = false;
                used[r] = 1;
            }
            C g = cmul(a[0], inv);
            if (mine) g = neg(inv);
            // the next pivot's column first: its search runs under the other columns' FMAs
#pragma unroll
            for (int j = 1; j < B; ++j) {
                C v = mine ? zc<C>() : a[j];
                v.x = fma(-g.x, pr[j].x, v.x);
                v.x = fma(g.y, pr[j].y, v.x);
                v.y = fma(-g.x, pr[j].y, v.y);
                v.y = fma(-g.y, pr[j].x, v.y);
                a[j - 1] = v;
                if (j == 1) search(v);
            }
            a[B - 1] = neg(g);
        }
        bar_panel(PW * 32);  // pnew complete
        // (a remote store inside the pivot loop would hold up its barriers)
        for (int e = tid; e < bw * Cf; e += PW * 32) *cl.map_shared_rank(piv_row + p0 + e % bw, e / bw) = pnew[e % bw];
        if (r < T) {
            C* Go = Gs + (size_t)(i & 1) * B * T;
#pragma unroll
            for (int j = 0; j < B; ++j) {
                const int c = j - (B - bw);  // after bw turns
                if (c >= 0) {
                    Go[(size_t)c * T + r] = a[j];
                    S[(size_t)r * ld + lc + c] = a[j];
                    if (Cf > 1) scr[(size_t)(p0 + c) * T + r] = a[j];
                }
            }
        }
    };

    // S += G R on a tile of rows and columns lc .. lc + CT - 1: 64 rows (two per
    // lane) for the first T / 64 tiles, then 32
    const int n64 = T / 64, ntr = n64 + (T - 64 * n64 + 31) / 32;
    auto update_tile = [&](const C* G, int bw, int rt, int lc) {
        if (rt < n64) {
            const int r = rt * 64 + lane;
            const C* const Gr[2] = {G + r, G + r + 32};
            C v[2][CT];
            gr_product<2, CT>(Gr, R + lc, bw, T, Tc, v);
#pragma unroll
            for (int h = 0; h < 2; ++h) {
                C* Sr = S + (size_t)(r + 32 * h) * ld + lc;
#pragma unroll
                for (int c = 0; c < CT; ++c) Sr[c] = cadd(Sr[c], v[h][c]);
            }
        } else {
            const int r = n64 * 64 + (rt - n64) * 32 + lane;
            const C* const Gr[1] = {G + min(r, T - 1)};
            C v[1][CT];
            gr_product<1, CT>(Gr, R + lc, bw, T, Tc, v);
            if (r < T) {
                C* Sr = S + (size_t)r * ld + lc;
#pragma unroll
                for (int c = 0; c < CT; ++c) Sr[c] = cadd(Sr[c], v[0][c]);
            }
        }
    };

    // the same for one element: FP64, where whole warps of work count and loads do not
    auto update_element = [&](const C* G, int bw, int r, int c) {
        C v = S[(size_t)r * ld + c];
        for (int j = 0; j < bw; ++j) v = cfma(G[(size_t)j * T + r], R[(size_t)j * Tc + c], v);
        S[(size_t)r * ld + c] = v;
    };

    for (int t = 0; t < len; ++t) {
        const int k = kfirst + t * kstep;
        const int64_t g0 = (int64_t)k * T;
        C* Dk = Dinv + (size_t)k * T * T;
        C* scr = E + (size_t)k * T * T;  // G's way to the other CTAs (E_mid's place is free)
        // 1. my columns of D_k = K_kk - K_{k,outer} E_outer
        for (int idx = tid; idx < T * ld; idx += nt) S[idx] = zc<C>();
        for (int i = tid; i < T; i += nt) {
            const int64_t g = g0 + i;
            used[i] = 0;
            int lo = 0, hi = 0, col = 0;
            C v = zc<C>();
            if (g < P.n) {
                lo = P.Lptr[g];
                hi = P.Lptr[g + 1];
                if (hi > lo) {
                    col = P.Lcol[lo];
                    v = Lval[lo];
                }
            }
            l0c[i] = col;
            l0v[i] = v;
            llo[i] = lo + 1;
            lhi[i] = hi;
        }
        if (k != mid) {  // the first coupling of my columns of K_{k,inner}, for step 4
            const int32_t* cp = P.up_ptr + (size_t)k * (T + 1);
            for (int c = tid; c < myc; c += nt) {
                const int lo = cp[c0 + c], hi = cp[c0 + c + 1];
                u0c[c] = hi > lo ? P.up_row[lo] : 0;
                u0v[c] = hi > lo ? from_c128<C>(sval(P, P.up_idx[lo], sg)) : zc<C>();
                ulo[c] = lo + 1;
                uhi[c] = hi;
            }
        }
        __syncthreads();
        for (int i = tid; i < T; i += nt) {
            const int64_t g = g0 + i;
            if (g < P.n) {
                const int64_t e1 = P.rp[g + 1];
                for (int64_t e = P.rp[g]; e < e1; e += 4) {  // 4 entries' loads in flight
                    int64_t lc[4];
                    C v[4];
#pragma unroll
                    for (int u = 0; u < 4; ++u) {
                        lc[u] = e + u < e1 ? (int64_t)P.ci[e + u] - g0 - c0 : -1;
                        v[u] = e + u < e1 ? from_c128<C>(sval(P, e + u, sg)) : zc<C>();
                    }
#pragma unroll
                    for (int u = 0; u < 4; ++u)
                        if (lc[u] >= 0 && lc[u] < myc) S[(size_t)i * ld + lc[u]] = v[u];
                }
            } else if (i >= c0 && i < c0 + myc) {
                S[(size_t)i * ld + (i - c0)] = from_c128<C>(make_double2(1.0, 0.0));
            }
        }
        __syncthreads();
        if ((phase ? nb > 1 : t > 0) && myc > 0) {
            // my columns, written by this CTA (phase 1: by the launch before)
            const C* Ep = E + (size_t)(phase ? max(mid - 1, 0) : k - kstep) * T * T + c0;
            const C* Ep2 = E + (size_t)min(mid + 1, nb - 1) * T * T + c0;
            for_elements(T, myc, SubCouplings<C>{S, ld, T, Ep, Ep2, l0v, l0c, llo, lhi, Lval, P.Lcol});
        }
        __syncthreads();
        // 2. Gauss-Jordan in panels
        if (q == 0 && warp < PW) panel(0, scr);
        if (Cf > 1) {
            cluster_arrive();
            cluster_wait();
        }
        __syncthreads();
        for (int i = 0; i < np; ++i) {
            const int p0 = i * B, bw = min(B, T - p0), own = p0 / Tc;
            const bool more = i + 1 < np, next = more && (p0 + B) / Tc == q;
            C* G = Gs + (size_t)(i & 1) * B * T;
            if (own != q) {  // T even: whole 16-byte units
                const float4* src = reinterpret_cast<const float4*>(scr + (size_t)p0 * T);
                float4* dst = reinterpret_cast<float4*>(G);
                const int units = (int)((size_t)bw * T * sizeof(C) / 16);
#pragma unroll 4
                for (int idx = tid; idx < units; idx += nt) dst[idx] = __ldcg(src + idx);
            }
            if (tid < bw) used[piv_row[p0 + tid]] = 1;
            const int lp = own == q ? p0 - c0 : -B;           // my columns of this panel
            const int ln = next ? p0 + B - c0 : -B;           // and of the next one
            for (int idx = tid; idx < bw * Tc; idx += nt) {
                const int j = idx / Tc, c = idx - j * Tc;
                if (c >= lp && c < lp + B) continue;
                C* Sr = S + (size_t)piv_row[p0 + j] * ld + c;
                R[idx] = *Sr;
                *Sr = zc<C>();
            }
            if (tid == 0) *ctr = 0;
            __syncthreads();
            if (next) {
                if constexpr (sizeof(C) == 16) {
                    for (int idx = tid; idx < T * B; idx += nt) update_element(G, bw, idx % T, ln + idx / T);
                } else {
                    for (int t = warp; t < ntr * (B / CT); t += nw) update_tile(G, bw, t % ntr, ln + (t / ntr) * CT);
                }
                __syncthreads();
                if (warp < PW) panel(i + 1, scr);
            }
            if (Cf > 1 && more) cluster_arrive();
            while (true) {
                int t = 0;
                if (lane == 0) t = atomicAdd(ctr, 1);
                t = __shfl_sync(0xffffffffu, t, 0);
                if constexpr (sizeof(C) == 16) {
                    // elements in runs of 32 over the columns but the panels' own
                    const int first = own == q ? lp : ln;
                    const int skip = min((own == q ? B : 0) + (next ? B : 0), myc - first);
                    const int cols = myc - skip;
                    if (t * 32 >= T * cols) break;
                    const int idx = t * 32 + lane, c = idx / T;
                    if (c < cols) update_element(G, bw, idx - c * T, skip > 0 && c >= first ? c + skip : c);
                } else {
                    if (t >= ntr * ncg) break;
                    const int lc = (t / ntr) * CT;
                    if (lc >= myc || (lc >= lp && lc < lp + B) || (lc >= ln && lc < ln + B)) continue;
                    update_tile(G, bw, t % ntr, lc);
                }
            }
            if (Cf > 1 && more) cluster_wait();
            __syncthreads();
        }
        // 3. Dinv_k[p][r_j] = S[r_p][j] for my columns j
        for (int p = warp; p < T; p += nw) {
            const C* Sp = S + (size_t)piv_row[p] * ld;
            for (int c = lane; c < myc; c += 32) Dk[(size_t)p * T + piv_row[c0 + c]] = Sp[c];
        }
        if (Cf > 1) {
            cluster_arrive();
            cluster_wait();
        }
        __syncthreads();
        // 4. my columns of E_k = Dinv_k K_{k,inner}
        if (k != mid && myc > 0) {
            C* Ek = E + (size_t)k * T * T + c0;
            for_elements(T, myc, FormE<C>{P, sg, T, Dk, Ek, u0v, u0c, ulo, uhi});
            __syncthreads();
        }
    }
}

namespace {
int* g_ferr = nullptr;

// shared memory that a slice of rows needs in the widest admitted launch: the
// rule that decides between this kernel and k_factor
size_t admit_bytes(int T, size_t cs) {
    const int Tc = (T + 7) / 8;
    return (size_t)Tc * T * cs + T * cs + (size_t)(3 * T + Tc + 4) * sizeof(int) + 40 * sizeof(double) + 64;
}

size_t smem_for(int T, int Tc, int B, size_t cs) {
    size_t el = (size_t)B * Tc + 2 * FC_MAXW * B + (size_t)2 * B * T + T + Tc + 2 + (size_t)T * (Tc + 1) + 1;
    return el * cs + ((size_t)5 * T + 3 * Tc + B + 4) * sizeof(int) + 2 * FC_MAXW * sizeof(uint4) + 16;
}

struct FactorShape {
    int Cf = 0, B = 0, Tc = 0, threads = 256;
    size_t smem = 0;
};

cudaLaunchConfig_t factor_config(int clusters, const FactorShape& f, cudaStream_t st, cudaLaunchAttribute* attr) {
    cudaLaunchConfig_t cfg = {};
    cfg.gridDim = dim3(clusters * f.Cf);
    cfg.blockDim = dim3(f.threads);
    cfg.dynamicSmemBytes = f.smem;
    cfg.stream = st;
    attr[0].id = cudaLaunchAttributeClusterDimension;
    attr[0].val.clusterDim.x = f.Cf;
    attr[0].val.clusterDim.y = 1;
    attr[0].val.clusterDim.z = 1;
    cfg.attrs = attr;
    cfg.numAttrs = 1;
    return cfg;
}

using FactorKernel = void (*)(Pencil, const int*, const double2*, void* const*, int*, int, int);

FactorKernel factor_kernel(size_t cs, int B, int threads) {
    if (cs == sizeof(double2)) return threads <= 384 ? k_factor_cl<double2, 4, 4, 384> : k_factor_cl<double2, 4, 4, 512>;
    if (B == 16) return threads <= 384 ? k_factor_cl<float2, 16, 8, 384> : k_factor_cl<float2, 16, 8, 512>;
    return threads <= 384 ? k_factor_cl<float2, 8, 8, 384> : k_factor_cl<float2, 8, 8, 512>;
}

// How many clusters of this shape the GPU holds at once (0: it cannot run).
// The answer depends on the device and the shape only and is kept.
int active_clusters(size_t cs, const FactorShape& f) {
    static std::mutex mu;
    static std::map<std::tuple<int, size_t, int, int, size_t, int>, int> known;
    int dev = 0;
    SIM_CUDA(cudaGetDevice(&dev));
    const auto key = std::make_tuple(dev, cs, f.B, f.Cf, f.smem, f.threads);
    std::lock_guard<std::mutex> lock(mu);
    const auto it = known.find(key);
    if (it != known.end()) return it->second;
    FactorKernel kern = factor_kernel(cs, f.B, f.threads);
    SIM_CUDA(cudaFuncSetAttribute(kern, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)f.smem));
    if (f.Cf > 8 &&
        cudaFuncSetAttribute(kern, cudaFuncAttributeNonPortableClusterSizeAllowed, 1) != cudaSuccess)
        (void)cudaGetLastError();
    cudaLaunchAttribute attr[1];
    const cudaLaunchConfig_t cfg = factor_config(1, f, nullptr, attr);
    int n = 0;
    if (cudaOccupancyMaxActiveClusters(&n, kern, &cfg) != cudaSuccess) {
        (void)cudaGetLastError();
        n = 0;
    }
    known[key] = n;
    return n;
}

// Launch shape by an estimate of the clocks of one block: T pivots in panels of
// B, each panel's chain (its pivots, the next panel's columns, and with more than
// one CTA the cluster barrier and G's way through L2: 1,500 clocks) plus a part of
// the CTA's own columns' work (the update, which shares the FP64 pipe or the issue
// slots with the panel, and the forming and storing of the block's columns) or that
// work plus a part of the chain, times the waves the shifts need.  Why the sum and
// not the larger: T = 200 complex64 on 4, 7, 13 CTAs 20.0, 17.4, 16.3 ms in panels of 8 (20.1, 18.2,
// 17.5 of 16); T = 102 on 1, 3, 7 CTAs 5.5, 4.6, 4.1 ms; T = 98 complex128 on 5, 7,
// 13 CTAs 16.7, 15.3, 12.7 ms; T = 30 on 1, 2, 4 CTAs 1.09, 1.02, 0.97 ms.
FactorShape choose_factor_shape(int T, size_t cs, int count) {
    FactorShape best;
    double best_cost = 1e300;
    const bool f64 = cs == sizeof(double2);
    const int PW = (T + 31) / 32;
    for (int C = 1; C <= 16; ++C)
        for (int B : {16, 8, 4}) {
            if ((B == 4) != f64) continue;
            FactorShape f;
            f.Cf = C;
            f.B = B;
            f.Tc = (T + C * B - 1) / (C * B) * B;
            if (C > 1 && (C - 1) * f.Tc >= T) continue;  // a CTA without columns
            f.threads = T <= 64 ? 256 : (T <= 256 ? 384 : 512);
            f.smem = smem_for(T, f.Tc, B, cs);
            if (f.smem > 225 * 1024) continue;
            const int active = active_clusters(cs, f);
            if (active <= 0) continue;
            const int np = (T + B - 1) / B;
            const double pivot = f64 ? 64.0 * B * PW + 1300.0 : 500.0 + 30.0 * B + 40.0 * PW;
            const double look = f64 ? 2.2 * T * B * B : 0.07 * T * B * B + 500.0;
            const double chain = B * pivot + look + (C > 1 ? 1500.0 : 300.0);
            const double own = (f64 ? 2.2 : 0.06) * (double)T * T * f.Tc / np;
            const double panel = std::max(chain + (f64 ? 0.65 : 0.8) * own, own + 0.5 * chain);
            const double cost = (double)((count + active - 1) / active) * np * panel;
            if (cost < best_cost) {
                best_cost = cost;
                best = f;
            }
        }
    return best;
}
}  // namespace

bool factor_shifts_cluster(const Pencil& P, int precision, const int* d_shift_list, int count,
                           const double2* d_sigma, void* const* d_factor_ptrs, cudaStream_t st) {
    if (count <= 0) return true;
    const size_t cs = precision == SIM_FP64 ? sizeof(double2) : sizeof(float2);
    if (P.T < 2 || P.T > 32 * FC_MAXW || admit_bytes(P.T, cs) > 220 * 1024) return false;
    const int sides = (P.mid > 0) + (P.mid + 1 < P.nb);
    const FactorShape f = choose_factor_shape(P.T, cs, count * std::max(1, sides));
    if (f.Cf == 0) return false;
    if (!g_ferr) {
        SIM_CUDA(cudaMalloc(&g_ferr, sizeof(int)));
        SIM_CUDA(cudaMemset(g_ferr, 0, sizeof(int)));
    }
    FactorKernel kern = factor_kernel(cs, f.B, f.threads);
    SIM_CUDA(cudaFuncSetAttribute(kern, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)f.smem));
    cudaLaunchAttribute attr[1];
    kprof_begin("factor", st);
    for (int phase = sides > 0 ? 0 : 1; phase < 2; ++phase) {
        const cudaLaunchConfig_t cfg = factor_config(phase ? count : count * sides, f, st, attr);
        SIM_CUDA(cudaLaunchKernelEx(&cfg, kern, P, d_shift_list, d_sigma, d_factor_ptrs, g_ferr, f.Tc, phase));
        SIM_LAUNCH_CHECK();
    }
    const double TT = (double)P.T * P.T;
    kprof_end("factor", st, count * (2.0 * P.nb * TT * cs), count * 8.0 * P.nb * TT * P.T);
    return true;
}

}  // namespace sim
