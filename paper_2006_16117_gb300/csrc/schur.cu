// Schur form of each shift's Hessenberg matrix and the level evaluation
// built on it (Sec. 3.2, Eqs. zjHm, rmLc1; Sec. 3.3, Eqs. eq:many, eq:error,
// DeltaSm).
//
// The projected solves of a square all use one H_m: at node z_j,
//     (I + α_j H_m) y_j = β e_1,   α_j = σ - z_j.
// With the complex Schur form H_m = Z T Z^H (T upper triangular, Z unitary),
// computed once per shift,
//     (I + α_j T) x_j = c,   c = β Z^H e_1,   y_j = Z x_j,
// so a node costs one triangular solve, and everything the level needs is
// available without forming y_j:  e_m^T y_j = z_m^T x_j (z_m^T the last row
// of Z) for the residual of Eq. eq:error, ||y_j|| = ||x_j||, and the norms of
// the two quadrature sums Σ_j w_j y_j = Z Σ_j w_j x_j of Eq. DeltaSm.  The
// paper's own formula (the eigendecomposition H_m = P D P^{-1}) gives the same
// quantities; the Schur form is its unitary, backward-stable counterpart.
//
// k_schur: one CTA per shift, the shifted QR algorithm of k_ritz applied to
// whole rows and columns with the rotations accumulated into the two rows of Z
// the level needs (the first and the last: a row of Z evolves on its own
// under the column rotations).
// k_eval_schur: one lane per quadrature node (a CTA holds the 8 nodes of 4
// squares), so every FP64 instruction does useful work in all lanes; T's
// entries are warp-uniform loads when the 4 squares share a shift (children
// of one square do).  The squares their own shift does not resolve are then
// evaluated against every shift of their pencil at once (square-shift pairs
// as items) and k_pick_shift takes the shift the direct evaluation's order
// would.  Only a zero pivot or a shift without a Schur form sends a square to
// the direct evaluation (k_eval_level).
#include <cfloat>

#include "fp64.cuh"
#include "hess.cuh"
#include "internal.h"
#include "levels.h"

namespace sim {

namespace {

__device__ __forceinline__ double cabs_s(double2 a) { return hypot(a.x, a.y); }

__device__ __forceinline__ double2 csqrt_s(double2 z) {
    const double r = cabs_s(z);
    const double re = sqrt(fmax(0.0, 0.5 * (r + z.x)));
    const double im = sqrt(fmax(0.0, 0.5 * (r - z.x)));
    return make_double2(re, z.y < 0.0 ? -im : im);
}

}  // namespace

// The FP64 pipe takes 64 clocks of its scheduler for a warp instruction, however
// few lanes are active, so k_schur spreads every rotation over lanes and warps
// (m = 50: 20.8 ms on one warp, most of it scalar code of lane 0, now 3.7 ms):
//  * update warps: a thread computes one real component of one rotated pair (three
//    FP64 instructions).  Step k applies left rotation k to rows k, k+1 and, two
//    steps behind, right rotation k-2 to columns k-2, k-1 of the rows that left
//    rotations no longer touch, and to the two rows of Z.
//  * a generator warp runs one rotation ahead: in step k it rotates column k+1's
//    pair itself (nobody else touches that column in step k) and forms rotation
//    k+1 from it, its sums, square roots and products side by side in four lanes
//    (13 dependent FP64 instructions instead of about 150).
//  * the deflation test takes a lane per subdiagonal, in the norm |re| + |im|.
constexpr int SC_UPD = 256;           // update threads: 4 per pair, at most m + 3 pairs
constexpr int SC_THREADS = SC_UPD + 32;

// Shared memory: A [n][ld] row-major, then rows 0 and n-1 of Z as rows n, n+1 (ld odd).
__global__ void __launch_bounds__(SC_THREADS) k_schur(const double2* Hall, int m, const int* meff_all,
                                                      const double* beta_all, int s0, double2* Tall, double2* Call,
                                                      double2* Qall, int* ok_all) {
    const int s = s0 + blockIdx.x;
    const int n = meff_all[s];
    const double2* Hs = Hall + (size_t)s * (m + 1) * m;  // column-major, leading dimension m + 1
    extern __shared__ double2 sh_schur[];
    double2* A = sh_schur;
    const int ld = m | 1;
    __shared__ double gc[64];
    __shared__ double2 gs[64];
    __shared__ double2 s_mu;
    __shared__ int s_l;
    __shared__ double s_nrm[SC_THREADS / 32];
    const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
    const bool gen = warp == SC_UPD / 32;
    int fail = (n < 1 || n > 60) ? 1 : 0;
    double nrm = 0.0;
    if (!fail) {
        for (int idx = tid; idx < n * n; idx += SC_THREADS) {
            const int r = idx / n, c = idx % n;
            const double2 h = (r <= c + 1) ? Hs[(size_t)c * (m + 1) + r] : make_double2(0.0, 0.0);
            A[r * ld + c] = h;
            nrm = fmax(nrm, fabs(h.x) + fabs(h.y));
        }
        for (int c = tid; c < n; c += SC_THREADS) {
            A[n * ld + c] = make_double2(c == 0 ? 1.0 : 0.0, 0.0);
            A[(n + 1) * ld + c] = make_double2(c == n - 1 ? 1.0 : 0.0, 0.0);
        }
    }
    for (int o = 16; o > 0; o >>= 1) nrm = fmax(nrm, __shfl_xor_sync(0xffffffffu, nrm, o));
    if (lane == 0) s_nrm[warp] = nrm;
    __syncthreads();
    for (int w = 0; w < SC_THREADS / 32; ++w) nrm = fmax(nrm, s_nrm[w]);

    // rotation k from (a, b) = (A[k][k], A[k+1][k]), by the generator warp
    auto generate = [&](int k, double2 a, double2 b) {
        // lane 0: |a|^2, 1: |b|^2, 2: re(a conj b), 3: im(a conj b)
        const double p = lane == 1 ? b.x : (lane == 3 ? a.y : a.x), q = lane == 0 ? a.x : b.x;
        const double r = lane == 1 ? b.y : (lane == 3 ? -a.x : a.y), t = lane == 0 ? a.y : b.y;
        const double d = fma(r, t, p * q);
        const double na2 = __shfl_sync(0xffffffffu, d, 0), nb2 = __shfl_sync(0xffffffffu, d, 1);
        const double h2 = na2 + nb2;
        if (na2 > 1e-280 && h2 < 1e280) {
            const double rs = rsqrt_nr(lane == 0 ? na2 : h2);
            const double pr = __shfl_sync(0xffffffffu, rs, 0) * __shfl_sync(0xffffffffu, rs, 1);  // 1 / (|a| h)
            const double v = d * pr;  // lane 0: |a| / h, 2 and 3: a conj(b) / (|a| h)
            if (lane == 0) gc[k] = v;
            if (lane == 2) gs[k].x = v;
            if (lane == 3) gs[k].y = v;
        } else if (lane == 0) {
            const double na = cabs_s(a), nb = cabs_s(b);
            double c;
            double2 sn;
            if (nb == 0.0) {
                c = 1.0;
                sn = make_double2(0.0, 0.0);
            } else if (na == 0.0) {
                c = 0.0;
                sn = make_double2(b.x / nb, -b.y / nb);
            } else {
                const double h = hypot(na, nb);
                c = na / h;
                const double2 ua = make_double2(a.x / na, a.y / na);
                sn = cmul(ua, make_double2(b.x / h, -b.y / h));
            }
            gc[k] = c;
            gs[k] = sn;
        }
        __syncwarp();
    };
    // component cmp (x'.re, x'.im, y'.re, y'.im) of the rotated pair:
    //   left  x' = c x + s y,        y' = c y - conj(s) x
    //   right x' = c x + conj(s) y,  y' = c y - s x
    auto rotated = [&](int cmp, bool left, double c, double2 sn, double2 x, double2 y) {
        const bool first = cmp < 2, im = cmp & 1;
        const double2 o = first ? x : y, e = first ? y : x;
        const double sx = first ? sn.x : -sn.x;
        const double sy = (im == left) ? sn.y : -sn.y;
        return fma(sy, im ? e.x : e.y, fma(sx, im ? e.y : e.x, c * (im ? o.y : o.x)));
    };

    int hi = n - 1, its = 0, sweeps = 0;
    while (!fail && hi > 0) {
        if (warp == 0) {
            // the largest l with a negligible subdiagonal A[l][l-1], l <= hi (0: none)
            int best = 0;
            for (int k = lane + 1; k <= hi; k += 32) {
                const double2 u = A[k * ld + k - 1], d0 = A[(k - 1) * ld + k - 1], d1 = A[k * ld + k];
                double d = (fabs(d0.x) + fabs(d0.y)) + (fabs(d1.x) + fabs(d1.y));
                if (d == 0.0) d = nrm;
                if (fabs(u.x) + fabs(u.y) <= DBL_EPSILON * d) best = k;
            }
            best = __reduce_max_sync(0xffffffffu, best);
            if (lane == 0) {
                if (best > 0) A[best * ld + best - 1] = make_double2(0.0, 0.0);
                s_l = best;
            }
        } else if (gen && lane == 0) {
            // Wilkinson shift from the trailing 2×2 block, exceptional every 10 sweeps
            const double2 p = A[(hi - 1) * ld + hi - 1], q = A[(hi - 1) * ld + hi];
            const double2 r = A[hi * ld + hi - 1], t = A[hi * ld + hi];
            double2 mu = t;
            if (its > 0 && its % 10 == 0) {
                mu.x += 0.75 * cabs_s(r);
            } else {
                const double2 d = make_double2(0.5 * (p.x - t.x), 0.5 * (p.y - t.y));
                const double2 qr = cmul(q, r);
                const double2 disc = csqrt_s(cadd(cmul(d, d), qr));
                const double2 den1 = cadd(d, disc), den2 = csub(d, disc);
                const double2 den = cabs2(den1) >= cabs2(den2) ? den1 : den2;
                if (den.x != 0.0 || den.y != 0.0) mu = csub(t, cdiv(qr, den));
            }
            s_mu = mu;
        }
        __syncthreads();
        const int l = s_l;
        if (l == hi) {
            --hi;
            its = 0;
            __syncthreads();  // s_l read before it is rewritten
            continue;
        }
        if (++sweeps > 30 * n) {
            fail = 1;
            break;
        }
        ++its;
        const double2 mu = s_mu;
        for (int k = l + tid; k <= hi; k += SC_THREADS) A[k * ld + k] = csub(A[k * ld + k], mu);
        __syncthreads();
        if (gen) generate(l, A[l * ld + l], A[(l + 1) * ld + l]);
        __syncthreads();
        // step k: left rotation k, and right rotation k-2 on the rows it has left behind
        for (int k = l; k <= hi + 1; ++k) {
            const bool dol = k < hi, dor = k - 2 >= l;
            if (gen) {
                if (k + 1 < hi) {
                    // column k+1 of left rotation k, then rotation k+1
                    double2* px = A + k * ld + k + 1;
                    double2* py = px + ld;
                    const double2 x = *px, y = *py;
                    const double v = rotated(lane & 3, true, gc[k], gs[k], x, y);
                    const double2 a = make_double2(__shfl_sync(0xffffffffu, v, 2), __shfl_sync(0xffffffffu, v, 3));
                    if (lane < 4) (lane < 2 ? reinterpret_cast<double*>(px) : reinterpret_cast<double*>(py))[lane & 1] = v;
                    generate(k + 1, a, A[(k + 2) * ld + k + 1]);
                }
            } else {
                // left: columns k .. n-1 (but k+1 where the generator has it); right: rows 0 .. k-1, Z's two
                const int nl = dol ? n - k : 0, rows = min(k, hi + 1), nrt = dor ? rows + 2 : 0;
                for (int it = tid >> 2; it < nl + nrt; it += SC_UPD / 4) {
                    const bool left = it < nl;
                    const int kk = left ? k : k - 2;
                    double2 *px, *py;
                    if (left) {
                        px = A + k * ld + k + it;
                        py = px + ld;
                    } else {
                        const int row = it - nl < rows ? it - nl : n + (it - nl - rows);
                        px = A + row * ld + kk;
                        py = px + 1;
                    }
                    const bool skip = left && it == 1 && k + 1 < hi;
                    const unsigned quad = 0xFu << (lane & ~3);
                    const double2 x = *px, y = *py;
                    const double v = rotated(tid & 3, left, gc[kk], gs[kk], x, y);
                    __syncwarp(quad);  // the pair's four lanes have read it
                    if (!skip) (tid & 2 ? reinterpret_cast<double*>(py) : reinterpret_cast<double*>(px))[tid & 1] = v;
                }
            }
            __syncthreads();
        }
        for (int k = l + tid; k <= hi; k += SC_THREADS) A[k * ld + k] = cadd(A[k * ld + k], mu);
        __syncthreads();
    }
    const double2 *Z0 = A + n * ld, *Zl = A + (n + 1) * ld;
    double2* T = Tall + (size_t)s * m * m;
    const double beta = beta_all[s];
    if (!fail) {
        for (int idx = tid; idx < n * n; idx += SC_THREADS) {
            const int r = idx / n, c = idx % n;
            T[r * m + c] = c >= r ? A[r * ld + c] : make_double2(0.0, 0.0);
        }
        for (int i = tid; i < n; i += SC_THREADS) {
            const double2 z0 = Z0[i];
            Call[(size_t)s * m + i] = make_double2(beta * z0.x, -beta * z0.y);
            Qall[(size_t)s * m + i] = Zl[i];
        }
    }
    if (tid == 0) ok_all[s] = fail ? 0 : 1;
}

// 4 squares of 8 nodes per CTA, a lane per node in each of its SE_WARPS warps, the
// rows of the triangular solve dealt out to the warps (row i to warp i mod 4), so
// that one square's chain uses all four FP64 pipes of an SM: a level often holds
// fewer squares than the GPU has warps, and then the time is one warp's chain
// (m = 50, 1,300 squares: 373 us a level with whole solves per warp, now about 190).  Column by column from
// the last: the owner of row i forms x_i from its sum and sends it round through
// shared memory; every warp then adds T_ri x_i to its rows r < i, whose T_ri it
// loaded one column ahead.
constexpr int SE_WARPS = 4;
constexpr int SE_ROWS = 13;  // rows per warp: m <= 52

// ALL = false: item t is square t against its own shift; a square it resolves
//   gets its results, the others todo[q] = 1.
// ALL = true: item t = (i, o) is square list[i] against shift lo + o of its
//   pencil's range [lo, hi), o < smax; the indicator, the largest node
//   residual and the zero-pivot / no-Schur-form flag go to rind, rrho, rbad.
template <bool ALL>
__global__ void __launch_bounds__(SE_WARPS * 32) k_eval_schur(ShiftTable st, LevelArgs a, uint8_t* todo,
                                                              const int64_t* list, int smax, int64_t nitems,
                                                              double* rind, double* rrho, uint8_t* rbad) {
    const int* ok_all = st.schOK;
    __shared__ double2 xs[2][32];             // x_i of every node, alternating
    __shared__ double red[SE_WARPS][5][32];   // yl (2), ||x||^2, the quadrature sums' squares
    __shared__ int s_bad;
    const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
    const int m = st.m;
    const int j = lane & 7;  // node
    for (int64_t t0 = (int64_t)blockIdx.x * 4; t0 < nitems; t0 += (int64_t)gridDim.x * 4) {
        const int64_t t = t0 + (lane >> 3);
        int64_t q = t;
        bool active = t < nitems;
        int s = 0, n = 0;
        if (ALL && active) {
            q = list[t / smax];
            int lo = 0, hi = st.S;
            if (st.pencil_of) {
                const int p = st.pencil_of[a.sid[q]];
                lo = st.p_sb[p];
                hi = st.p_se[p];
            }
            s = lo + (int)(t % smax);
            active = s < hi;
        }
        double re_lo = a.re_lo, im_lo = a.im_lo, side = a.side;
        bool good = false;
        if (active) {
            if (!ALL) s = a.sid[q];
            if (st.pencil_of) {
                const int p = st.pencil_of[s];
                re_lo = st.p_re_lo[p];
                im_lo = st.p_im_lo[p];
                side = st.p_side[p];
            }
            good = ok_all[s] != 0;
            n = good ? st.meff[s] : 0;
        } else {
            s = 0;
        }
        const double2 c = square_center(re_lo, im_lo, side, active ? a.ix[q] : 0, active ? a.iy[q] : 0);
        const double2 off = node_offset(j, side);
        const double2 z = make_double2(__dadd_rn(c.x, off.x), __dadd_rn(c.y, off.y));
        const double2 sig = active ? st.sigma[s] : make_double2(0.0, 0.0);
        const double2 alpha = make_double2(__dsub_rn(sig.x, z.x), __dsub_rn(sig.y, z.y));
        const double2 w8 = cscale(off, 0.125);
        const double2* T = st.schT + (size_t)s * m * m;
        const double2* Cv = st.schC + (size_t)s * m;
        const double2* Qv = st.schQ + (size_t)s * m;
        const int nmax = __reduce_max_sync(0xffffffffu, n);  // every warp holds the same nodes
        if (threadIdx.x == 0) s_bad = 0;
        // this warp's rows r = warp + 4 u: sums, reciprocals of 1 + α T_rr, next column's T
        double2 acc[SE_ROWS], tn[SE_ROWS];
#pragma unroll
        for (int u = 0; u < SE_ROWS; ++u) {
            acc[u] = make_double2(0.0, 0.0);
            const int r = warp + SE_WARPS * u, i = n - 1;
            tn[u] = r < i ? __ldg(T + (size_t)r * m + i) : make_double2(0.0, 0.0);
        }
        double2 yl = make_double2(0.0, 0.0);
        double yn2 = 0.0, n8 = 0.0, n4 = 0.0;
        bool zero_pivot = false;
        // this warp's next row: 1 / (1 + α T_rr) and c_r, made ahead of its turn
        double2 inv, cr;
        auto next_row = [&](int r) {
            inv = cr = make_double2(0.0, 0.0);
            if (r >= 0 && r < n) {
                const double2 trr = __ldg(T + (size_t)r * m + r);
                cr = __ldg(Cv + r);
                double2 den;
                den.x = fma(alpha.x, trr.x, fma(-alpha.y, trr.y, 1.0));
                den.y = fma(alpha.x, trr.y, alpha.y * trr.x);
                if (den.x == 0.0 && den.y == 0.0) zero_pivot = true;
                else inv = crecip(den);
            }
        };
        {
            const int r = nmax - 1 - ((nmax - 1 - warp) & (SE_WARPS - 1));  // the last row of this warp
            next_row(r);
        }
        __syncthreads();
        for (int i = nmax - 1; i >= 0; --i) {
            const bool mine = (i & (SE_WARPS - 1)) == warp;
            double2 xi = make_double2(0.0, 0.0);
            if (mine) {
                // x_i = (c_i - α Σ_{k>i} T_ik x_k) / (1 + α T_ii)
                double2 sum = make_double2(0.0, 0.0);
#pragma unroll
                for (int u = 0; u < SE_ROWS; ++u)
                    if (u == i / SE_WARPS) sum = acc[u];
                const double2 rhs = make_double2(fma(-alpha.x, sum.x, fma(alpha.y, sum.y, cr.x)),
                                                 fma(-alpha.x, sum.y, fma(-alpha.y, sum.x, cr.y)));
                xi = cmul(rhs, inv);
                xs[i & 1][lane] = xi;
            }
            __syncthreads();
            const double2 x = xs[i & 1][lane];
#pragma unroll
            for (int u = SE_ROWS - 1; u >= 0; --u) {
                const int r = warp + SE_WARPS * u;
                if (r < i) {  // warp-uniform
                    // (a node of a smaller order has x = 0 and T = 0 in the columns beyond it)
                    acc[u] = cfma(tn[u], x, acc[u]);
                    tn[u] = r < i - 1 && i - 1 < n ? __ldg(T + (size_t)r * m + i - 1) : make_double2(0.0, 0.0);
                }
            }
            if (mine) {
                // off the chain: what the level needs of component i, and this warp's next row
                if (i < n) {
                    yl = cfma(__ldg(Qv + i), xi, yl);
                    yn2 = fma(xi.x, xi.x, fma(xi.y, xi.y, yn2));
                }
                // the quadrature sums of component i over the square's 8 lanes: lanes with
                // bit 2 clear sum the real parts, the others the imaginary ones; even
                // lanes then hold the coarse rule's sum (half of it: its weights are twice
                // the fine rule's), and all lanes add the odd nodes for the fine rule
                const double2 p = cmul(w8, xi);
                const bool up = (lane & 4) != 0;
                double v = (up ? p.y : p.x) + __shfl_xor_sync(0xffffffffu, up ? p.x : p.y, 4);
                v += __shfl_xor_sync(0xffffffffu, v, 2);
                n4 = fma(v, v, n4);
                v += __shfl_xor_sync(0xffffffffu, v, 1);
                n8 = fma(v, v, n8);
                next_row(i - SE_WARPS);
            }
        }
        if (zero_pivot) good = false;
        red[warp][0][lane] = yl.x;
        red[warp][1][lane] = yl.y;
        red[warp][2][lane] = yn2;
        red[warp][3][lane] = n8;
        red[warp][4][lane] = n4;
        if (__any_sync(0xffffffffu, zero_pivot)) {
            // which nodes: a bit per lane
            const unsigned b = __ballot_sync(0xffffffffu, zero_pivot);
            if (lane == 0) atomicOr(&s_bad, (int)b);
        }
        __syncthreads();
        if (warp == 0) {
            double v[5];
#pragma unroll
            for (int e = 0; e < 5; ++e) {
                v[e] = red[0][e][lane];
#pragma unroll
                for (int w = 1; w < SE_WARPS; ++w) v[e] += red[w][e][lane];
            }
            if ((unsigned)s_bad >> lane & 1u) good = false;
            yl = make_double2(v[0], v[1]);
            yn2 = v[2];
            // real plus imaginary parts' squares; the coarse rule's from an even lane
            n8 = v[3] + __shfl_xor_sync(0xffffffffu, v[3], 4);
            n4 = v[4] + __shfl_xor_sync(0xffffffffu, v[4], 4);
            n4 = 4.0 * __shfl_sync(0xffffffffu, n4, lane & ~7);
            // residual of Eq. eq:error at this node, as the direct evaluation forms it
            double r = 0.0;
            if (active && good && n > 0) {
                const double hlast = cabsd(st.H[(size_t)s * (m + 1) * m + (size_t)(n - 1) * (m + 1) + n]);
                const double num = cabsd(alpha) * hlast * cabsd(yl);
                const double den = st.scale == 0 ? sqrt(yn2) : st.beta[s];
                r = num / den;
                if (!(r == r) || isinf(r)) r = INFINITY;
                if (num == 0.0) r = 0.0;
            }
            int bad = (active && (!good || n == 0)) ? 1 : 0;
            double rmax = r;
#pragma unroll
            for (int o = 1; o < 8; o <<= 1) {
                rmax = fmax(rmax, __shfl_xor_sync(0xffffffffu, rmax, o));
                bad |= __shfl_xor_sync(0xffffffffu, bad, o);
            }
            const double s8 = sqrt(n8), s4 = sqrt(n4);
            const double ind = s4 > 0.0 ? s8 / s4 : (s8 > 0.0 ? INFINITY : 0.0);
            if (ALL && t < nitems && j == 0) {
                rind[t] = ind;
                rrho[t] = active ? rmax : INFINITY;
                rbad[t] = active ? (uint8_t)bad : (uint8_t)0;
            }
            if (!ALL && active && j == 0) {
                if (!bad && rmax <= st.eps) {
                    a.ind[q] = ind;
                    a.mark[q] = ind > st.delta0 ? 1 : 0;
                    a.flag[q] = 0;
                    todo[q] = 0;
                } else {
                    todo[q] = 1;
                }
            }
        }
        __syncthreads();  // red, s_bad and xs are free again
    }
}

void schur_shifts(const double2* H, int m, const int* meff, const double* beta, int s0, int count, double2* T,
                  double2* C, double2* Q, int* ok, cudaStream_t st) {
    if (count <= 0) return;
    const size_t sm = (size_t)(m + 2) * (m | 1) * sizeof(double2);
    SIM_CUDA(cudaFuncSetAttribute(k_schur, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)sm));
    k_schur<<<count, SC_THREADS, sm, st>>>(H, m, meff, beta, s0, T, C, Q, ok);
    SIM_LAUNCH_CHECK();
}

// The squares their own shift left (todo != 0), listed in any order.
__global__ void k_list_todo(const uint8_t* todo, int64_t count, int64_t* list, unsigned long long* n) {
    const int64_t q = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
    if (q < count && todo[q]) list[atomicAdd(n, 1ull)] = (int64_t)q;
}

// One thread per listed square: the result the direct evaluation's shift order
// gives (own shift first, then the others nearest-first by |σ - c|, ties by the
// lower id; the first that resolves the square is used; if none does, the own
// shift's indicator and "unresolvable").  A square with any zero pivot or
// missing Schur form among its shifts stays todo for the direct evaluation.
__global__ void k_pick_shift(ShiftTable st, LevelArgs a, const int64_t* list, int64_t ntodo, int smax,
                             const double* rind, const double* rrho, const uint8_t* rbad, uint8_t* todo) {
    const int64_t i = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
    if (i >= ntodo) return;
    const int64_t q = list[i];
    const int own = a.sid[q];
    int lo = 0, hi = st.S;
    double re_lo = a.re_lo, im_lo = a.im_lo, side = a.side;
    if (st.pencil_of) {
        const int p = st.pencil_of[own];
        lo = st.p_sb[p];
        hi = st.p_se[p];
        re_lo = st.p_re_lo[p];
        im_lo = st.p_im_lo[p];
        side = st.p_side[p];
    }
    const int64_t r0 = i * (int64_t)smax;
    for (int s = lo; s < hi; ++s)
        if (rbad[r0 + (s - lo)]) return;  // left to the direct evaluation
    const double2 c = square_center(re_lo, im_lo, side, a.ix[q], a.iy[q]);
    int used = own, tried = 1;
    bool res = rrho[r0 + (own - lo)] <= st.eps;
    if (!res) {
        double bd = INFINITY;
        int best = -1;
        for (int s = lo; s < hi; ++s) {
            if (s == own || !(rrho[r0 + (s - lo)] <= st.eps)) continue;
            const double d = hypot(st.sigma[s].x - c.x, st.sigma[s].y - c.y);
            if (d < bd || (d == bd && s < best)) {
                bd = d;
                best = s;
            }
        }
        if (best >= 0) {
            res = true;
            used = best;
            for (int s = lo; s < hi; ++s) {
                if (s == own) continue;
                const double d = hypot(st.sigma[s].x - c.x, st.sigma[s].y - c.y);
                if (d < bd || (d == bd && s <= best)) ++tried;
            }
        } else {
            tried = hi - lo;
        }
    }
    if (a.retries && tried > 1) atomicAdd(a.retries, (unsigned long long)(tried - 1));
    const double ind = res ? rind[r0 + (used - lo)] : rind[r0 + (own - lo)];
    a.ind[q] = ind;
    a.mark[q] = res ? (ind > st.delta0 ? 1 : 0) : 1;
    a.flag[q] = res ? 0 : 1;
    a.sid[q] = used;
    todo[q] = 0;
}

void eval_level_schur(const ShiftTable& st, const LevelArgs& a, uint8_t* todo, cudaStream_t stream) {
    if (a.count <= 0) return;
    const int grid = (int)std::min<int64_t>((a.count + 3) / 4, 152 * 64);
    kprof_begin("eval_level_schur", stream);
    k_eval_schur<false><<<grid, SE_WARPS * 32, 0, stream>>>(st, a, todo, nullptr, 1, a.count, nullptr, nullptr,
                                                             nullptr);
    SIM_LAUNCH_CHECK();
    // per square: 8 triangular solves of order m (m²/2 complex multiply-adds each)
    kprof_end("eval_level_schur", stream, 0.0, a.count * 8.0 * 4.0 * st.m * st.m);
}

void eval_level_schur_retries(const ShiftTable& st, const LevelArgs& a, uint8_t* todo, int64_t ntodo, int smax,
                              DeviceArena& ar, cudaStream_t stream) {
    if (ntodo <= 0 || smax <= 0) return;
    int64_t* list = ar.get<int64_t>("lvl_list", ntodo);
    unsigned long long* cnt = ar.get<unsigned long long>("lvl_list_n", 1);
    const int64_t nitems = ntodo * (int64_t)smax;
    double* rind = ar.get<double>("lvl_rind", nitems);
    double* rrho = ar.get<double>("lvl_rrho", nitems);
    uint8_t* rbad = ar.get<uint8_t>("lvl_rbad", nitems);
    SIM_CUDA(cudaMemsetAsync(cnt, 0, sizeof(unsigned long long), stream));
    k_list_todo<<<cdiv_up(a.count, 256), 256, 0, stream>>>(todo, a.count, list, cnt);
    SIM_LAUNCH_CHECK();
    const int grid = (int)std::min<int64_t>((nitems + 3) / 4, 152 * 64);
    kprof_begin("eval_level_schur", stream);
    k_eval_schur<true><<<grid, SE_WARPS * 32, 0, stream>>>(st, a, todo, list, smax, nitems, rind, rrho, rbad);
    SIM_LAUNCH_CHECK();
    k_pick_shift<<<cdiv_up(ntodo, 128), 128, 0, stream>>>(st, a, list, ntodo, smax, rind, rrho, rbad, todo);
    SIM_LAUNCH_CHECK();
    kprof_end("eval_level_schur", stream, 0.0, nitems * 8.0 * 4.0 * st.m * st.m);
}

}  // namespace sim
