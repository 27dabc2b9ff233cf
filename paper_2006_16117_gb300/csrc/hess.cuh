// Device helpers shared by the level kernels and the multiplicity kernels:
// quadrature node offsets, square centres, staging of a Hessenberg matrix and
// the warp-level Hessenberg solve (I + alpha H) y = beta e1.
#pragma once

#include "common.cuh"
#include "fp64.cuh"

namespace sim {

constexpr double SQRT1_2 = 0.70710678118654752440;

__device__ __forceinline__ double mag1(double2 a) { return fabs(a.x) + fabs(a.y); }

// node offsets z_j - c on the circle circumscribing a square of side s, j = 0..7
__device__ __forceinline__ double2 node_offset(int j, double s) {
    const double r = __dmul_rn(s, SQRT1_2);
    const double hs = 0.5 * s;
    switch (j) {
        case 0: return make_double2(r, 0.0);
        case 1: return make_double2(hs, hs);
        case 2: return make_double2(0.0, r);
        case 3: return make_double2(-hs, hs);
        case 4: return make_double2(-r, 0.0);
        case 5: return make_double2(-hs, -hs);
        case 6: return make_double2(0.0, -r);
        default: return make_double2(hs, -hs);
    }
}

__device__ __forceinline__ double2 square_center(double re_lo, double im_lo, double s, int64_t ix, int64_t iy) {
    return make_double2(__dadd_rn(re_lo, __dmul_rn((double)ix + 0.5, s)),
                        __dadd_rn(im_lo, __dmul_rn((double)iy + 0.5, s)));
}

// Stage shift s's Hessenberg (column-major (m+1) x m in global) row-major into
// Hs[r*m + c] (r < m) and return h_{m+1,m}.
__device__ __forceinline__ void stage_H(const double2* H, int m, int meff, double2* Hs) {
    for (int e = threadIdx.x; e < meff * meff; e += blockDim.x) {
        int r = e / meff, c = e % meff;
        Hs[r * meff + c] = (r <= c + 1) ? H[(size_t)c * (m + 1) + r] : make_double2(0.0, 0.0);
    }
}

// v - a b in four operations
__device__ __forceinline__ double2 sub_product(double2 v, double2 a, double2 b) {
    return make_double2(fma(-a.x, b.x, fma(a.y, b.y, v.x)), fma(-a.x, b.y, fma(-a.y, b.x, v.y)));
}

// One warp solves (I + alpha H) y = beta e1 (order m <= 63, H row-major in Hs with
// leading dimension m) and leaves y in ys[0..m).  U: packed upper-triangular
// scratch of m(m+1)/2 entries.  Returns |y_{m-1}| and ||y||^2 (warp-uniform).
//
// An FP64 instruction costs a warp 64 clocks however many lanes it serves, so
// what counts is their number, about 1,850 a solve at m = 50 (5,500 with divisions
// and the right-hand side on every lane: 4,096 squares of 8 nodes took 9.9 ms, now
// 4.95):
//  * the right-hand side is column m of the rows;
//  * a pivot's reciprocal (crecip) serves the elimination and, kept by the pivot's
//    lane, the back substitution;
//  * columns below 32 are done with from row 32 on.
// The system is not divided by alpha, although H's rows would then serve as they
// stand (330 instructions fewer): the rounding of 1 / alpha goes into every diagonal
// entry alike, and the median error of |y_{m-1}| / ||y|| grows 2 to 3 times.
__device__ __forceinline__ void warp_hess_solve(const double2* Hs, int m, double2 alpha, double beta, double2* U, double2* ys,
                                double& ylast, double& ynorm2) {
    const int lane = threadIdx.x & 31;
    const int c0 = lane, c1 = lane + 32;
    const double2 zero = make_double2(0.0, 0.0);
    // entry (r, c) of I + alpha H: alpha h rounded before 1 is added, as an FMA onto the
    // 1 would round its first product to the 1's last place (a fifth more error)
    auto entry = [&](int r, int c) -> double2 {
        if (c >= m) return zero;
        double2 v = cmul(alpha, Hs[r * m + c]);
        if (c == r) v.x += 1.0;
        return v;
    };
    double2 a0 = entry(0, c0), a1 = entry(0, c1);
    if (c0 == m) a0 = make_double2(beta, 0.0);
    if (c1 == m) a1 = make_double2(beta, 0.0);
    double2 iv0 = zero, iv1 = zero;  // reciprocals of U's diagonal in this lane's columns
    for (int k = 0; k < m; ++k) {
        const bool low = k < 32;  // columns 0..31 still in work
        const bool more = k + 1 < m;
        double2 b0 = low && more ? entry(k + 1, c0) : zero;
        double2 b1 = more ? entry(k + 1, c1) : zero;
        const int src = k & 31;
        double2 ak, bk;
        ak.x = __shfl_sync(0xffffffffu, low ? a0.x : a1.x, src);
        ak.y = __shfl_sync(0xffffffffu, low ? a0.y : a1.y, src);
        bk.x = __shfl_sync(0xffffffffu, low ? b0.x : b1.x, src);
        bk.y = __shfl_sync(0xffffffffu, low ? b0.y : b1.y, src);
        if (more && mag1(bk) > mag1(ak)) {
            double2 t;
            t = a0; a0 = b0; b0 = t;
            t = a1; a1 = b1; b1 = t;
            t = ak; ak = bk; bk = t;
        }
        // U row k, and the transformed right-hand side
        const int ofs = k * m - (k * (k - 1)) / 2;
        if (c0 >= k && c0 < m) U[ofs + (c0 - k)] = a0;
        if (c1 >= k && c1 < m) U[ofs + (c1 - k)] = a1;
        if (c0 == m) ys[k] = a0;
        if (c1 == m) ys[k] = a1;
        const double2 inv = (ak.x == 0.0 && ak.y == 0.0) ? zero : crecip(ak);
        if (lane == src) {
            if (low) iv0 = inv;
            else iv1 = inv;
        }
        const double2 l = cmul(bk, inv);
        // (a column that is done with only holds garbage from here on)
        if (low) a0 = sub_product(b0, l, a0);
        a1 = sub_product(b1, l, a1);
    }
    __syncwarp();
    // column-oriented back substitution: lane owns rows lane and lane+32
    double2 r0 = (c0 < m) ? ys[c0] : zero;
    double2 r1 = (c1 < m) ? ys[c1] : zero;
    __syncwarp();
    for (int j = m - 1; j >= 0; --j) {
        const bool hi = j >= 32;
        const double2 t = hi ? cmul(r1, iv1) : cmul(r0, iv0);
        double2 yj;
        yj.x = __shfl_sync(0xffffffffu, t.x, j & 31);
        yj.y = __shfl_sync(0xffffffffu, t.y, j & 31);
        if (lane == (j & 31)) {
            if (hi) r1 = yj;
            else r0 = yj;
        }
        const int q0 = c0 * m - (c0 * (c0 - 1)) / 2 + (j - c0);
        if (c0 < j) r0 = sub_product(r0, U[q0], yj);
        if (j > 32 && c1 < j) r1 = sub_product(r1, U[c1 * m - (c1 * (c1 - 1)) / 2 + (j - c1)], yj);
    }
    if (c0 < m) ys[c0] = r0;
    if (c1 < m) ys[c1] = r1;
    double nrm = 0.0;
    if (c0 < m) nrm = cabs2(r0);
    if (c1 < m) nrm += cabs2(r1);
    ynorm2 = warp_sum(nrm);
    const double last = cabsd(m <= 32 ? r0 : r1);
    ylast = __shfl_sync(0xffffffffu, last, (m - 1) & 31);
    __syncwarp();
}


}  // namespace sim
