// Krylov side of SIM-M on the GPU: the Cayley transform's shifted operator
// (A - σB) and its inverse, and the Arnoldi process for M = (A - σB)^{-1} B
// (Sec. 2, Eqs. AzBxf, IMxb, eq:arnoldi).
//
//  * factor_shifts  : block-tridiagonal factorisation of A - σB, eliminated
//                     from both ends to the middle block, for many shifts at
//                     once, one CTA per shift (the blocks that the cluster
//                     kernel of factor_cluster.cu does not hold); each
//                     diagonal Schur complement D_k is inverted by Gauss–Jordan
//                     with partial pivoting.  Storage: Dinv_k = D_k^{-1} and
//                     E_k = Dinv_k K_{k,inner(k)}, both dense T×T, in complex128
//                     (FP64 mode) or complex64 (mixed mode).
//  * (the solve x = (A - σB)^{-1} r through those factors is the cluster
//    kernel of solve_cluster.cu)
//  * inner_solve    : batched FGMRES(k) in FP64 with the factorisation as right
//                     preconditioner, CGS2 on its basis, Givens rotations and an
//                     explicit residual check per cycle.  In mixed mode this is
//                     GMRES-based iterative refinement of a complex64 solve.
//  * arnoldi        : m steps of w = M v_j = (A - σB)^{-1} B v_j with classical
//                     Gram–Schmidt applied twice (CGS2) in FP64.
#include <algorithm>
#include <cmath>
#include <cstdio>
#include <stdexcept>
#include <vector>

#include "internal.h"
#include "levels.h"
#include "gs.h"
#include "autotune.h"
#include "separable.h"
#include "solve_cluster.h"

namespace sim {

// ---------------------------------------------------------------------------
// block-tridiagonal factorisation
// ---------------------------------------------------------------------------
template <class C> __device__ __forceinline__ C czero();
template <> __device__ __forceinline__ double2 czero<double2>() { return make_double2(0.0, 0.0); }
template <> __device__ __forceinline__ float2 czero<float2>() { return make_float2(0.f, 0.f); }

__device__ __forceinline__ double2 shifted_val(const Pencil& P, int64_t e, double2 sg) {
    double2 a = P.Ka[e], b = P.Kb[e];
    return make_double2(a.x - (sg.x * b.x - sg.y * b.y), a.y - (sg.x * b.y + sg.y * b.x));
}

template <class C> __device__ __forceinline__ double mag1(C a) { return fabs((double)a.x) + fabs((double)a.y); }

constexpr int FACTOR_THREADS = 512;

template <class C>
__global__ void __launch_bounds__(FACTOR_THREADS) k_factor(Pencil P, const int* shift_list, const double2* sigma,
                                                           void* const* fptrs, int* err) {
    const int T = P.T, nb = P.nb;
    const int s = shift_list[blockIdx.x];
    C* Dinv = reinterpret_cast<C*>(fptrs[s]);
    C* E = Dinv + (size_t)nb * T * T;
    const double2 sg = sigma[s];
    extern __shared__ unsigned char smem_raw[];
    C* rowp = reinterpret_cast<C*>(smem_raw);
    C* colp = rowp + T;
    int* piv = reinterpret_cast<int*>(colp + T);
    double* redv = reinterpret_cast<double*>(piv + T + (T & 1));
    int* redi = reinterpret_cast<int*>(redv + 32);
    const int tid = threadIdx.x, bd = blockDim.x;
    const int lane = tid & 31, warp = tid >> 5, nw = bd >> 5;
    const size_t TT = (size_t)T * T;

    {
        C* Lval = Dinv + factor_lval_offset(P);
        for (int64_t e = tid; e < P.nnzL; e += bd) Lval[e] = from_c128<C>(shifted_val(P, P.Lidx[e], sg));
    }
    // from both ends to the middle: 0 .. mid-1, then nb-1 .. mid+1, then mid
    const int mid = P.mid;
    for (int t = 0; t < nb; ++t) {
        const int k = t < mid ? t : (t < nb - 1 ? nb - 1 - (t - mid) : mid);
        C* D = Dinv + (size_t)k * TT;
        const int64_t g0 = (int64_t)k * T;
        for (int i = warp; i < T; i += nw)
            for (int c = lane; c < T; c += 32) D[(size_t)i * T + c] = czero<C>();
        __syncthreads();
        for (int i = tid; i < T; i += bd) {
            int64_t g = g0 + i;
            if (g < P.n) {
                for (int64_t e = P.rp[g]; e < P.rp[g + 1]; ++e) {
                    int64_t j = P.ci[e];
                    if (j >= g0 && j < g0 + T) D[(size_t)i * T + (j - g0)] = from_c128<C>(shifted_val(P, e, sg));
                }
            } else {
                D[(size_t)i * T + i] = from_c128<C>(make_double2(1.0, 0.0));
            }
        }
        __syncthreads();
        {
            // E of the outer neighbour; mid: block mid-1's, columns from T on block mid+1's
            const C* Ep = E + (size_t)(k <= mid ? max(k - 1, 0) : min(k + 1, nb - 1)) * TT;
            const C* Ep2 = E + (size_t)min(k + 1, nb - 1) * TT;
            const C* Lval = Dinv + factor_lval_offset(P);
            for (int i = warp; i < T; i += nw) {
                const int64_t g = g0 + i;
                if (g >= P.n) continue;
                const int e0 = P.Lptr[g], e1 = P.Lptr[g + 1];
                for (int c = lane; c < T; c += 32) {
                    C acc = czero<C>();
                    for (int e = e0; e < e1; ++e) {
                        const int col = P.Lcol[e];
                        acc = cfma(Lval[e], col < T ? Ep[(size_t)col * T + c] : Ep2[(size_t)(col - T) * T + c], acc);
                    }
                    D[(size_t)i * T + c] = csub(D[(size_t)i * T + c], acc);
                }
            }
            __syncthreads();
        }
        // Gauss–Jordan inversion in place with partial pivoting (|re| + |im|)
        for (int p = 0; p < T; ++p) {
            double best = -1.0;
            int bi = p;
            for (int r = p + tid; r < T; r += bd) {
                double v = mag1(D[(size_t)r * T + p]);
                if (v > best) { best = v; bi = r; }
            }
            for (int o = 16; o > 0; o >>= 1) {
                double ov = __shfl_xor_sync(0xffffffffu, best, o);
                int oi = __shfl_xor_sync(0xffffffffu, bi, o);
                if (ov > best || (ov == best && oi < bi)) { best = ov; bi = oi; }
            }
            if (lane == 0) { redv[warp] = best; redi[warp] = bi; }
            __syncthreads();
            if (tid == 0) {
                double b = redv[0];
                int i0 = redi[0];
                for (int w = 1; w < nw; ++w)
                    if (redv[w] > b || (redv[w] == b && redi[w] < i0)) { b = redv[w]; i0 = redi[w]; }
                piv[p] = i0;
                if (!(b > 0.0)) atomicExch(err, 1);  // singular Schur complement
            }
            __syncthreads();
            const int r = piv[p];
            if (r != p) {
                for (int c = tid; c < T; c += bd) {
                    C a = D[(size_t)p * T + c];
                    D[(size_t)p * T + c] = D[(size_t)r * T + c];
                    D[(size_t)r * T + c] = a;
                }
                __syncthreads();
            }
            C pv = D[(size_t)p * T + p];
            if (pv.x == 0 && pv.y == 0) pv.x = (decltype(pv.x))1e-30;  // singular: flagged above
            const C inv = cdiv(from_c128<C>(make_double2(1.0, 0.0)), pv);
            for (int c = tid; c < T; c += bd) {
                rowp[c] = (c == p) ? inv : cmul(D[(size_t)p * T + c], inv);
                colp[c] = D[(size_t)c * T + p];
            }
            __syncthreads();
            for (int i = warp; i < T; i += nw) {
                C* Di = D + (size_t)i * T;
                if (i == p) {
                    for (int c = lane; c < T; c += 32) Di[c] = rowp[c];
                } else {
                    const C f = colp[i];
                    for (int c = lane; c < T; c += 32) {
                        C base = (c == p) ? czero<C>() : Di[c];
                        const C rp = rowp[c];
                        base.x -= f.x * rp.x - f.y * rp.y;
                        base.y -= f.x * rp.y + f.y * rp.x;
                        Di[c] = base;
                    }
                }
            }
            __syncthreads();
        }
        for (int p = T - 1; p >= 0; --p) {
            const int r = piv[p];
            if (r != p) {
                for (int i = tid; i < T; i += bd) {
                    C a = D[(size_t)i * T + p];
                    D[(size_t)i * T + p] = D[(size_t)i * T + r];
                    D[(size_t)i * T + r] = a;
                }
                __syncthreads();
            }
        }
        // E_k = Dinv_k K_{k,inner(k)}, that block in column-compressed form
        if (k != mid) {
            C* Ek = E + (size_t)k * TT;
            const int32_t* cp = P.up_ptr + (size_t)k * (T + 1);
            for (int rr = warp; rr < T; rr += nw)
                for (int c = lane; c < T; c += 32) {
                    C acc = czero<C>();
                    for (int q = cp[c]; q < cp[c + 1]; ++q)
                        acc = cfma(D[(size_t)rr * T + P.up_row[q]], from_c128<C>(shifted_val(P, P.up_idx[q], sg)), acc);
                    Ek[(size_t)rr * T + c] = acc;
                }
        }
        __syncthreads();
    }
}

static size_t factor_smem(int T, int precision) {
    size_t cs = precision == SIM_FP64 ? sizeof(double2) : sizeof(float2);
    return 2 * T * cs + (T + 2) * sizeof(int) + 32 * sizeof(double) + 32 * sizeof(int) + 16;
}

void factor_shifts(const Pencil& P, int precision, const int* d_shift_list, int count, const double2* d_sigma,
                   void* const* d_factor_ptrs, cudaStream_t st) {
    if (count <= 0) return;
    static int* d_err = nullptr;
    if (!d_err) SIM_CUDA(cudaMalloc(&d_err, sizeof(int)));
    SIM_CUDA(cudaMemsetAsync(d_err, 0, sizeof(int), st));
    size_t sm = factor_smem(P.T, precision);
    kprof_begin("factor", st);
    if (precision == SIM_FP64) {
        SIM_CUDA(cudaFuncSetAttribute(k_factor<double2>, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)sm));
        k_factor<double2><<<count, FACTOR_THREADS, sm, st>>>(P, d_shift_list, d_sigma, d_factor_ptrs, d_err);
        SIM_LAUNCH_CHECK();
    } else {
        SIM_CUDA(cudaFuncSetAttribute(k_factor<float2>, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)sm));
        k_factor<float2><<<count, FACTOR_THREADS, sm, st>>>(P, d_shift_list, d_sigma, d_factor_ptrs, d_err);
        SIM_LAUNCH_CHECK();
    }
    {
        const double cs = precision == SIM_FP64 ? sizeof(double2) : sizeof(float2);
        const double TT = (double)P.T * P.T;
        kprof_end("factor", st, count * (2.0 * P.nb * TT * cs), count * 8.0 * P.nb * TT * P.T);
    }
}

// ---------------------------------------------------------------------------
// sparse applies
// ---------------------------------------------------------------------------
// ||v||^2 over the CTA's (256) threads to *out
__device__ __forceinline__ void block_norm2(double2 v, double* out) {
    __shared__ double red[8];
    const double s = warp_sum(fma(v.x, v.x, v.y * v.y));
    __syncthreads();  // an earlier sum has been read
    if ((threadIdx.x & 31) == 0) red[threadIdx.x >> 5] = s;
    __syncthreads();
    if (threadIdx.x == 0) {
        double t = red[0];
        for (int w = 1; w < 8; ++w) t += red[w];
        *out = t;
    }
}

// y = (A - σB) x, or y = rhs - (A - σB) x when rhs_slot >= 0, for SPMV_RJ
// active jobs per thread: a thread owns one row and reads its indices and
// values once for all of its jobs (the jobs' shifts differ only on B's
// entries), then gathers each job's x.  Every job's row sum runs over the
// row's entries in order, so the result does not depend on SPMV_RJ, which the
// autotuner picks per matrix (1, 2, 4 or 8).
// With a right-hand side each CTA also leaves ||y||^2 of its rows in js.rpart.
template <int SPMV_RJ>
__global__ void __launch_bounds__(256) k_spmv_jobs(Pencil P, JobSpace js, int x_slot, int y_slot, int rhs_slot,
                                                   const double2* sigma, int nactive) {
    const int64_t row = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
    const int jb = blockIdx.y * SPMV_RJ;
    if (rhs_slot < 0 && row >= P.n) return;
    const bool in = row < P.n;
    const int64_t g = in ? row : P.n - 1;  // the last CTA's spare threads only take part in the sums
    const int nj = min(SPMV_RJ, nactive - jb);
    const double2* x[SPMV_RJ];
    double2 sg[SPMV_RJ], acc[SPMV_RJ];
#pragma unroll
    for (int r = 0; r < SPMV_RJ; ++r) {
        const int job = js.d_active[jb + (r < nj ? r : 0)];
        sg[r] = sigma[js.d_jobshift[job]];
        x[r] = js.vec + (size_t)job * js.vstride + (size_t)x_slot * js.n;
        acc[r] = make_double2(0.0, 0.0);
    }
    const int64_t e0 = P.rp[g], e1 = P.rp[g + 1];
    if (P.b_kind <= 1) {
        // B = I or diagonal: A - σB differs from A on the diagonal only, where
        // σB_gg is subtracted (a select rather than a branch keeps the loads in flight)
        const double2 b = P.Bdiag[g];
        double2 sb[SPMV_RJ];
#pragma unroll
        for (int r = 0; r < SPMV_RJ; ++r) sb[r] = cmul(sg[r], b);
        for (int64_t e = e0; e < e1; ++e) {
            const int64_t j = P.ci[e];
            const double2 a = P.Ka[e];
            const bool d = j == g;
#pragma unroll
            for (int r = 0; r < SPMV_RJ; ++r) {
                if (r < nj) {
                    const double2 v = make_double2(d ? a.x - sb[r].x : a.x, d ? a.y - sb[r].y : a.y);
                    acc[r] = cfma(v, x[r][j], acc[r]);
                }
            }
        }
    } else {
        for (int64_t e = e0; e < e1; ++e) {
            const int64_t j = P.ci[e];
            const double2 a = P.Ka[e], b = P.Kb[e];
#pragma unroll
            for (int r = 0; r < SPMV_RJ; ++r) {
                if (r < nj) acc[r] = cfma(csub(a, cmul(sg[r], b)), x[r][j], acc[r]);
            }
        }
    }
#pragma unroll
    for (int r = 0; r < SPMV_RJ; ++r) {
        if (r >= nj) break;
        const int job = js.d_active[jb + r];
        double2 v = acc[r];
        if (rhs_slot >= 0) v = csub(js.vec[(size_t)job * js.vstride + (size_t)rhs_slot * js.n + g], v);
        if (in) js.vec[(size_t)job * js.vstride + (size_t)y_slot * js.n + g] = v;
        if (rhs_slot >= 0) block_norm2(in ? v : make_double2(0.0, 0.0), js.rpart + (size_t)job * js.nblk + blockIdx.x);
    }
}

static void spmv_launch_rj(int rj, const Pencil& P, const JobSpace& js, int nactive, int x_slot, int y_slot,
                           int rhs_slot, const double2* d_sigma, cudaStream_t st) {
    const dim3 grid(cdiv_up(P.n, 256), cdiv_up(nactive, rj));
    switch (rj) {
        case 1: k_spmv_jobs<1><<<grid, 256, 0, st>>>(P, js, x_slot, y_slot, rhs_slot, d_sigma, nactive); break;
        case 2: k_spmv_jobs<2><<<grid, 256, 0, st>>>(P, js, x_slot, y_slot, rhs_slot, d_sigma, nactive); break;
        case 8: k_spmv_jobs<8><<<grid, 256, 0, st>>>(P, js, x_slot, y_slot, rhs_slot, d_sigma, nactive); break;
        default: k_spmv_jobs<4><<<grid, 256, 0, st>>>(P, js, x_slot, y_slot, rhs_slot, d_sigma, nactive); break;
    }
    SIM_LAUNCH_CHECK();
}

// y = (A - σB)x (or rhs - (A - σB)x) for the active jobs of the inner solver, timed as "spmv":
// algorithmic bytes: the matrix (20·nnz + 4(n+1)) once per RJ jobs, and per
// job x and y (32n, +16n with rhs); 8·nnz flops per job.  Jobs per thread
// (RJ) autotuned per matrix and batch size class.
static void launch_spmv(const Pencil& P, const JobSpace& js, int nactive, int x_slot, int y_slot, int rhs_slot,
                        const double2* d_sigma, cudaStream_t st) {
    static const int rjs[4] = {1, 2, 4, 8};
    const int cls = nactive < 4 ? nactive : (nactive < 16 ? 4 : 16);
    const std::string key = "spmv:" + std::to_string(P.n) + ":" + std::to_string(P.nnz) + ":" + std::to_string(cls);
    bool timing = false;
    const int rj = nactive == 1 ? 1 : rjs[autotune_begin(key, 4, st, &timing)];
    kprof_begin("spmv", st);
    spmv_launch_rj(rj, P, js, nactive, x_slot, y_slot, rhs_slot, d_sigma, st);
    if (timing) autotune_end(key, st);
    kprof_end("spmv", st,
              cdiv_up(nactive, rj) * (20.0 * P.nnz + 4.0 * (P.n + 1)) + nactive * (rhs_slot >= 0 ? 48.0 : 32.0) * P.n,
              nactive * 8.0 * P.nnz);
}

void spmv_shifted_jobs(const Pencil& P, const JobSpace& js, int nactive, const double*, int x_slot, int y_slot,
                       const double2* d_sigma, cudaStream_t st) {
    if (nactive <= 0) return;
    // untimed: also the path of the no-allocation entry point
    spmv_launch_rj(4, P, js, nactive, x_slot, y_slot, -1, d_sigma, st);
}

// y = (A - σB) x on the caller's vectors, σ by value: the same sums in the same
// order as k_spmv_jobs.  A thread per row: a call of a few thousand rows is bounded by
// its launch and the wait for it, so it is one launch (three uploads, two copies of the
// vectors and the job kernel before).  n = 40,000: 40 -> 23 us a call.
__global__ void __launch_bounds__(256) k_apply_shifted(Pencil P, double2 sg, const double2* x, double2* y) {
    const int64_t g = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
    if (g >= P.n) return;
    double2 acc = make_double2(0.0, 0.0);
    const int64_t e0 = P.rp[g], e1 = P.rp[g + 1];
    if (P.b_kind <= 1) {
        const double2 sb = cmul(sg, P.Bdiag[g]);
        for (int64_t e = e0; e < e1; ++e) {
            const int64_t j = P.ci[e];
            const double2 a = P.Ka[e];
            acc = cfma(j == g ? csub(a, sb) : a, x[j], acc);
        }
    } else {
        for (int64_t e = e0; e < e1; ++e) acc = cfma(csub(P.Ka[e], cmul(sg, P.Kb[e])), x[P.ci[e]], acc);
    }
    y[g] = acc;
}

void apply_shifted(const Pencil& P, double2 sg, const double2* x, double2* y, cudaStream_t st) {
    k_apply_shifted<<<cdiv_up(P.n, 256), 256, 0, st>>>(P, sg, x, y);
    SIM_LAUNCH_CHECK();
}

__global__ void k_apply_B(Pencil P, const double2* x, double2* y) {
    int64_t g = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
    if (g >= P.n) return;
    if (P.b_kind == 0) { y[g] = x[g]; return; }
    if (P.b_kind == 1) { y[g] = cmul(P.Bdiag[g], x[g]); return; }
    double2 acc = make_double2(0.0, 0.0);
    for (int64_t e = P.rp[g]; e < P.rp[g + 1]; ++e) acc = cfma(P.Kb[e], x[P.ci[e]], acc);
    y[g] = acc;
}

void apply_B(const Pencil& P, const double2* x, double2* y, cudaStream_t st) {
    k_apply_B<<<cdiv_up(P.n, 256), 256, 0, st>>>(P, x, y);
    SIM_LAUNCH_CHECK();
}

// u_job = B v_{j, job}  for all active jobs (V slot j -> vec slot)
__global__ void k_apply_B_jobs(Pencil P, JobSpace js, int j, int y_slot) {
    const int job = js.d_active[blockIdx.y];
    const double2* x = js.V + ((size_t)job * (js.m + 1) + j) * js.n;
    double2* y = js.vec + (size_t)job * js.vstride + (size_t)y_slot * js.n;
    int64_t g = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
    if (g >= P.n) return;
    if (P.b_kind == 0) { y[g] = x[g]; return; }
    if (P.b_kind == 1) { y[g] = cmul(P.Bdiag[g], x[g]); return; }
    double2 acc = make_double2(0.0, 0.0);
    for (int64_t e = P.rp[g]; e < P.rp[g + 1]; ++e) acc = cfma(P.Kb[e], x[P.ci[e]], acc);
    y[g] = acc;
}

// ---------------------------------------------------------------------------
// batched FGMRES(k) with the block factorisation as right preconditioner
// ---------------------------------------------------------------------------
// x = Z y (+ x after the first cycle), y from the end of the cycle (gs_finish.cuh);
// each CTA leaves ||x||^2 of its rows in js.xpart
__global__ void __launch_bounds__(256) k_gm_update_x(JobSpace js, int first) {
    const int job = js.d_active[blockIdx.y];
    const int k = js.k;
    const int steps = js.istat[(size_t)job * IS_N + IS_STEPS];
    const int64_t gi = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
    double2 x = make_double2(0.0, 0.0);
    if (gi < js.n) {
        double2* base = js.vec + (size_t)job * js.vstride + gi;
        if (!first) x = base[(size_t)VS_X * js.n];
        const double2* z = base + (size_t)vs_Z(k) * js.n;
#pragma unroll 4
        for (int q = 0; q < steps; ++q) x = cfma(z[(size_t)q * js.n], js.y[(size_t)job * k + q], x);
        base[(size_t)VS_X * js.n] = x;
    }
    block_norm2(x, js.xpart + (size_t)job * js.nblk + blockIdx.x);
}

// The end of a cycle of one job with the squared residual norm s and ||x||^2 = sx.
__device__ void gm_check_job(const JobSpace& js, int job, double s, double sx, double tol, int max_iter,
                             const double2* sigma, double anorm, double bnorm) {
    double* sc = js.scal + (size_t)job * SC_N;
    int* is = js.istat + (size_t)job * IS_N;
    const double r = sqrt(s);
    const double rel = sc[SC_RNORM0] > 0 ? r / sc[SC_RNORM0] : 0.0;
    const double prev = sc[SC_GAMMA] > 0 && sc[SC_RNORM0] > 0 ? sc[SC_GAMMA] / sc[SC_RNORM0] : INFINITY;
    sc[SC_WORST] = rel;
    if (rel <= tol) {
        is[IS_DONE] = 1;
        return;
    }
    // The rounding floor of the explicit residual b - (A - σB)x in FP64: about
    // ε ||A - σB|| ||x|| / ||b|| (||A - σB|| <= ||A||_inf + |σ| ||B||_inf); near an
    // eigenvalue ||x|| / ||b|| is large and the floor rises above tol.
    const double2 sg = sigma[js.d_jobshift[job]];
    const double floor_rel = sc[SC_RNORM0] > 0
                                 ? 32.0 * 1.1102230246251565e-16 * (anorm + hypot(sg.x, sg.y) * bnorm) * sqrt(sx) /
                                       sc[SC_RNORM0]
                                 : 0.0;
    const double lim = fmax(tol, floor_rel);
    // A restart cycle that did not halve the residual has stagnated.  Stop early
    // only at the rounding floor: after one such cycle if the residual is already
    // within 10 max(tol, floor), else after two in a row.  An early stop (or the
    // iteration cap) accepts the solve within 100 max(tol, floor), counted as
    // loose, else fails.
    const int stall = rel > 0.5 * prev ? is[IS_STALL] + 1 : 0;
    is[IS_STALL] = stall;
    if (is[IS_ITERS] >= max_iter || (stall >= 1 && rel <= 10.0 * lim) || stall >= 2) {
        const int ok = rel <= 100.0 * lim;
        is[IS_DONE] = ok ? 1 : -1;
        is[IS_LOOSE] = ok;
    }
}

// explicit residual norm and ||x|| from their partial sums, one CTA per job: done
// if <= tol * rnorm0; the job's state goes to the host's copy
__global__ void __launch_bounds__(256) k_gm_check(JobSpace js, double tol, int max_iter, const double2* sigma,
                                                  double anorm, double bnorm) {
    const int job = js.d_active[blockIdx.x];
    double s = 0.0, sx = 0.0;
    for (int c = threadIdx.x; c < js.nblk; c += 256) {
        s += js.rpart[(size_t)job * js.nblk + c];
        sx += js.xpart[(size_t)job * js.nblk + c];
    }
    s = warp_sum(s);
    sx = warp_sum(sx);
    __shared__ double red[2][8];
    if ((threadIdx.x & 31) == 0) {
        red[0][threadIdx.x >> 5] = s;
        red[1][threadIdx.x >> 5] = sx;
    }
    __syncthreads();
    if (threadIdx.x != 0) return;
    s = sx = 0.0;
    for (int w = 0; w < 8; ++w) {
        s += red[0][w];
        sx += red[1][w];
    }
    gm_check_job(js, job, s, sx, tol, max_iter, sigma, anorm, bnorm);
    for (int i = 0; i < IS_N; ++i) js.h_istat[job * IS_N + i] = js.istat[job * IS_N + i];
    js.h_worst[job] = js.scal[(size_t)job * SC_N + SC_WORST];
}

namespace {

// The active list on the device, in this order (nothing to do if it is there).
void upload_active(const JobSpace& js, const std::vector<int>& a, cudaStream_t st) {
    JobHost& h = *js.host;
    if (h.uploaded == a) return;
    // the previous upload must have left the pinned buffer before it is refilled
    SIM_CUDA(cudaEventSynchronize(h.act_ev));
    std::copy(a.begin(), a.end(), h.act);
    SIM_CUDA(cudaMemcpyAsync(js.d_active, h.act, sizeof(int) * a.size(), cudaMemcpyHostToDevice, st));
    SIM_CUDA(cudaEventRecord(h.act_ev, st));
    h.uploaded = a;
}

GSArgs gs_args(const JobSpace& js) {
    GSArgs a;
    a.n = js.n;
    a.active = js.d_active;
    a.h_istat = js.h_istat;
    a.part = js.partial;
    a.pw = js.pw;
    a.hsum = js.hsum;
    a.fin = js.fin;
    a.need = js.need;
    a.ticket = js.ticket;
    a.J = js.J;
    return a;
}

GmArgs gm_args(const JobSpace& js, int mode, int i, int first, double tol, int max_iter) {
    GmArgs g;
    g.mode = mode;
    g.k = js.k;
    g.i = i;
    g.first = first;
    g.tol = tol;
    g.max_iter = max_iter;
    g.Hg = js.Hg;
    g.cs = js.cs;
    g.sn = js.sn;
    g.g = js.g;
    g.y = js.y;
    g.scal = js.scal;
    g.istat = js.istat;
    return g;
}

}  // namespace

bool inner_solve(const Pencil& P, const sim_options& opt, JobSpace& js, const std::vector<int>& jobs,
                 const double2* d_sigma, void* const* d_factor_ptrs, cudaStream_t st, InnerStats& stats) {
    if (jobs.empty()) return true;
    const int k = js.k;
    auto rows_grid = [&](int na) { return dim3(cdiv_up(js.n, 256), na); };
    const int* ist = js.h_istat;
    std::vector<int> cyc = jobs;  // jobs that start a cycle
    bool first = true;
    bool ok = true;
    // Iterations that every job of the last solve took: the host issues that many
    // without waiting for the flags in between (a job whose cycle has ended takes no
    // further columns, whatever is computed for it).
    int& usual = js.host->usual_steps;
    while (!cyc.empty()) {
        upload_active(js, cyc, st);
        {
            // q_0 = r / ||r||, the cycle's state
            GSArgs a = gs_args(js);
            a.w = js.vec + (size_t)VS_Q0 * js.n;
            a.wstride = js.vstride;
            a.src = js.vec + (size_t)(first ? VS_RHS : VS_R) * js.n;
            a.sstride = js.vstride;
            a.gm = gm_args(js, GmArgs::START, 0, first ? 1 : 0, opt.inner_tol, opt.inner_max_iter);
            gram_schmidt(a, (int)cyc.size(), st);
        }
        std::vector<int> act = cyc;
        for (int i = 0; i < k && !act.empty(); ++i) {
            const int na = (int)act.size();
            upload_active(js, act, st);
            if (P.sep)
                separable_apply(P.sep->S, opt.precision, js, act, VS_Q0 + i, vs_Z(k) + i, d_sigma, *P.sep->ar, st);
            else if (!js.h_jobshift ||
                     !block_solve_cluster(P, opt.precision, js, act, VS_Q0 + i, vs_Z(k) + i, d_sigma, d_factor_ptrs, st))
                throw std::runtime_error("LIMIT:block size " + std::to_string(P.T) +
                                         " too large for the cluster block solve's shared memory");
            launch_spmv(P, js, na, vs_Z(k) + i, VS_Q0 + i + 1, -1, d_sigma, st);
            GSArgs a = gs_args(js);
            a.basis = js.vec + (size_t)VS_Q0 * js.n;
            a.bstride = js.vstride;
            a.w = js.vec + (size_t)(VS_Q0 + i + 1) * js.n;
            a.wstride = js.vstride;
            a.cnt = i + 1;
            a.dgks = 1;
            a.gm = gm_args(js, GmArgs::STEP, i, 0, opt.inner_tol, opt.inner_max_iter);
            gram_schmidt(a, na, st);
            if (first && i + 1 < usual) continue;
            SIM_CUDA(cudaStreamSynchronize(st));
            block_solve_check(*js.host);
            std::vector<int> next;
            for (int j : act)
                if (!ist[j * IS_N + IS_CYCLE_DONE]) next.push_back(j);
            act.swap(next);
        }
        const int ni = (int)cyc.size();
        upload_active(js, cyc, st);
        k_gm_update_x<<<rows_grid(ni), 256, 0, st>>>(js, first ? 1 : 0);
        SIM_LAUNCH_CHECK();
        launch_spmv(P, js, ni, VS_X, VS_R, VS_RHS, d_sigma, st);
        k_gm_check<<<ni, 256, 0, st>>>(js, opt.inner_tol, opt.inner_max_iter, d_sigma, P.anorm, P.bnorm);
        SIM_LAUNCH_CHECK();
        SIM_CUDA(cudaStreamSynchronize(st));
        block_solve_check(*js.host);
        if (first) {
            usual = k;
            for (int j : cyc) usual = std::min(usual, ist[j * IS_N + IS_STEPS]);
        }
        first = false;
        std::vector<int> again;
        for (int j : cyc) {
            int d = ist[j * IS_N + IS_DONE];
            if (d == 0) again.push_back(j);
            if (d == -1) ok = false;
        }
        cyc.swap(again);
    }
    for (int j : jobs) {
        int it = ist[j * IS_N + IS_ITERS];
        stats.solves += 1;
        stats.iters += it;
        stats.max_iters = std::max(stats.max_iters, it);
        stats.worst = std::max(stats.worst, js.h_worst[j]);
        stats.loose += ist[j * IS_N + IS_LOOSE];
        if (ist[j * IS_N + IS_DONE] != 1) ok = false;
    }
    return ok;
}

// ---------------------------------------------------------------------------
// Arnoldi with CGS2 for all jobs of the space
// ---------------------------------------------------------------------------
__global__ void k_arnoldi_init(JobSpace js, int nactive) {
    int t = blockIdx.x * blockDim.x + threadIdx.x;
    if (t >= nactive) return;
    const int job = js.d_active[t];
    js.meff[job] = js.m;
    js.istat[job * IS_N + IS_BROKEN] = 0;
    js.h_istat[job * IS_N + IS_BROKEN] = 0;
    double2* H = js.H + (size_t)job * (js.m + 1) * js.m;
    for (int e = 0; e < (js.m + 1) * js.m; ++e) H[e] = make_double2(0.0, 0.0);
}

__global__ void k_store_beta(JobSpace js, int nactive) {
    int t = blockIdx.x * blockDim.x + threadIdx.x;
    if (t >= nactive) return;
    const int job = js.d_active[t];
    js.beta[job] = js.g[(size_t)job * (js.k + 1)].x;
}

bool arnoldi(const Pencil& P, const sim_options& opt, JobSpace& js, const double2* d_sigma,
             void* const* d_factor_ptrs, cudaStream_t st, InnerStats& stats, bool single_pass) {
    const int J = js.J, m = js.m;
    std::vector<int> all(J);
    for (int j = 0; j < J; ++j) all[j] = j;
    auto rows_grid = [&](int na) { return dim3(cdiv_up(js.n, 256), na); };
    bool ok = inner_solve(P, opt, js, all, d_sigma, d_factor_ptrs, st, stats);  // b = K^{-1} f
    upload_active(js, all, st);
    k_arnoldi_init<<<cdiv_up(J, 128), 128, 0, st>>>(js, J);
    SIM_LAUNCH_CHECK();
    {
        // beta = ||b||, v_1 = b / beta   (the norm lands in g[job*(k+1)] as scratch)
        GSArgs a = gs_args(js);
        a.w = js.V;
        a.wstride = (int64_t)(m + 1) * js.n;
        a.src = js.vec + (size_t)VS_X * js.n;
        a.sstride = js.vstride;
        a.hcol = js.g;
        a.hstride = js.k + 1;
        gram_schmidt(a, J, st);
    }
    k_store_beta<<<cdiv_up(J, 128), 128, 0, st>>>(js, J);
    SIM_LAUNCH_CHECK();
    std::vector<int> act = all;
    for (int j = 0; j < m && !act.empty(); ++j) {
        const int na = (int)act.size();
        upload_active(js, act, st);
        k_apply_B_jobs<<<rows_grid(na), 256, 0, st>>>(P, js, j, VS_RHS);
        SIM_LAUNCH_CHECK();
        ok = inner_solve(P, opt, js, act, d_sigma, d_factor_ptrs, st, stats) && ok;
        upload_active(js, act, st);
        GSArgs a = gs_args(js);
        a.basis = js.V;
        a.bstride = (int64_t)(m + 1) * js.n;
        a.w = js.V + (size_t)(j + 1) * js.n;
        a.wstride = (int64_t)(m + 1) * js.n;
        a.src = js.vec + (size_t)VS_X * js.n;
        a.sstride = js.vstride;
        a.hcol = js.H + (size_t)j * (m + 1);
        a.hstride = (int64_t)(m + 1) * m;
        a.cnt = j + 1;
        a.Hfull = js.H;
        a.Hstride = (int64_t)(m + 1) * m;
        a.Hld = m + 1;
        a.j = j;
        a.btol = opt.breakdown_tol;
        a.meff = js.meff;
        a.istat = js.istat;
        a.single = single_pass ? 1 : 0;
        gram_schmidt(a, na, st);
        SIM_CUDA(cudaStreamSynchronize(st));
        std::vector<int> next;
        for (int q : act)
            if (!js.h_istat[q * IS_N + IS_BROKEN]) next.push_back(q);
        act.swap(next);
    }
    SIM_CUDA(cudaStreamSynchronize(st));
    return ok;
}

int max_jobs_for_memory(int64_t n, int m, int k) {
    size_t fr = 0, tot = 0;
    SIM_CUDA(cudaMemGetInfo(&fr, &tot));
    const double per_job = (double)(vs_count(k) + m + 1 + 2) * (double)n * sizeof(double2);
    const double jobs = 0.4 * (double)tot / per_job;
    return (int)std::max(1.0, std::min(jobs, 1e6));
}

JobSpace make_jobspace(DeviceArena& ar, cudaStream_t st, int J, int k, int m, int64_t n, const std::string& tag) {
    JobSpace js;
    js.J = J;
    js.k = k;
    js.m = m;
    js.n = n;
    const int nv = vs_count(js.k);
    js.vstride = (int64_t)nv * js.n;
    js.vec = ar.get<double2>(tag + "vec", (int64_t)J * js.vstride);
    js.V = ar.get<double2>(tag + "V", (int64_t)J * (js.m + 1) * js.n);
    js.H = ar.get<double2>(tag + "H", (int64_t)J * (js.m + 1) * js.m);
    js.beta = ar.get<double>(tag + "beta", J);
    js.meff = ar.get<int>(tag + "meff", J);
    js.Hg = ar.get<double2>(tag + "Hg", (int64_t)J * (js.k + 1) * js.k);
    js.cs = ar.get<double2>(tag + "cs", (int64_t)J * js.k);
    js.sn = ar.get<double2>(tag + "sn", (int64_t)J * js.k);
    js.g = ar.get<double2>(tag + "g", (int64_t)J * (js.k + 1));
    js.scal = ar.get<double>(tag + "scal", (int64_t)J * SC_N);
    js.istat = ar.get<int>(tag + "istat", (int64_t)J * IS_N);
    js.y = ar.get<double2>(tag + "y", (int64_t)J * js.k);
    js.pw = std::max(js.m + 2, js.k + 2);
    js.partial = ar.get<double2>(tag + "partial", gs_grid_partials(js.n, J, js.pw));
    js.hsum = ar.get<double2>(tag + "hsum", (int64_t)2 * J * js.pw);
    js.fin = ar.get<double>(tag + "fin", J);
    js.need = ar.get<int>(tag + "need", J);
    js.ticket = ar.get<int>(tag + "ticket", J);
    js.nblk = cdiv_up(js.n, 256);
    js.xpart = ar.get<double>(tag + "xpart", (int64_t)J * js.nblk);
    js.rpart = ar.get<double>(tag + "rpart", (int64_t)J * js.nblk);
    js.host = ar.job_host(tag, J);
    js.h_istat = js.host->istat;
    js.h_worst = js.host->worst;
    js.d_jobshift = ar.get<int>(tag + "jobshift", J);
    js.d_active = ar.get<int>(tag + "active", J);
    SIM_CUDA(cudaMemsetAsync(js.istat, 0, sizeof(int) * J * IS_N, st));
    SIM_CUDA(cudaMemsetAsync(js.scal, 0, sizeof(double) * J * SC_N, st));
    SIM_CUDA(cudaMemsetAsync(js.ticket, 0, sizeof(int) * J, st));
    return js;
}

}  // namespace sim
