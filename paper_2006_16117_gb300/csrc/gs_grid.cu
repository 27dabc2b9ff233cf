// The Gram–Schmidt step of gs_cluster.cu over the whole GPU: for vectors that a
// cluster's shared memory does not hold, and for few jobs of long vectors, where
// 16 SMs a job would leave the FP64 pipes of the others idle (one to five jobs of
// n = 40,000: 15 us a launch of sums, 21 of an update, where a cluster of 8 CTAs
// took 152 us a call; one job of n = 10^6, up to seven vectors: 55 and 58 us).
//
// A job's rows are cut into chunks, a CTA each, so that the active jobs' chunks
// fill the GPU once; a thread holds its rows of w in registers.  Every kernel
// ends with a sum over the chunks: a CTA writes its partial sums, and the last
// one of a job to finish (a ticket counter) adds them in chunk order — the order
// does not depend on which CTA that is — and, after the last pass, takes the step
// of gs_finish.cuh.
//   k_gsg_dots     h = B^H w (and ||w||^2 for the selective second pass)
//   k_gsg_update   w -= B h, then the next pass's sums or the norm
//   k_gsg_scale    w scaled by 1 / norm
// The kernels of a second pass that is not needed return at once.
#include <algorithm>
#include <cmath>

#include "cluster_fit.h"
#include "gs.h"
#include "gs_finish.cuh"

namespace sim {

namespace {

constexpr int GG_T = 256;
constexpr int GG_MAXV = 64;

struct GgShared {
    double red[GG_T / 32][2 * GG_MAXV + 4];
    double2 h[GG_MAXV + 2];
    double2 h1[GG_MAXV + 2];
    double seg[2 * GG_T];
    double fro[GG_T / 32];
    int last;
};

template <int PER>
__device__ __forceinline__ void load_rows(const double2* p, int64_t r0, int64_t n, double2 (&wv)[PER]) {
#pragma unroll
    for (int t = 0; t < PER; ++t) {
        const int64_t r = r0 + threadIdx.x + t * GG_T;
        wv[t] = r < n ? p[r] : make_double2(0.0, 0.0);
    }
}

// this CTA's sums conj(q_i) . w, i < cnt, and ||w||^2 after them if wanted, to S.red
template <int PER>
__device__ __forceinline__ void chunk_sums(const GSArgs& a, const double2* B, const double2 (&wv)[PER], int64_t r0,
                                           int cnt, bool with_norm, GgShared& S) {
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    for_groups(cnt, [&](auto tag, int i0) {
        constexpr int G = decltype(tag)::value;
        double2 acc[G];
#pragma unroll
        for (int g = 0; g < G; ++g) acc[g] = make_double2(0.0, 0.0);
        const double2* qv = B + (size_t)i0 * a.n + r0 + threadIdx.x;
#pragma unroll
        for (int t = 0; t < PER; ++t) {
            if (r0 + threadIdx.x + t * GG_T < a.n) {
#pragma unroll
                for (int g = 0; g < G; ++g) conj_mac(acc[g], qv[(size_t)g * a.n + t * GG_T], wv[t]);
            }
        }
        const double2 s = warp_sum_group<G>(acc);
        if ((lane & (32 / G - 1)) == 0) {
            const int i = i0 + lane / (32 / G);
            S.red[warp][2 * i] = s.x;
            S.red[warp][2 * i + 1] = s.y;
        }
    });
    if (with_norm) {
        double s = 0.0;
#pragma unroll
        for (int t = 0; t < PER; ++t) s = fma(wv[t].x, wv[t].x, fma(wv[t].y, wv[t].y, s));
        s = warp_sum(s);
        if (lane == 0) {
            S.red[warp][2 * cnt] = s;
            S.red[warp][2 * cnt + 1] = 0.0;
        }
    }
}

// Adds the job's V values over its CTAs: true in the last CTA to arrive, which has
// the totals in S.h.
__device__ __forceinline__ bool job_totals(const GSArgs& a, int V, int aj, GgShared& S) {
    const int tid = threadIdx.x, nchunk = gridDim.x;
    double* part = reinterpret_cast<double*>(a.part + ((size_t)aj * nchunk) * a.pw);
    __syncthreads();
    for (int t = tid; t < 2 * V; t += GG_T) {
        double s = S.red[0][t];
#pragma unroll
        for (int w = 1; w < GG_T / 32; ++w) s += S.red[w][t];
        part[(size_t)blockIdx.x * 2 * a.pw + t] = s;
    }
    __threadfence();
    __syncthreads();
    if (tid == 0) S.last = atomicAdd(a.ticket + aj, 1) == nchunk - 1;
    __syncthreads();
    if (!S.last) return false;
    __threadfence();
    // nseg threads a value, each over a contiguous range of chunks
    const int nseg = max(1, GG_T / (2 * V)), per = (nchunk + nseg - 1) / nseg;
    for (int t = tid; t < 2 * V * nseg; t += GG_T) {
        const int v = t % (2 * V), sg = t / (2 * V);
        const int c1 = min(nchunk, (sg + 1) * per);
        double s = 0.0;
#pragma unroll 8
        for (int c = sg * per; c < c1; ++c) s += __ldcg(part + (size_t)c * 2 * a.pw + v);
        S.seg[t] = s;
    }
    __syncthreads();
    for (int v = tid; v < 2 * V; v += GG_T) {
        double s = S.seg[v];
        for (int sg = 1; sg < nseg; ++sg) s += S.seg[v + sg * 2 * V];
        reinterpret_cast<double*>(S.h)[v] = s;
    }
    if (tid == 0) a.ticket[aj] = 0;
    __syncthreads();
    return true;
}

// the totals' way to the next kernel: pass 0 or 1
__device__ __forceinline__ double2* pass_sums(const GSArgs& a, int pass, int aj) {
    return a.hsum + ((size_t)pass * a.J + aj) * a.pw;
}

template <int PER>
__global__ void __launch_bounds__(GG_T) k_gsg_dots(GSArgs a, int pass) {
    const int aj = blockIdx.y;
    if (pass == 1 && a.dgks && !a.need[aj]) return;
    const int job = a.active[aj];
    __shared__ GgShared S;
    const double2* B = a.basis + (size_t)job * a.bstride;
    const double2* src = a.src && pass == 0 ? a.src + (size_t)job * a.sstride : a.w + (size_t)job * a.wstride;
    const int64_t r0 = (int64_t)blockIdx.x * GG_T * PER;
    double2 wv[PER];
    load_rows<PER>(src, r0, a.n, wv);
    const bool with_norm = pass == 0 && a.dgks;
    chunk_sums<PER>(a, B, wv, r0, a.cnt, with_norm, S);
    const int V = a.cnt + (with_norm ? 1 : 0);
    if (!job_totals(a, V, aj, S)) return;
    for (int i = threadIdx.x; i < V; i += GG_T) pass_sums(a, pass, aj)[i] = S.h[i];
}

// w -= B h of this pass (cnt = 0: only the norm); then with `next` the second
// pass's sums, else the norm and, if this was the last pass, the final step
template <int PER>
__global__ void __launch_bounds__(GG_T) k_gsg_update(GSArgs a, int pass, int next) {
    const int aj = blockIdx.y;
    if (pass == 1 && a.dgks && !a.need[aj]) return;
    const int job = a.active[aj], tid = threadIdx.x;
    __shared__ GgShared S;
    const double2* B = a.basis + (size_t)job * a.bstride;
    double2* w = a.w + (size_t)job * a.wstride;
    const double2* src = a.src && pass == 0 ? a.src + (size_t)job * a.sstride : w;
    const int64_t r0 = (int64_t)blockIdx.x * GG_T * PER;
    for (int i = tid; i < a.cnt; i += GG_T) S.h[i] = pass_sums(a, pass, aj)[i];
    double2 wv[PER];
    load_rows<PER>(src, r0, a.n, wv);
    __syncthreads();
    if (a.cnt > 0) {
#pragma unroll 4
        for (int i = 0; i < a.cnt; ++i) {
            const double2* qv = B + (size_t)i * a.n + r0 + tid;
            const double2 hi = S.h[i];
#pragma unroll
            for (int t = 0; t < PER; ++t)
                if (r0 + tid + t * GG_T < a.n) sub_mac(wv[t], qv[t * GG_T], hi);
        }
#pragma unroll
        for (int t = 0; t < PER; ++t) {
            const int64_t r = r0 + tid + t * GG_T;
            if (r < a.n) w[r] = wv[t];
        }
    }
    const int cnt = next ? a.cnt : 0;
    chunk_sums<PER>(a, B, wv, r0, cnt, !next, S);
    __syncthreads();  // S.h read by every thread before the totals overwrite it
    if (!job_totals(a, next ? cnt : 1, aj, S)) return;
    if (next) {
        for (int i = tid; i < cnt; i += GG_T) pass_sums(a, 1, aj)[i] = S.h[i];
        return;
    }
    const double nn = S.h[0].x;
    if (a.dgks && pass == 0 && a.cnt > 0) {
        const int need = !(nn > 0.5 * pass_sums(a, 0, aj)[a.cnt].x);
        if (tid == 0) a.need[aj] = need;
        if (need) return;
    }
    // the coefficients: pass 0's, plus pass 1's if there was one
    for (int i = tid; i < a.cnt; i += GG_T) {
        const double2 h0 = pass_sums(a, 0, aj)[i];
        S.h1[i] = pass == 1 ? cadd(h0, pass_sums(a, 1, aj)[i]) : h0;
    }
    __syncthreads();
    const double hn = sqrt(nn);
    bool broken = !(hn > 0.0);
    if (a.Hfull) {
        const double f = hess_frobenius2(a, job, S.h1, [&](double v) {
            v = warp_sum(v);
            if ((tid & 31) == 0) S.fro[tid >> 5] = v;
            __syncthreads();
            double t = 0.0;
            for (int i = 0; i < GG_T / 32; ++i) t += S.fro[i];
            return t;
        });
        if (hn <= a.btol * sqrt(f)) broken = true;
    }
    if (tid == 0) a.fin[aj] = broken ? 1.0 : 1.0 / hn;
    if (tid < 32) gs_finish(a, job, S.h1, hn, broken);
}

__global__ void __launch_bounds__(GG_T) k_gsg_scale(GSArgs a, int from_src) {
    const int aj = blockIdx.y, job = a.active[aj];
    const double f = a.fin[aj];
    double2* w = a.w + (size_t)job * a.wstride;
    const double2* src = from_src ? a.src + (size_t)job * a.sstride : w;
    const int64_t r = (int64_t)blockIdx.x * GG_T + threadIdx.x;
    if (r >= a.n) return;
    if (f != 1.0 || from_src) w[r] = cscale(src[r], f);
}

// Rows per thread: the chunks of the active jobs fill the GPU once at two CTAs
// an SM, 16 rows a thread at most.
int rows_per_thread(int64_t n, int nactive) {
    int per = 1;
    while (per < 16 && (int64_t)nactive * cdiv_up(n, (int64_t)GG_T * per) > 2 * sm_count()) per *= 2;
    return per;
}

template <int PER> void run(const GSArgs& a, int nactive, cudaStream_t st) {
    const dim3 grid(cdiv_up(a.n, (int64_t)GG_T * PER), nactive);
    const dim3 egrid(cdiv_up(a.n, GG_T), nactive);
    const int from_src = a.cnt == 0 && a.src;
    auto dots = [&](int pass) {
        k_gsg_dots<PER><<<grid, GG_T, 0, st>>>(a, pass);
        SIM_LAUNCH_CHECK();
    };
    auto update = [&](int pass, int next) {
        k_gsg_update<PER><<<grid, GG_T, 0, st>>>(a, pass, next);
        SIM_LAUNCH_CHECK();
    };
    if (a.cnt == 0) {
        update(0, 0);
    } else if (a.single) {
        dots(0);
        update(0, 0);
    } else if (a.dgks) {
        dots(0);
        update(0, 0);
        dots(1);
        update(1, 0);
    } else {
        dots(0);
        update(0, 1);
        update(1, 0);
    }
    k_gsg_scale<<<egrid, GG_T, 0, st>>>(a, from_src);
    SIM_LAUNCH_CHECK();
}

}  // namespace

// A launch costs about 6,000 clocks with its sum over the chunks; FP64
// instructions as in the cluster form, over all SMs.
double gs_grid_cost(int64_t n, int cnt, int passes, int nactive) {
    const int per = rows_per_thread(n, nactive);
    const double ctas = (double)nactive * cdiv_up(n, (int64_t)GG_T * per);
    const double per_warp = per * (4.0 * cnt * passes + 6.0) + 1.2 * cnt * passes + 20.0;
    const double launches = cnt == 0 ? 2.0 : (passes == 4 ? 4.0 : 3.5);
    return per_warp * 64.0 * 2.0 * std::ceil(ctas / sm_count()) + launches * 6000.0;
}

int64_t gs_grid_partials(int64_t n, int J, int pw) {
    int64_t most = 0;
    for (int na = 1; na <= J; na *= 2) {
        // between na and 2 na jobs the rows per thread only grow
        const int64_t jobs = std::min<int64_t>(2 * (int64_t)na - 1, J);
        most = std::max(most, jobs * cdiv_up(n, (int64_t)GG_T * rows_per_thread(n, na)));
    }
    return most * pw;
}

void gs_grid(const GSArgs& a, int nactive, cudaStream_t st) {
    if (a.cnt > GG_MAXV || nactive > a.J) throw CudaError{cudaErrorInvalidValue, "gs_grid: range"};
    switch (rows_per_thread(a.n, nactive)) {
        case 1: run<1>(a, nactive, st); break;
        case 2: run<2>(a, nactive, st); break;
        case 4: run<4>(a, nactive, st); break;
        case 8: run<8>(a, nactive, st); break;
        default: run<16>(a, nactive, st); break;
    }
}

}  // namespace sim
