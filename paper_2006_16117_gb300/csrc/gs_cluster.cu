// Batched classical Gram–Schmidt, applied twice (CGS2), once, or with the
// Daniel–Gragg–Kaufman–Stewart test for the second pass, in one launch: the
// orthogonalisation of w against the cnt basis vectors of its job, the norm,
// the Arnoldi breakdown test, the normalisation and the FGMRES step (Sec. 3.1's
// Arnoldi process; the inner FGMRES uses the same step).
//
// One thread-block cluster per job.  CTA q of the cluster owns E·NT consecutive
// rows and keeps its piece of w in shared memory, so w is read once and written
// once; every pass over the basis is one streaming read.  The complex
// multiply-adds are FP64 and on this GPU the FP64 pipe (two lanes a clock per
// SM), not HBM, bounds the step: the cluster is as large as the number of jobs
// leaves room for, and the sums over lanes are made for eight vectors at a time.
// The partial sums are added in the CTA and across the cluster by reading each
// peer CTA's through distributed shared memory, in rank order — every CTA forms
// the same totals and takes the same decisions.  The only waits are the hardware
// cluster barriers; the partial sums alternate between two buffers, so that a
// pass needs one of them.
//
// gram_schmidt() takes this form or the grid kernels (gs_grid.cu), whichever an
// estimate says is faster: this one cannot use more than 16 SMs a job.  n up to
// 3,600 (six pencils, one to three jobs a call): 52 -> 23 us a call, the Givens
// step's own kernel (7 us) and a copy of w included.
#include <cooperative_groups.h>

#include "cluster_fit.h"
#include "gs.h"
#include "gs_finish.cuh"
#include "gs_shape.h"

namespace cg = cooperative_groups;

namespace sim {

namespace {

constexpr int GC_MAXT = 256;
constexpr int GC_WARPS = GC_MAXT / 32;

struct GcShared {
    double red[GC_WARPS][2 * GC_MAXV + 4];  // per-warp sums, (re, im) per value
    double part[2][2 * GC_MAXV + 4];        // this CTA's sums (read by the peers)
    double2 tot[GC_MAXV + 2];               // cluster totals
    double2 h1[GC_MAXV];                    // coefficients so far
    double fro[GC_WARPS];
};

__global__ void __launch_bounds__(GC_MAXT, 2) k_gs_cluster(GSArgs a, int E) {
    cg::cluster_group cl = cg::this_cluster();
    const int Cg = (int)cl.num_blocks();
    const int q = (int)cl.block_rank();
    const int job = a.active[blockIdx.x / Cg];
    const int tid = threadIdx.x, NT = blockDim.x, lane = tid & 31, warp = tid >> 5, nw = NT >> 5;
    __shared__ GcShared S;
    extern __shared__ double2 wsm[];  // [E][NT]: this CTA's rows of w
    const double2* B = a.basis + (size_t)job * a.bstride;
    double2* w = a.w + (size_t)job * a.wstride;
    const double2* src = a.src ? a.src + (size_t)job * a.sstride : w;
    const int64_t base = (int64_t)q * NT * E + tid;
    const int cnt = a.cnt;
    // rows of this thread: e < Er are below n
    const int Er = base < a.n ? (int)min((int64_t)E, (a.n - base + NT - 1) / NT) : 0;

#pragma unroll 4
    for (int e = 0; e < E; ++e)
        wsm[e * NT + tid] = e < Er ? src[base + (int64_t)e * NT] : make_double2(0.0, 0.0);
    auto sq = [&]() {
        double s = 0.0;
        for (int e = 0; e < Er; ++e) {
            const double2 v = wsm[e * NT + tid];
            s = fma(v.x, v.x, fma(v.y, v.y, s));
        }
        return s;
    };
    int buf = 0;
    // totals of V values whose warps' sums are in S.red
    auto totals = [&](int V) {
        __syncthreads();
        for (int t = tid; t < 2 * V; t += NT) {
            double s = S.red[0][t];
            for (int i = 1; i < nw; ++i) s += S.red[i][t];
            S.part[buf][t] = s;
        }
        cl.sync();  // every CTA's sums are written
        for (int t = tid; t < 2 * V; t += NT) {
            double s = 0.0;
            for (int r = 0; r < Cg; ++r) s += cl.map_shared_rank(&S.part[buf][0], r)[t];
            reinterpret_cast<double*>(S.tot)[t] = s;
        }
        buf ^= 1;  // a peer may still read these: the next sums go to the other buffer
        __syncthreads();
    };
    auto put_norm = [&](int at, double v) {
        v = warp_sum(v);
        if (lane == 0) {
            S.red[warp][2 * at] = v;
            S.red[warp][2 * at + 1] = 0.0;
        }
    };
    // h_i = conj(q_i) . w for i < cnt (and ||w||^2 in slot cnt if `with_norm`)
    auto dots = [&](bool with_norm) {
        for_groups(cnt, [&](auto tag, int i0) {
            constexpr int G = decltype(tag)::value;
            double2 acc[G];
#pragma unroll
            for (int g = 0; g < G; ++g) acc[g] = make_double2(0.0, 0.0);
            const double2* qv = B + (size_t)i0 * a.n + base;
#pragma unroll 2
            for (int e = 0; e < Er; ++e) {
                const double2 v = wsm[e * NT + tid];
#pragma unroll
                for (int g = 0; g < G; ++g) conj_mac(acc[g], qv[(size_t)g * a.n + (int64_t)e * NT], v);
            }
            const double2 s = warp_sum_group<G>(acc);
            if ((lane & (32 / G - 1)) == 0) {
                const int i = i0 + lane / (32 / G);
                S.red[warp][2 * i] = s.x;
                S.red[warp][2 * i + 1] = s.y;
            }
        });
        if (with_norm) put_norm(cnt, sq());
        totals(cnt + (with_norm ? 1 : 0));
    };
    // w -= sum_i q_i h_i with h in S.tot[0..cnt): per element, all i
    auto update = [&]() {
        for (int e = 0; e < Er; ++e) {
            double2 v = wsm[e * NT + tid];
            const double2* qv = B + base + (int64_t)e * NT;
#pragma unroll 8
            for (int i = 0; i < cnt; ++i) sub_mac(v, qv[(size_t)i * a.n], S.tot[i]);
            wsm[e * NT + tid] = v;
        }
    };
    auto norm2 = [&]() {
        put_norm(0, sq());
        totals(1);
        return S.tot[0].x;
    };

    double nn = 0.0;  // ||w||^2 after the last pass
    if (cnt == 0) {
        nn = norm2();
    } else {
        dots(a.dgks != 0);
        const double nb = a.dgks ? S.tot[cnt].x : 0.0;  // ||w||^2 before the first pass
        for (int i = tid; i < cnt; i += NT) S.h1[i] = S.tot[i];
        update();
        // the barriers in totals order S.h1's writes before its reads below
        bool second = !a.single;
        if (a.dgks || a.single) {
            nn = norm2();
            if (a.dgks && !a.single) second = !(nn > 0.5 * nb);
        }
        if (second) {
            dots(false);
            // S.tot now holds the second-pass coefficients
            for (int i = tid; i < cnt; i += NT) S.h1[i] = cadd(S.h1[i], S.tot[i]);
            update();
            nn = norm2();
        }
        __syncthreads();  // S.h1 complete
    }
    const double hn = sqrt(nn);
    bool broken = !(hn > 0.0);
    if (a.Hfull) {
        const double f = hess_frobenius2(a, job, S.h1, [&](double v) {
            v = warp_sum(v);
            if (lane == 0) S.fro[warp] = v;
            __syncthreads();
            double t = 0.0;
            for (int i = 0; i < nw; ++i) t += S.fro[i];
            return t;
        });
        if (hn <= a.btol * sqrt(f)) broken = true;
    }
    if (q == 0 && warp == 0) gs_finish(a, job, S.h1, hn, broken);
    const double inv = broken ? 1.0 : 1.0 / hn;
#pragma unroll 4
    for (int e = 0; e < Er; ++e) {
        const double2 v = wsm[e * NT + tid];
        w[base + (int64_t)e * NT] = broken ? v : cscale(v, inv);
    }
    cl.sync();  // no CTA leaves while a peer reads its sums
}

// The shape of a launch that this device can place (E = 0: none).
GsShape cluster_shape(int64_t n, int cnt, int passes, int nactive) {
    return gs_cluster_shape(n, cnt, passes, nactive, sm_count(), [](int C, int threads, size_t smem) {
        return clusters_that_fit((const void*)k_gs_cluster, C, threads, smem) > 0;
    });
}

void launch_cluster(const GSArgs& a, int nactive, const GsShape& s, cudaStream_t st) {
    cudaLaunchConfig_t cfg = {};
    cfg.gridDim = dim3(nactive * s.Cg);
    cfg.blockDim = dim3(s.NT);
    cfg.dynamicSmemBytes = s.smem;
    cfg.stream = st;
    cudaLaunchAttribute attr[1];
    attr[0].id = cudaLaunchAttributeClusterDimension;
    attr[0].val.clusterDim.x = s.Cg;
    attr[0].val.clusterDim.y = 1;
    attr[0].val.clusterDim.z = 1;
    cfg.attrs = attr;
    cfg.numAttrs = 1;
    SIM_CUDA(cudaLaunchKernelEx(&cfg, k_gs_cluster, a, s.E));
    SIM_LAUNCH_CHECK();
}

}  // namespace

double gs_cluster_cost(int64_t n, int cnt, int passes, int nactive) {
    return cluster_shape(n, cnt, passes, nactive).cost;
}

void gram_schmidt(const GSArgs& args, int nactive, cudaStream_t st) {
    if (nactive <= 0) return;
    GSArgs a = args;
    if (a.single) a.dgks = 0;  // for either form
    const int passes = a.cnt == 0 ? 0 : (a.dgks || a.single ? 2 : 4);
    // algorithmic bytes: w read and written once; the basis streamed once per
    // pass (two passes with the selective test in its usual outcome, four for CGS2)
    kprof_begin("gram_schmidt", st);
    // (the occupancy query only where its answer matters)
    const double grid = gs_grid_cost(a.n, a.cnt, passes, nactive);
    GsShape s = gs_cluster_shape(a.n, a.cnt, passes, nactive, sm_count(), [](int, int, size_t) { return true; });
    if (s.cost <= grid) s = cluster_shape(a.n, a.cnt, passes, nactive);
    if (s.cost <= grid)
        launch_cluster(a, nactive, s, st);
    else
        gs_grid(a, nactive, st);
    kprof_end("gram_schmidt", st, nactive * ((double)passes * a.cnt + 2.0) * a.n * sizeof(double2),
              nactive * 8.0 * (passes * a.cnt + 1.0) * a.n);
}

}  // namespace sim
