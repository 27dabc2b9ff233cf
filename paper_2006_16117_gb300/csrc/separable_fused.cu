// The fast-diagonalisation preconditioner of a two-dimensional pencil in one
// kernel, complex64 (mixed precision; the formulas are in separable.h).
//
// The separate kernels (separable.cu, separable_tc.cu) are seven launches an
// apply, and on grids of up to a few hundred points a side neither their tiles
// nor their memory traffic fill the GPU.  Here a cluster of C CTAs keeps a job's
// vector in shared memory from the scaling to the scaling: CTA q holds Rc lines
// along axis 0, multiplies them by Q_0 and sends every value to the CTA that
// holds its line along axis 1 (distributed shared memory); there come Q_1, the
// division and Q_1 again (the mode products of different axes commute), and the
// values go back for the second Q_0.  Three cluster barriers an apply.
//
// A product is a GEMM of complex rows with a real symmetric matrix on the FP32
// cores: a thread forms RT rows x KT outputs, a complex value times a real one in
// one paired FMA; the rows come from shared memory, Q through a ring of stages
// there.  FP32 products need no splitting as
// on the tensor cores, and every value is summed in FP32 over its line in order.
#include <cooperative_groups.h>

#include <algorithm>
#include <cmath>

#include "cluster_fit.h"
#include "fp64.cuh"
#include "internal.h"
#include "levels.h"
#include "separable.h"
#include "separable_fused_shape.h"

namespace cg = cooperative_groups;

namespace sim {

namespace {

__device__ __forceinline__ int pad4(int n) { return sf_pad4(n); }

__device__ __forceinline__ void copy_async_16(void* dst, const void* src) {
    asm volatile("cp.async.cg.shared.global [%0], [%1], 16;" ::"r"((uint32_t)__cvta_generic_to_shared(dst)), "l"(src)
                 : "memory");
}

// f.put(f.column(k), r, Σ_j X[r][j] Q[j][k]) for r < rows, k < N.  X: [rows][ldx] in
// shared memory, zero from column N to ldx = pad4(N); Q: pad4(N) x pad4(N), zero
// beyond N, streamed through three stages of shared memory (read directly, its L2
// latency of about 370 clocks per two reduction steps was the time of a product).
// A thread forms RT rows x KT columns at a time.  Every thread of the CTA calls it.
template <int RT, int KT, class F>
__device__ __forceinline__ void rows_times_q(const float2* X, int ldx, int rows, int N, const float* __restrict__ Q,
                                             float* stage, const F& f) {
    constexpr int K4 = KT / 4;
    const int ldq = pad4(N), nk = (ldq + KT - 1) / KT, nr = (rows + RT - 1) / RT, items = nk * nr;
    const int KC = sf_stage_rows(ldq), nc = (ldq + KC - 1) / KC, per_stage = KC * ldq;
    auto fill = [&](int c) {
        if (c < nc) {
            float* dst = stage + (size_t)(c % SF_STAGES) * per_stage;
            const float* src = Q + (size_t)c * per_stage;
            const int units = min(KC, ldq - c * KC) * ldq / 4;
            for (int i = threadIdx.x; i < units; i += SF_T) copy_async_16(dst + 4 * i, src + 4 * i);
        }
        asm volatile("cp.async.commit_group;" ::: "memory");
    };
    for (int first = 0; first < items; first += SF_T) {
        const int item = min(first + (int)threadIdx.x, items - 1);
        const bool valid = first + (int)threadIdx.x < items;
        const bool busy = __any_sync(0xffffffffu, valid);
        const int k = item % nk * KT, r0 = item / nk * RT;
        const float4* x[RT];
#pragma unroll
        for (int r = 0; r < RT; ++r) x[r] = reinterpret_cast<const float4*>(X + (size_t)min(r0 + r, rows - 1) * ldx);
        int q[K4];
#pragma unroll
        for (int h = 0; h < K4; ++h) q[h] = min(k + 4 * h, ldq - 4);
        float2 acc[RT][KT];
#pragma unroll
        for (int r = 0; r < RT; ++r)
#pragma unroll
            for (int c = 0; c < KT; ++c) acc[r][c] = make_float2(0.f, 0.f);
        __syncthreads();  // the stages of the round before are free
#pragma unroll
        for (int c = 0; c < SF_STAGES - 1; ++c) fill(c);
        for (int c = 0; c < nc; ++c) {
            asm volatile("cp.async.wait_group %0;" ::"n"(SF_STAGES - 2) : "memory");
            __syncthreads();  // chunk c is there, and chunk c - 1 has been read
            fill(c + SF_STAGES - 1);
            if (!busy) continue;
            const float* Qs = stage + (size_t)(c % SF_STAGES) * per_stage;
            const int jn = min(KC, ldq - c * KC), jx = c * KC / 2;
#pragma unroll 4
            for (int j = 0; j < jn; j += 2) {
                float4 q0[K4], q1[K4];
#pragma unroll
                for (int h = 0; h < K4; ++h) {
                    q0[h] = *reinterpret_cast<const float4*>(Qs + (size_t)j * ldq + q[h]);
                    q1[h] = *reinterpret_cast<const float4*>(Qs + (size_t)(j + 1) * ldq + q[h]);
                }
#pragma unroll
                for (int r = 0; r < RT; ++r) {
                    const float4 v = x[r][jx + j / 2];
                    const float2 v0 = make_float2(v.x, v.y), v1 = make_float2(v.z, v.w);
#pragma unroll
                    for (int h = 0; h < K4; ++h) {
                        float2* a = acc[r] + 4 * h;
                        a[0] = __ffma2_rn(make_float2(q0[h].x, q0[h].x), v0, a[0]);
                        a[1] = __ffma2_rn(make_float2(q0[h].y, q0[h].y), v0, a[1]);
                        a[2] = __ffma2_rn(make_float2(q0[h].z, q0[h].z), v0, a[2]);
                        a[3] = __ffma2_rn(make_float2(q0[h].w, q0[h].w), v0, a[3]);
                        a[0] = __ffma2_rn(make_float2(q1[h].x, q1[h].x), v1, a[0]);
                        a[1] = __ffma2_rn(make_float2(q1[h].y, q1[h].y), v1, a[1]);
                        a[2] = __ffma2_rn(make_float2(q1[h].z, q1[h].z), v1, a[2]);
                        a[3] = __ffma2_rn(make_float2(q1[h].w, q1[h].w), v1, a[3]);
                    }
                }
            }
        }
        if (!valid) continue;
#pragma unroll
        for (int c = 0; c < KT; ++c) {
            if (k + c >= N) break;
            const auto col = f.column(k + c);
#pragma unroll
            for (int r = 0; r < RT; ++r)
                if (r0 + r < rows) f.put(col, r0 + r, acc[r][c]);
        }
    }
}

// values of line r to the CTA that holds line k of the other axis, at r + at
struct SendLines {
    cg::cluster_group& cl;
    float2* buf;
    int per, ld, at;  // lines per CTA and length of a line there
    __device__ __forceinline__ float2* column(int k) const {
        const int owner = k / per;
        return cl.map_shared_rank(buf, owner) + (k - owner * per) * ld + at;
    }
    __device__ __forceinline__ void put(float2* col, int r, float2 v) const { col[r] = v; }
};

// v / (Σ_d λ - σb): the denominator formed in FP64 and rounded once
struct Divide {
    float2* A;
    int ld;
    const double2* lsum;  // at this CTA's first line
    int N0;
    double2 sb;
    __device__ __forceinline__ int column(int k) const { return k; }
    __device__ __forceinline__ void put(int k, int c, float2 v) const {
        const float2 d = narrow(csub(__ldg(lsum + (int64_t)k * N0 + c), sb));
        const float inv = 1.0f / (d.x * d.x + d.y * d.y);
        A[c * ld + k] = make_float2((v.x * d.x + v.y * d.y) * inv, (v.y * d.x - v.x * d.y) * inv);
    }
};

struct Output {
    double2* out;  // at this CTA's first line
    const float2* sc;
    int N0;
    __device__ __forceinline__ int column(int k) const { return k; }
    __device__ __forceinline__ void put(int k, int r, float2 v) const {
        const int g = r * N0 + k;
        const float2 s = __ldg(sc + g);
        out[g] = widen(make_float2(v.x * s.x - v.y * s.y, v.x * s.y + v.y * s.x));
    }
};

// Rc lines along axis 0 and Cc along axis 1 per CTA (the last CTA may have fewer)
template <int RT, int KT>
__global__ void __launch_bounds__(SF_T) k_sep_fused(JobSpace js, int in_slot, int out_slot, const double2* sigma,
                                                    double2 b, int N0, int N1, const float* __restrict__ Q0,
                                                    const float* __restrict__ Q1, const float2* __restrict__ sin32,
                                                    const float2* __restrict__ sout32,
                                                    const double2* __restrict__ lsum, int Rc, int Cc) {
    cg::cluster_group cl = cg::this_cluster();
    const int C = (int)cl.num_blocks(), q = (int)cl.block_rank();
    const int job = js.d_active[blockIdx.x / C];
    const int ld0 = pad4(N0), ld1 = pad4(N1), tid = threadIdx.x;
    const int size = max(Rc * ld0, Cc * ld1);
    extern __shared__ __align__(16) float2 sf_raw[];
    float2 *A = sf_raw, *Bf = sf_raw + size;  // both hold [Rc][ld0] or [Cc][ld1]
    float* stage = reinterpret_cast<float*>(Bf + size);
    const int row0 = q * Rc, rows = max(0, min(Rc, N1 - row0));
    const int col0 = q * Cc, cols = max(0, min(Cc, N0 - col0));
    // every CTA of the cluster is running before it is written to, its buffers cleared
    // (the padding of the lines has to be zero)
    for (int i = tid; i < 2 * size; i += SF_T) sf_raw[i] = make_float2(0.f, 0.f);
    cl.sync();
    const double2* in = js.vec + (size_t)job * js.vstride + (size_t)in_slot * js.n;
    double2* out = js.vec + (size_t)job * js.vstride + (size_t)out_slot * js.n;
    const int64_t g0 = (int64_t)row0 * N0;
    // four loads in flight before the first conversion
    for (int i0 = tid; i0 < rows * N0; i0 += 4 * SF_T) {
        double2 x[4];
        float2 sc[4];
#pragma unroll
        for (int u = 0; u < 4; ++u) {
            const int i = i0 + u * SF_T;
            x[u] = i < rows * N0 ? in[g0 + i] : make_double2(0.0, 0.0);
            sc[u] = i < rows * N0 ? sin32[g0 + i] : make_float2(0.f, 0.f);
        }
#pragma unroll
        for (int u = 0; u < 4; ++u) {
            const int i = i0 + u * SF_T;
            const float2 v = narrow(x[u]);
            if (i < rows * N0)
                A[i / N0 * ld0 + i % N0] = make_float2(v.x * sc[u].x - v.y * sc[u].y, v.x * sc[u].y + v.y * sc[u].x);
        }
    }
    __syncthreads();
    if (rows > 0) rows_times_q<RT, KT>(A, ld0, rows, N0, Q0, stage, SendLines{cl, Bf, Cc, ld1, row0});
    cl.sync();
    // axis 1, the division, axis 1; A is free and becomes [Cc][ld1]
    if (ld0 != ld1 || Rc != Cc) {
        for (int i = tid; i < size; i += SF_T) A[i] = make_float2(0.f, 0.f);
        __syncthreads();
    } else {
        for (int i = tid; i < cols * (ld1 - N1); i += SF_T) A[i / (ld1 - N1) * ld1 + N1 + i % (ld1 - N1)] = make_float2(0.f, 0.f);
        __syncthreads();
    }
    const double2 sb = cmul(sigma[js.d_jobshift[job]], b);
    if (cols > 0) rows_times_q<RT, KT>(Bf, ld1, cols, N1, Q1, stage, Divide{A, ld1, lsum + col0, N0, sb});
    cl.sync();  // every CTA has read its lines in Bf
    if (rows > 0)  // the padding of the lines that come back
        for (int i = tid; i < Rc * (ld0 - N0); i += SF_T) Bf[i / (ld0 - N0) * ld0 + N0 + i % (ld0 - N0)] = make_float2(0.f, 0.f);
    if (cols > 0) rows_times_q<RT, KT>(A, ld1, cols, N1, Q1, stage, SendLines{cl, Bf, Rc, ld0, col0});
    cl.sync();
    if (rows > 0) rows_times_q<RT, KT>(Bf, ld0, rows, N0, Q0, stage, Output{out + g0, sout32 + g0, N0});
}

__global__ void k_sep_pad(const float* Q32, int N, int Np, float* Qp) {
    const int64_t t = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
    if (t >= (int64_t)Np * Np) return;
    const int r = (int)(t / Np), c = (int)(t % Np);
    Qp[t] = r < N && c < N ? Q32[(size_t)r * N + c] : 0.f;
}

// The same for the separate kernels: a product's CTAs (128 rows of real and
// imaginary parts each, two to an SM) take 6,000 clocks and 35 per output column for
// each 32 reduction indices, the elementwise passes 8,000 and their traffic, a
// launch 2,000.  Many jobs of a few hundred points a side fill the tensor cores and
// stay there (64 pencils of 219 points: 0.3 ms against 0.5).
double separate_cost(int N0, int N1, int na) {
    const double n = (double)N0 * N1;
    auto product = [&](int N, int rows) {
        const int NT = std::min(256, (N + 15) / 16 * 16);
        const double ctas = std::ceil(2.0 * rows / 128.0) * std::ceil((double)N / NT) * na;
        return std::ceil(ctas / (2.0 * sm_count())) * std::ceil(N / 32.0) * (6000.0 + 35.0 * NT);
    };
    return 2.0 * product(N0, N1) + 2.0 * product(N1, N0) + 3.0 * (8000.0 + n * na * 48.0 / 3300.0) + 7.0 * 2000.0;
}

template <int RT, int KT>
void launch_fused(const Separable& S, const JobSpace& js, int na, int in_slot, int out_slot, const double2* d_sigma,
                  const FusedShape& f, cudaStream_t st) {
    auto kern = k_sep_fused<RT, KT>;
    cudaLaunchConfig_t cfg = {};
    cfg.gridDim = dim3(na * f.C);
    cfg.blockDim = dim3(SF_T);
    cfg.dynamicSmemBytes = f.smem;
    cfg.stream = st;
    cudaLaunchAttribute attr[1];
    attr[0].id = cudaLaunchAttributeClusterDimension;
    attr[0].val.clusterDim.x = f.C;
    attr[0].val.clusterDim.y = 1;
    attr[0].val.clusterDim.z = 1;
    cfg.attrs = attr;
    cfg.numAttrs = 1;
    SIM_CUDA(cudaLaunchKernelEx(&cfg, kern, js, in_slot, out_slot, d_sigma, S.b, (int)S.dims[0], (int)S.dims[1],
                                (const float*)S.Qp[0], (const float*)S.Qp[1], (const float2*)S.sin32,
                                (const float2*)S.sout32, (const double2*)S.lsum, f.Rc, f.Cc));
    SIM_LAUNCH_CHECK();
}

FusedShape shape_on_device(const Separable& S, int na) {
    return fused_shape_that_fits((int)S.dims[0], (int)S.dims[1], na, sm_count(), [](const FusedShape& f) {
        const void* kern = f.tile == 0 ? (const void*)k_sep_fused<1, 4>
                                       : (f.tile == 1 ? (const void*)k_sep_fused<2, 4> : (const void*)k_sep_fused<4, 4>);
        return clusters_that_fit(kern, f.C, SF_T, f.smem) > 0;
    });
}

}  // namespace

void sep_pad_table(const float* Q32, int N, float* Qp, cudaStream_t st) {
    const int Np = sf_pad4(N);
    k_sep_pad<<<cdiv_up((int64_t)Np * Np, 256), 256, 0, st>>>(Q32, N, Np, Qp);
    SIM_LAUNCH_CHECK();
}

bool sep_fused_applies(const Separable& S, int precision) {
    return precision != SIM_FP64 && S.tc && S.ndim == 2 && S.dims[0] <= 2048 && S.dims[1] <= 2048 &&
           shape_on_device(S, 1).C > 0;
}

bool sep_fused_2d(const Separable& S, const JobSpace& js, int na, int in_slot, int out_slot, const double2* d_sigma,
                  cudaStream_t st) {
    const FusedShape f = shape_on_device(S, na);
    if (f.C == 0 || f.cost > separate_cost((int)S.dims[0], (int)S.dims[1], na)) return false;
    kprof_begin("sep_fused", st);  // instrumentation: a part of "separable"
    switch (f.tile) {
        case 0: launch_fused<1, 4>(S, js, na, in_slot, out_slot, d_sigma, f, st); break;
        case 1: launch_fused<2, 4>(S, js, na, in_slot, out_slot, d_sigma, f, st); break;
        default: launch_fused<4, 4>(S, js, na, in_slot, out_slot, d_sigma, f, st); break;
    }
    kprof_end("sep_fused", st, na * 32.0 * (double)js.n,
              na * 8.0 * (double)js.n * (double)(S.dims[0] + S.dims[1]));
    return true;
}

}  // namespace sim
