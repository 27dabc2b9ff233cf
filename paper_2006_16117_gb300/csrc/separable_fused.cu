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
// cores: a thread forms RT rows x 4 outputs, a complex value times a real one in
// one paired FMA; the rows come from shared memory as broadcasts, Q through L1
// (coalesced, four rows ahead in registers).  FP32 products need no splitting as
// on the tensor cores, and every value is summed in FP32 over its line in order.
#include <cooperative_groups.h>

#include <algorithm>
#include <atomic>
#include <cmath>

#include "internal.h"
#include "levels.h"
#include "separable.h"

namespace cg = cooperative_groups;

namespace sim {

namespace {

constexpr int SF_T = 256;

__host__ __device__ constexpr int pad4(int n) { return (n + 3) / 4 * 4; }

// store(r, k, Σ_j X[r][j] Q[j][k]) for r < rows, k < N.  X: [rows][ldx] in shared
// memory, zero from column N to ldx = pad4(N); Q: pad4(N) x pad4(N), zero beyond N.
template <int RT, class F>
__device__ __forceinline__ void rows_times_q(const float2* X, int ldx, int rows, int N, const float* __restrict__ Q,
                                             F store) {
    const int ldq = pad4(N), nk = ldq / 4, nr = (rows + RT - 1) / RT;
    for (int item = threadIdx.x; item < nk * nr; item += SF_T) {
        const int k = item % nk * 4, r0 = item / nk * RT;
        const float4* x[RT];
#pragma unroll
        for (int r = 0; r < RT; ++r) x[r] = reinterpret_cast<const float4*>(X + (size_t)min(r0 + r, rows - 1) * ldx);
        const float* q = Q + k;
        float2 acc[RT][4];
#pragma unroll
        for (int r = 0; r < RT; ++r)
#pragma unroll
            for (int c = 0; c < 4; ++c) acc[r][c] = make_float2(0.f, 0.f);
        float4 qn[4];
#pragma unroll
        for (int j = 0; j < 4; ++j) qn[j] = __ldg(reinterpret_cast<const float4*>(q + (size_t)j * ldq));
        for (int j0 = 0; j0 < ldq; j0 += 4) {
            float4 qc[4];
#pragma unroll
            for (int j = 0; j < 4; ++j) qc[j] = qn[j];
            if (j0 + 4 < ldq) {
#pragma unroll
                for (int j = 0; j < 4; ++j)
                    qn[j] = __ldg(reinterpret_cast<const float4*>(q + (size_t)(j0 + 4 + j) * ldq));
            }
#pragma unroll
            for (int h = 0; h < 2; ++h) {
                const float4 q0 = qc[2 * h], q1 = qc[2 * h + 1];
#pragma unroll
                for (int r = 0; r < RT; ++r) {
                    const float4 v = x[r][j0 / 2 + h];
                    const float2 v0 = make_float2(v.x, v.y), v1 = make_float2(v.z, v.w);
                    acc[r][0] = __ffma2_rn(make_float2(q0.x, q0.x), v0, acc[r][0]);
                    acc[r][1] = __ffma2_rn(make_float2(q0.y, q0.y), v0, acc[r][1]);
                    acc[r][2] = __ffma2_rn(make_float2(q0.z, q0.z), v0, acc[r][2]);
                    acc[r][3] = __ffma2_rn(make_float2(q0.w, q0.w), v0, acc[r][3]);
                    acc[r][0] = __ffma2_rn(make_float2(q1.x, q1.x), v1, acc[r][0]);
                    acc[r][1] = __ffma2_rn(make_float2(q1.y, q1.y), v1, acc[r][1]);
                    acc[r][2] = __ffma2_rn(make_float2(q1.z, q1.z), v1, acc[r][2]);
                    acc[r][3] = __ffma2_rn(make_float2(q1.w, q1.w), v1, acc[r][3]);
                }
            }
        }
#pragma unroll
        for (int r = 0; r < RT; ++r)
#pragma unroll
            for (int c = 0; c < 4; ++c)
                if (r0 + r < rows && k + c < N) store(r0 + r, k + c, acc[r][c]);
    }
}

// Rc lines along axis 0 and Cc along axis 1 per CTA (the last CTA may have fewer)
template <int RT>
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
    const int row0 = q * Rc, rows = max(0, min(Rc, N1 - row0));
    const int col0 = q * Cc, cols = max(0, min(Cc, N0 - col0));
    // every CTA of the cluster is running before it is written to, its buffers cleared
    // (the padding of the lines has to be zero)
    for (int i = tid; i < 2 * size; i += SF_T) sf_raw[i] = make_float2(0.f, 0.f);
    cl.sync();
    const double2* in = js.vec + (size_t)job * js.vstride + (size_t)in_slot * js.n;
    double2* out = js.vec + (size_t)job * js.vstride + (size_t)out_slot * js.n;
    const int64_t g0 = (int64_t)row0 * N0;
#pragma unroll 4
    for (int i = tid; i < rows * N0; i += SF_T) {
        const float2 x = from_c128<float2>(in[g0 + i]), s = sin32[g0 + i];
        A[i / N0 * ld0 + i % N0] = make_float2(x.x * s.x - x.y * s.y, x.x * s.y + x.y * s.x);
    }
    __syncthreads();
    if (rows > 0)
        rows_times_q<RT>(A, ld0, rows, N0, Q0, [&](int r, int k, float2 v) {
            cl.map_shared_rank(Bf, k / Cc)[k % Cc * ld1 + row0 + r] = v;
        });
    cl.sync();
    // axis 1, the division, axis 1; A is free and becomes [Cc][ld1]
    if (ld0 != ld1 || Rc != Cc) {
        for (int i = tid; i < size; i += SF_T) A[i] = make_float2(0.f, 0.f);
        __syncthreads();
    } else {
        for (int i = tid; i < cols * (ld1 - N1); i += SF_T) A[i / (ld1 - N1) * ld1 + N1 + i % (ld1 - N1)] = make_float2(0.f, 0.f);
        __syncthreads();
    }
    const double2 s = sigma[js.d_jobshift[job]];
    const double2 sb = cmul(s, b);
    if (cols > 0)
        rows_times_q<RT>(Bf, ld1, cols, N1, Q1, [&](int c, int k, float2 v) {
            const float2 d = from_c128<float2>(csub(lsum[(int64_t)k * N0 + col0 + c], sb));
            const float inv = 1.0f / (d.x * d.x + d.y * d.y);
            A[c * ld1 + k] = make_float2((v.x * d.x + v.y * d.y) * inv, (v.y * d.x - v.x * d.y) * inv);
        });
    cl.sync();  // every CTA has read its lines in Bf
    if (rows > 0)  // the padding of the lines that come back
        for (int i = tid; i < Rc * (ld0 - N0); i += SF_T) Bf[i / (ld0 - N0) * ld0 + N0 + i % (ld0 - N0)] = make_float2(0.f, 0.f);
    if (cols > 0)
        rows_times_q<RT>(A, ld1, cols, N1, Q1, [&](int c, int k, float2 v) {
            cl.map_shared_rank(Bf, k / Rc)[k % Rc * ld0 + col0 + c] = v;
        });
    cl.sync();
    if (rows > 0)
        rows_times_q<RT>(Bf, ld0, rows, N0, Q0, [&](int r, int k, float2 v) {
            const int64_t g = g0 + (int64_t)r * N0 + k;
            const float2 sc = sout32[g];
            out[g] = to_c128(make_float2(v.x * sc.x - v.y * sc.y, v.x * sc.y + v.y * sc.x));
        });
}

__global__ void k_sep_pad(const float* Q32, int N, int Np, float* Qp) {
    const int64_t t = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
    if (t >= (int64_t)Np * Np) return;
    const int r = (int)(t / Np), c = (int)(t % Np);
    Qp[t] = r < N && c < N ? Q32[(size_t)r * N + c] : 0.f;
}

struct FusedShape {
    int C = 0, Rc = 0, Cc = 0, RT = 4;
    size_t smem = 0;
    double cost = 1e300;
};

// Cluster size by an estimate of the clocks of an apply: the products at half the
// FP32 rate over the threads that have work, and 2,000 clocks a cluster barrier.
FusedShape fused_shape(int N0, int N1, int na) {
    FusedShape best;
    for (int C = 1; C <= 16; ++C) {
        FusedShape f;
        f.Rc = (N1 + C - 1) / C;
        f.Cc = (N0 + C - 1) / C;
        if (C > 1 && ((C - 1) * f.Rc >= N1 || (C - 1) * f.Cc >= N0)) continue;  // a CTA without lines
        f.C = C;
        f.smem = 2 * sizeof(float2) * (size_t)std::max(f.Rc * pad4(N0), f.Cc * pad4(N1));
        if (f.smem > 220 * 1024) continue;
        for (int RT : {4, 8}) {
            auto product = [&](int rows, int N) {
                const double items = (double)(pad4(N) / 4) * ((rows + RT - 1) / RT);
                // an item: RT x 4 x N paired FMAs; 256 threads, 64 paired FMAs a clock
                return std::ceil(items / SF_T) * SF_T * RT * 4.0 * N / 64.0 / (RT == 8 ? 0.6 : 0.45);
            };
            const int per_sm = f.smem <= 110 * 1024 ? 2 : 1;
            const double waves = std::ceil((double)na * C / (152.0 * per_sm)) * (na * C > 152 ? 2.0 / per_sm * per_sm : 1.0);
            const double cost = waves * (2.0 * product(f.Rc, N0) + 2.0 * product(f.Cc, N1)) + (C > 1 ? 9000.0 : 4000.0);
            if (cost < best.cost) {
                best = f;
                best.RT = RT;
                best.cost = cost;
            }
        }
    }
    return best;
}

template <int RT>
void launch_fused(const Separable& S, const JobSpace& js, int na, int in_slot, int out_slot, const double2* d_sigma,
                  const FusedShape& f, cudaStream_t st) {
    static std::atomic<uint64_t> ready{0};  // devices whose kernel attributes are set
    int dev = 0;
    SIM_CUDA(cudaGetDevice(&dev));
    if (dev > 63 || !(ready.load() >> dev & 1)) {
        SIM_CUDA(cudaFuncSetAttribute(k_sep_fused<RT>, cudaFuncAttributeMaxDynamicSharedMemorySize, 220 * 1024));
        SIM_CUDA(cudaFuncSetAttribute(k_sep_fused<RT>, cudaFuncAttributeNonPortableClusterSizeAllowed, 1));
        if (dev <= 63) ready.fetch_or(1ull << dev);
    }
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
    SIM_CUDA(cudaLaunchKernelEx(&cfg, k_sep_fused<RT>, js, in_slot, out_slot, d_sigma, S.b, (int)S.dims[0],
                                (int)S.dims[1], (const float*)S.Qp[0], (const float*)S.Qp[1],
                                (const float2*)S.sin32, (const float2*)S.sout32, (const double2*)S.lsum, f.Rc, f.Cc));
    SIM_LAUNCH_CHECK();
}

}  // namespace

void sep_pad_table(const float* Q32, int N, float* Qp, cudaStream_t st) {
    const int Np = pad4(N);
    k_sep_pad<<<cdiv_up((int64_t)Np * Np, 256), 256, 0, st>>>(Q32, N, Np, Qp);
    SIM_LAUNCH_CHECK();
}

bool sep_fused_2d(const Separable& S, const JobSpace& js, int na, int in_slot, int out_slot, const double2* d_sigma,
                  cudaStream_t st) {
    if (S.ndim != 2 || S.dims[0] > 2048 || S.dims[1] > 2048) return false;
    const FusedShape f = fused_shape((int)S.dims[0], (int)S.dims[1], na);
    if (f.C == 0) return false;
    if (f.RT == 8) launch_fused<8>(S, js, na, in_slot, out_slot, d_sigma, f, st);
    else launch_fused<4>(S, js, na, in_slot, out_slot, d_sigma, f, st);
    return true;
}

}  // namespace sim
