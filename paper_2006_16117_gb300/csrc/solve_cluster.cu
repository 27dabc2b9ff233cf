// Block solve x = (A - σB)^{-1} r on thread-block clusters.
//
// The factors of one shift are the dense T×T blocks Dinv_k of every block row
// and E_k of every block row but the middle one, mid (krylov.cu): the
// elimination runs from both ends to the middle.  With L_k the couplings of
// block k to its outer neighbour (mid: to both neighbours) a solve is
//   forward   t_k = Dinv_k (r_k - L_k t_outer)        from the ends to mid,
//             x_mid = Dinv_mid (r_mid - L_mid [t_{mid-1}; t_{mid+1}]),
//   backward  x_k = t_k - E_k x_inner                 from mid to the ends:
// two chains of about nb dependent GEMVs that run side by side, a cluster each,
// instead of one of 2nb-1.  Launch 0 runs the forward halves; launch 1 the
// backward ones, each cluster computing x_mid for itself first (t_{mid±1} come
// from a copy in the job's VS_W slot, as side 0 may already have overwritten
// its own), so that no cluster waits for another.  One right-hand side, T = 200,
// nb = 200, complex64: 696 us as one chain, 378 as two.
//
// Only the vectors depend on the previous step, the matrices do not.  So
// each CTA of a cluster owns a slice of rows of every block, and two producer
// warps stream the slices, in chain order, through a ring of shared-memory
// stages (one 1-D bulk copy per row into a padded row, completing on the
// stage's "full" mbarrier) as far ahead as the ring allows; the consumers
// release a stage on its "empty" mbarrier.  Per step each of the eight consumer
// warps forms the right-hand side in its own columns, then for each chunk of rows
// runs the GEMV over them with one row per lane (or a row per group of lanes); the
// warps' partial sums are added through shared memory and the new rows of the
// vector sent into every CTA's shared memory with st.async, which completes on the
// receiver's per-step mbarrier.  Up to R right-hand sides of the same shift
// share each pass over the matrices (the k random vectors of the
// multiplicity step).
//
// What bounds a chain step is the number of instructions a warp runs through once:
// with two or three warps a scheduler and straight-line code that fits no
// instruction buffer each costs about five clocks.  Hence a kernel per phase and
// per "one chunk a step" (ONE), the inputs brought by the producers, one barrier a
// step, the vector stored to memory a step later by warps that wait anyway, and row
// layouts that are powers of two.  Launch 1 starts under launch 0 and fills its first
// stage (5 us a solve).  Two sides, T = 200 complex64: 378 -> 263 us (a step 3,800 -> 2,900
// clocks forward, 3,100 -> 2,300 backward); T = 102 197 -> 123; eight right-hand sides at
// T = 102 196 -> 138 us a launch; complex128 T = 30 106 -> 53, T = 98 335 -> 195.  With 56 shifts at T = 200 the matrices bound it:
// 1,446 -> 1,159 us (5.0 TB/s) in complex64, 12.4 -> 10.2 ms in complex128 (FP64 pipe).
//
// Every wait on an mbarrier has an iteration limit; a thread whose wait runs
// out records an error, which the inner solver throws when it has waited for the
// stream (block_solve_check), and the CTA stops computing and issuing copies, keeps
// taking part in its barriers (so no thread waits forever), and waits (again
// bounded) for its own copies in flight before it exits.
#include <cooperative_groups.h>

#include <algorithm>
#include <cstdio>
#include <map>
#include <type_traits>
#include <vector>

#include "internal.h"
#include "solve_cluster.h"

namespace cg = cooperative_groups;

namespace sim {

namespace {

__device__ __forceinline__ uint32_t smem_u32(const void* p) { return (uint32_t)__cvta_generic_to_shared(p); }

__device__ __forceinline__ void mbar_init(uint64_t* bar, uint32_t count) {
    asm volatile("mbarrier.init.shared::cta.b64 [%0], %1;" ::"r"(smem_u32(bar)), "r"(count) : "memory");
}

__device__ __forceinline__ void mbar_expect_tx(uint64_t* bar, uint32_t bytes) {
    asm volatile("mbarrier.arrive.expect_tx.shared::cta.b64 _, [%0], %1;" ::"r"(smem_u32(bar)), "r"(bytes)
                 : "memory");
}

__device__ __forceinline__ bool mbar_try_wait(uint64_t* bar, uint32_t parity) {
    uint32_t ok;
    asm volatile(
        "{\n"
        " .reg .pred p;\n"
        " mbarrier.try_wait.parity.shared::cta.b64 p, [%1], %2;\n"
        " selp.u32 %0, 1, 0, p;\n"
        "}\n"
        : "=r"(ok)
        : "r"(smem_u32(bar)), "r"(parity)
        : "memory");
    return ok != 0;
}

__device__ __forceinline__ void tma_load_1d(void* dst, const void* src, uint32_t bytes, uint64_t* bar) {
    asm volatile(
        "cp.async.bulk.shared::cluster.global.mbarrier::complete_tx::bytes [%0], [%1], %2, [%3];" ::"r"(
            smem_u32(dst)),
        "l"(src), "r"(bytes), "r"(smem_u32(bar))
        : "memory");
}

// wait with cluster-scope acquire: the data arrived through st.async from other CTAs
__device__ __forceinline__ bool mbar_try_wait_cluster(uint64_t* bar, uint32_t parity) {
    uint32_t ok;
    asm volatile(
        "{\n"
        " .reg .pred p;\n"
        " mbarrier.try_wait.parity.acquire.cluster.shared::cta.b64 p, [%1], %2;\n"
        " selp.u32 %0, 1, 0, p;\n"
        "}\n"
        : "=r"(ok)
        : "r"(smem_u32(bar)), "r"(parity)
        : "memory");
    return ok != 0;
}

__device__ __forceinline__ uint32_t mapa_u32(const void* local, uint32_t rank) {
    uint32_t r;
    asm volatile("mapa.shared::cluster.u32 %0, %1, %2;" : "=r"(r) : "r"(smem_u32(local)), "r"(rank));
    return r;
}

// store one complex value into another CTA's shared memory; the bytes count
// against that CTA's mbarrier (addresses from mapa_u32)
__device__ __forceinline__ void st_async_c(uint32_t raddr, float2 v, uint32_t rbar) {
    asm volatile("st.async.shared::cluster.mbarrier::complete_tx::bytes.v2.f32 [%0], {%1, %2}, [%3];" ::"r"(raddr),
                 "f"(v.x), "f"(v.y), "r"(rbar)
                 : "memory");
}
__device__ __forceinline__ void st_async_c(uint32_t raddr, double2 v, uint32_t rbar) {
    asm volatile("st.async.shared::cluster.mbarrier::complete_tx::bytes.v2.f64 [%0], {%1, %2}, [%3];" ::"r"(raddr),
                 "d"(v.x), "d"(v.y), "r"(rbar)
                 : "memory");
}

constexpr long long WAIT_LIMIT = 1ll << 26;  // try_wait polls before a wait is declared failed

template <class C> __device__ __forceinline__ C zero_c();
template <> __device__ __forceinline__ double2 zero_c<double2>() { return make_double2(0.0, 0.0); }
template <> __device__ __forceinline__ float2 zero_c<float2>() { return make_float2(0.f, 0.f); }


}  // namespace

// 16 bytes of complex values: two complex64 or one complex128
template <class C> struct Vec16;
template <> struct Vec16<float2> {
    using T = float4;
    static constexpr int N = 2;
    __device__ static __forceinline__ float2 get(const float4& v, int e) {
        return e == 0 ? make_float2(v.x, v.y) : make_float2(v.z, v.w);
    }
};
template <> struct Vec16<double2> {
    using T = double2;
    static constexpr int N = 1;
    __device__ static __forceinline__ double2 get(const double2& v, int) { return v; }
};

constexpr int PF_T = 256;                         // largest T whose step inputs are fetched ahead
constexpr int RW = 9;                             // a row's partial sums, padded off the banks
constexpr int NE = 2;                             // couplings of a row fetched ahead
constexpr int CL_WARPS = 8;                       // consumer warps: the GEMVs and the vector work
constexpr int PROD = 64;                         // threads that issue the copies (two warps)
constexpr int CL_THREADS = CL_WARPS * 32 + PROD;

// barrier of the consumer warps only (the producer warps never join it)
__device__ __forceinline__ void consumer_sync() {
    static_assert(CL_WARPS * 32 == 256, "named barrier thread count");
    asm volatile("bar.sync 1, 256;" ::: "memory");
}

__device__ __forceinline__ void mbar_arrive(uint64_t* bar) {
    asm volatile("mbarrier.arrive.shared::cta.b64 _, [%0];" ::"r"(smem_u32(bar)) : "memory");
}

// BYTES of src to shared memory, or zeros
template <int BYTES> __device__ __forceinline__ void copy_async(void* dst, const void* src, bool there = true) {
    const uint32_t n = there ? BYTES : 0;
    if constexpr (BYTES == 16)
        asm volatile("cp.async.cg.shared.global [%0], [%1], 16, %2;" ::"r"(smem_u32(dst)), "l"(src), "r"(n) : "memory");
    else
        asm volatile("cp.async.ca.shared.global [%0], [%1], %2, %3;" ::"r"(smem_u32(dst)), "l"(src), "n"(BYTES), "r"(n)
                     : "memory");
}
// an arrival on the barrier once this thread's copies so far are done
__device__ __forceinline__ void arrive_after_copies(uint64_t* bar) {
    asm volatile("cp.async.mbarrier.arrive.noinc.shared.b64 [%0];" ::"r"(smem_u32(bar)) : "memory");
}
__device__ __forceinline__ void copies_done() { asm volatile("cp.async.wait_all;" ::: "memory"); }

__device__ __forceinline__ bool failed_flag(const int* f) { return *(const volatile int*)f != 0; }

// The launch's groups: R jobs each, -1 past a group's last.  As a parameter up to
// MAX jobs (a copy between the kernels of a stream costs about 5 us of its time), in
// device memory (`far`) beyond.
struct Groups {
    static constexpr int MAX = 512;
    const int* far;
    short near[MAX];
    __device__ __forceinline__ int job(int i) const { return far ? far[i] : near[i]; }
};

// MINB: CTAs per SM the launch is built for (2 caps the registers at 112 so
// that two CTAs of at most ~112 KB of shared memory share an SM)
template <class C, int R, int MINB, bool ONE, int phase>
__global__ void __launch_bounds__(CL_THREADS, MINB) k_block_solve_cl(Pencil P, JobSpace js, int in_slot,
                                                                  int out_slot, void* const* fptrs,
                                                                  const __grid_constant__ Groups groups, int SR, int NS, int TP, int pf_ok,
                                                                  int* err) {
    cg::cluster_group cl = cg::this_cluster();
    const int Ccl = (int)cl.num_blocks();
    const int q = (int)cl.block_rank();
    const int T = P.T, nb = P.nb, mid = P.mid;
    const int sides = mid + 1 < nb ? 2 : 1;
    const int side = (int)(blockIdx.x / Ccl) % sides, grp = (int)(blockIdx.x / Ccl) / sides;
    const int half = side ? nb - 1 - mid : mid;  // this side's blocks
    // steps: phase 0 the forward half; phase 1 x_mid, then the backward half
    const int nsteps = phase ? half + 1 : half;
    auto block_of = [&](int b) {
        return phase ? (side ? mid + b : mid - b) : (side ? nb - 1 - b : b);
    };
    const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
    using VT = typename Vec16<C>::T;
    constexpr int VN = Vec16<C>::N;
    using Rt = decltype(zero_c<C>().x);

    // the group's job vectors (in shared memory: indexed by runtime job numbers)
    __shared__ const double2* s_in[R];
    __shared__ double2* s_out[R];
    __shared__ int s_fail;
    int nr = 1;
#pragma unroll
    for (int j = 1; j < R; ++j)
        if (groups.job(grp * R + j) >= 0) nr = j + 1;
    const int job0 = groups.job(grp * R);
    if (tid < R) {
        const int jb = groups.job(grp * R + tid);
        const int jj = jb >= 0 ? jb : job0;
        s_in[tid] = js.vec + (size_t)jj * js.vstride + (size_t)in_slot * js.n;
        s_out[tid] = js.vec + (size_t)jj * js.vstride + (size_t)out_slot * js.n;
    }
    const int s = js.d_jobshift[job0];
    const C* Dinv = reinterpret_cast<const C*>(fptrs[s]);
    const C* E = Dinv + (size_t)nb * T * T;
    const C* Lval = Dinv + factor_lval_offset(P);

    const int Tc = (T + Ccl - 1) / Ccl;
    const int r0 = min(T, q * Tc), r1 = min(T, r0 + Tc);
    const int myrows = r1 - r0;
    const int Cact = (T + Tc - 1) / Tc;  // CTAs that have rows: the others take no part

    extern __shared__ __align__(128) unsigned char raw[];
    C* stage = reinterpret_cast<C*>(raw);                  // [NS][SR][TP]: rows padded to TP
    C* vbuf = stage + (size_t)NS * SR * TP;                // [3][R][T]: the chain's vectors
    C* sbuf = vbuf + (size_t)3 * R * T;                    // [R][T]: r_k - L_k t_outer
    C* red = sbuf + (size_t)R * T;                         // [2][R][SR][RW]: per-warp partial sums
    double2* tpf = reinterpret_cast<double2*>(red + (size_t)2 * RW * R * SR);
    // (tpf [3][R][SR]: t_k of this and the next two steps' rows)
    // fetched ahead if pf_ok: r_k [2][R][T], the first couplings' values and columns
    // [2][NE][T], the bounds of the rows' couplings [4][2][T]
    double2* rpf = tpf + (size_t)3 * R * SR;
    C* apf = reinterpret_cast<C*>(rpf + (pf_ok ? (size_t)2 * R * T : 0));
    int* cpf = reinterpret_cast<int*>(apf + (pf_ok ? (size_t)2 * NE * T : 0));
    int* bpf = cpf + (pf_ok ? (size_t)2 * NE * T : 0);
    uint64_t* full = reinterpret_cast<uint64_t*>(bpf + (pf_ok ? (size_t)8 * T : 0));     // [NS] stage filled
    uint64_t* empty = full + NS;                                                         // [NS] stage consumed
    uint64_t* vbar = empty + NS;                                                         // [3] vector received

    if (tid == 0) {
        s_fail = 0;
        for (int i = 0; i < NS; ++i) {
            mbar_init(&full[i], 1 + PROD);  // the bulk copies' expected bytes, and the producers
            mbar_init(&empty[i], 1);
        }
        for (int i = 0; i < 3; ++i) mbar_init(&vbar[i], 1);
        asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
    }
    __syncthreads();
    const uint32_t vec_bytes = (uint32_t)((size_t)T * nr * sizeof(C));  // one step's vector, all rows
    if (tid == 0)
        for (int i = 0; i < 3 && i <= nsteps - 2; ++i) mbar_expect_tx(&vbar[i], vec_bytes);  // steps 0, 1, 2
    cl.sync();  // every CTA of the cluster is running, barriers initialised and armed, before any remote store
    // Launch 1 starts while launch 0 runs (where SMs are free) and fills its first stage; it
    // waits for launch 0's end before it reads or writes a vector.  The factors are older
    // than launch 0, which starts after everything before it has ended.
    if (phase == 0) asm volatile("griddepcontrol.launch_dependents;" ::: "memory");
    auto vectors_ready = [&] {
        if (phase == 1) asm volatile("griddepcontrol.wait;" ::: "memory");
    };

    // A wait that gives up once the CTA has failed, or after WAIT_LIMIT polls.
    auto bounded = [&](auto&& done, int code) {
        if (__builtin_expect(done(), 1)) return true;
        for (long long it = 0; !failed_flag(&s_fail); ++it) {
            if (done()) return true;
            if (it > WAIT_LIMIT) {
                s_fail = 1;
                atomicExch(err, code);  // pinned host memory
            }
        }
        return false;
    };

    if (myrows == 0) {
    } else if (warp >= CL_WARPS) {
        // ---- producers: chunk c = up to SR rows of one block, one 1-D bulk copy
        // per row into its padded row of stage c % NS, once that stage is consumed.
        //
        // With the chunks come, through asynchronous copies by their lanes that count
        // on the same "full" barriers, the inputs of the right-hand sides (a load to a
        // consumer's register would be waited for wherever the compiler moves that
        // register): forward, of every column, r_k and the first NE couplings of the
        // row, whose bounds came a step earlier; backward (ONE) t_k of this CTA's rows.
        // They share two buffers, so with one chunk a step they come one chunk after
        // their own: the stage of chunk c is free when chunk c - 3 is consumed, the
        // inputs' buffer of chunk c - 1 as well.
        constexpr int LAG = ONE ? 1 : 0;
        const int pt = tid - CL_WARPS * 32;
        auto fetch_bounds = [&](int bb) {
            if (phase != 0 || !pf_ok || bb >= nsteps) return;
            const int64_t g = (int64_t)block_of(bb) * T;
            int* d = bpf + (bb & 3) * 2 * T;
            for (int i = pt; i < T; i += PROD) {
                const bool in = g + i < P.n;
                const int* src = P.Lptr + (in ? g + i : 0);
                copy_async<4>(d + i, src, in);
                copy_async<4>(d + T + i, src + 1, in);
            }
        };
        auto fetch_inputs = [&](int bb) {
            if (bb < 0) return;
            const int64_t g = (int64_t)block_of(bb) * T;
            if (phase == 0 && pf_ok) {
                const int* d = bpf + (bb & 3) * 2 * T;
                const int at = (bb & 1) * NE * T;
                double2* rd = rpf + (bb & 1) * R * T;
                for (int i = pt; i < T; i += PROD) {
                    const int lo = d[i], cnt = d[T + i] - lo;
#pragma unroll
                    for (int e = 0; e < NE; ++e)
                        if (e < cnt) {
                            copy_async<4>(cpf + at + e * T + i, P.Lcol + lo + e);
                            copy_async<sizeof(C)>(apf + at + e * T + i, Lval + lo + e);
                        }
                    const bool in = g + i < P.n;
                    for (int j = 0; j < nr; ++j) copy_async<16>(rd + j * T + i, s_in[j] + (in ? g + i : 0), in);
                }
            } else if (phase == 1 && ONE && bb > 0) {
                for (int i = pt; i < myrows; i += PROD) {
                    const bool in = g + r0 + i < P.n;
                    for (int j = 0; j < nr; ++j)
                        copy_async<16>(tpf + ((bb % 3) * R + j) * SR + i, s_out[j] + (in ? g + r0 + i : 0), in);
                }
            }
        };
        int slot = 0, round = 0, issued = 0;  // c = round * NS + slot
        bool ok = true;
        fetch_bounds(0);
        for (int b = 0; b < nsteps && ok; ++b) {
            const C* M = (phase == 0 || b == 0 ? Dinv : E) + (size_t)block_of(b) * T * T;
            for (int rs = r0; rs < r1; rs += SR) {
                if (lane == 0) {
                    if (round > 0)
                        ok = bounded([&] { return mbar_try_wait(&empty[slot], (uint32_t)((round - 1) & 1)); }, 4);
                    if (failed_flag(&s_fail)) ok = false;
                }
                ok = __shfl_sync(0xffffffffu, (int)ok, 0) != 0;
                if (!ok) break;
                const int rows = min(SR, r1 - rs);
                C* dst = stage + (size_t)slot * SR * TP;
                if (pt == 0) mbar_expect_tx(&full[slot], (uint32_t)((size_t)rows * T * sizeof(C)));
                __syncwarp();
                asm volatile("fence.proxy.async.shared::cta;" ::: "memory");
                for (int i = pt; i < rows; i += PROD)
                    tma_load_1d(dst + (size_t)i * TP, M + (size_t)(rs + i) * T, (uint32_t)(T * sizeof(C)),
                                &full[slot]);
                if (b == 0 && rs == r0) vectors_ready();
                if (!ONE && myrows <= SR && b >= 2) {
                    // one chunk a step in this CTA: the inputs' buffer, as above.  The outcome
                    // is not kept in lane 0 alone (it would leave the loop by itself, and the
                    // others wait for it in the next shuffle): a wait that ran out has set
                    // s_fail, which the next chunk's check hands to the whole warp.
                    if (lane == 0)
                        bounded([&] { return mbar_try_wait(&empty[(b - 2) % NS], (uint32_t)(((b - 2) / NS) & 1)); }, 4);
                    __syncwarp();
                }
                if (rs == r0) {
                    copies_done();  // the bounds asked for a step ago
                    __syncwarp();
                    fetch_inputs(b - LAG);
                    fetch_bounds(b + 1);
                }
                if constexpr (ONE) {
                    if (b > 0) arrive_after_copies(&full[slot == 0 ? NS - 1 : slot - 1]);
                } else {
                    arrive_after_copies(&full[slot]);
                }
                ++issued;
                if (++slot == NS) {
                    slot = 0;
                    ++round;
                }
            }
        }
        if constexpr (ONE) {
            // the last chunk's inputs: their buffer is free when the chunk two before is
            const int c = nsteps - 1;
            if (ok && c >= 0) {
                if (lane == 0 && c >= 2)
                    ok = bounded([&] { return mbar_try_wait(&empty[(c - 2) % NS], (uint32_t)(((c - 2) / NS) & 1)); }, 4);
                ok = __shfl_sync(0xffffffffu, (int)ok, 0) != 0;
                copies_done();
                __syncwarp();
                if (ok) fetch_inputs(c);
                arrive_after_copies(&full[c % NS]);
            } else if (issued > 0) {
                arrive_after_copies(&full[(issued - 1) % NS]);
            }
        }
        copies_done();
        // stopped by a failure: the last issued copies may still be in flight,
        // and this CTA's shared memory must outlive them
        if (pt == 0 && (!ok || failed_flag(&s_fail))) {
            for (int d = max(0, issued - NS); d < issued; ++d) {
                long long it = 0;
                while (!mbar_try_wait(&full[d % NS], (uint32_t)((d / NS) & 1)) && ++it < WAIT_LIMIT) {
                }
            }
        }
    } else {
        // ---- consumers.  A step is a chain of short phases, and with two or three
        // warps a scheduler an instruction of such a chain costs about five clocks
        // whatever it does: everything that does not depend on the vector (indices,
        // inputs, the stage's wait, remote addresses) is done ahead of its arrival.
        //
        // A complex128 value is dealt to two lanes, one a component: an FP64 instruction
        // holds its scheduler's pipe 64 clocks however few lanes are active.
        constexpr int NC = sizeof(C) == 16 ? 2 : 1;
        constexpr int V = 2 / NC;  // real values a lane holds of one complex value
        // this warp's 16-byte column units of every row, and its columns
        const int U = T / VN;
        const int u0 = (warp * U) / CL_WARPS, u1 = ((warp + 1) * U) / CL_WARPS;
        const int c0 = u0 * VN, nc = (u1 - u0) * VN;
        const int dir = (phase == 0) != (side != 0) ? 1 : -1;  // block_of(b + 1) - block_of(b)

        // The rows of a chunk and their lanes: lane = row r (of 2^lg >= rows), then the
        // column phase cp of CP = 2^lgc, no more phases than the warp has units.  ONE: a
        // CTA's rows are one chunk, and all of this is loop-invariant.
        struct Lay {
            int rows, lg, lgc, r, cp;
            bool on;
        };
        auto layout = [&](int rows) {
            Lay y;
            y.rows = rows;
            y.lg = rows > 1 ? 32 - __clz(rows - 1) : 0;
            y.lgc = min(5 - y.lg, u1 - u0 > 1 ? 32 - __clz(u1 - u0 - 1) : 0);
            y.r = lane & ((1 << y.lg) - 1);
            y.cp = lane >> y.lg;
            y.on = y.r < rows && y.cp < (1 << y.lgc);
            return y;
        };
        Lay L = layout(min(SR, myrows));

        // t_k of a chunk's rows, several chunks a step: warp w takes those of job j = w out
        // of its partial sums
        auto fetch_t = [&](int64_t gr, int rows) {
            if (lane < rows && warp < nr)
                copy_async<16>(tpf + warp * SR + lane, s_out[warp] + (gr + lane < P.n ? gr + lane : 0), gr + lane < P.n);
        };
        // How the rows of a chunk are finished.  EVERY (up to two jobs in complex64):
        // every warp adds up all rows' partial sums for itself and sends them to its own
        // CTAs, a store to one CTA at a time whose lanes' addresses are contiguous.
        // Otherwise LPE lanes share a (row, job), each adding up its share of the partial
        // sums (complex128: of one component) and sending to its share of the CTAs.
        constexpr bool EVERY = NC == 1 && R <= 2;
        constexpr int LPE = R <= 2 ? 8 : (R == 4 || NC == 2 ? 4 : 2);
        constexpr int DSTEP = EVERY ? CL_WARPS : LPE;
        const int dst = EVERY ? warp : tid % LPE;  // first CTA this thread sends to
        uint32_t rvec[2], rbar[2];
#pragma unroll
        for (int x = 0; x < 2; ++x) {
            rvec[x] = mapa_u32(vbuf, min(dst + x * DSTEP, Ccl - 1));
            rbar[x] = mapa_u32(vbar, min(dst + x * DSTEP, Ccl - 1));
        }

        vectors_ready();
        int slot = 0, chunk = 0;
        uint32_t spar = 0, vpar = 0;     // parities of the stages' round and of the vectors' round
        int cur = 0, prv = 2;            // b % 3, (b - 1) % 3
        for (int b = 0; b < nsteps; ++b) {
            const bool fwd = phase == 0 || b == 0;
            const int64_t g0 = (int64_t)block_of(b) * T;
            const C* vprev = vbuf + prv * R * T;   // t_outer (fwd) or x_inner (bwd)
            const bool last = b == nsteps - 1;     // nobody reads the last vector: not sent
            // the step's inputs, off the chain
            constexpr bool EARLY = R <= 2;  // more jobs: too many registers
            constexpr int PF = NC;          // entries a lane
            int in_n[PF], in_c[PF][NE];
            C in_a[PF][NE];
            Rt in_r[PF][EARLY ? R : 1][V];
            C in_t = zero_c<C>();
            auto read_part = [&](const double2* p, int cm, Rt (&v)[V]) {
                const double* d = reinterpret_cast<const double*>(p);
                if constexpr (NC == 2) {
                    v[0] = d[cm];
                } else {
                    v[0] = (Rt)d[0];
                    v[1] = (Rt)d[1];
                }
            };
            // the stage and the inputs: there long before the vector
            bounded([&] { return mbar_try_wait(&full[slot], spar); }, 2);
            const double2* rin = rpf + (b & 1) * R * T + c0;
            const int* bin = bpf + (b & 3) * 2 * T + c0;
            if (phase == 0 && pf_ok) {
#pragma unroll
                for (int x = 0; x < PF; ++x) {
                    const int id = lane + 32 * x, i = id / NC;
                    in_n[x] = 0;
                    if (id < nc * NC) {
                        in_n[x] = bin[T + i] - bin[i];
                        const int at = (b & 1) * NE * T + c0 + i;
#pragma unroll
                        for (int e = 0; e < NE; ++e)
                            if (e < in_n[x]) {
                                in_c[x][e] = cpf[at + e * T];
                                in_a[x][e] = apf[at + e * T];
                            }
                        if constexpr (EARLY) {
#pragma unroll
                            for (int j = 0; j < R; ++j)
                                if (j < nr) read_part(rin + j * T + i, id % NC, in_r[x][j]);
                        }
                    }
                }
            }
            if constexpr (ONE && R == 1)
                if (!fwd && warp == 0 && L.on) in_t = from_c128<C>(tpf[cur * SR + L.r]);
            if (b > 0) {
                // the previous step's vector: every CTA's rows, delivered by st.async
                bounded([&] { return mbar_try_wait_cluster(&vbar[prv], vpar); }, 3);
                // re-arm that barrier for step b+2 now: no CTA can send step b+2's rows
                // before it has ours of step b+1, so the expected bytes are always
                // registered before the first of them arrives
                if (tid == 0 && b + 2 <= nsteps - 2) mbar_expect_tx(&vbar[prv], vec_bytes);
            }
            if (fwd) {
                // s_k = r_k - L_k t_outer in this warp's columns
                if (phase == 0 && pf_ok) {
#pragma unroll
                    for (int x = 0; x < PF; ++x) {
                        const int id = lane + 32 * x, i = id / NC, cm = id % NC;
                        if (id < nc * NC) {
#pragma unroll
                            for (int j = 0; j < R; ++j) {
                                if (j >= nr) break;
                                Rt v[V];
                                if constexpr (EARLY) {
#pragma unroll
                                    for (int c = 0; c < V; ++c) v[c] = in_r[x][j][c];
                                } else {
                                    read_part(rin + j * T + i, cm, v);
                                }
                                const C* tj = vprev + j * T;
                                auto entry = [&](const C a, const C t) {
                                    if constexpr (NC == 2) {
                                        v[0] = fma(-a.x, cm ? t.y : t.x, v[0]);
                                        v[0] = fma(cm ? -a.y : a.y, cm ? t.x : t.y, v[0]);
                                    } else {
                                        v[0] -= a.x * t.x - a.y * t.y;
                                        v[1] -= a.x * t.y + a.y * t.x;
                                    }
                                };
#pragma unroll
                                for (int e = 0; e < NE; ++e)
                                    if (e < in_n[x]) entry(in_a[x][e], tj[in_c[x][e]]);
                                for (int e = bin[i] + NE; e < bin[i] + in_n[x]; ++e) entry(Lval[e], tj[P.Lcol[e]]);
                                C* d = sbuf + j * T + c0 + i;
                                if constexpr (NC == 2) reinterpret_cast<double*>(d)[cm] = v[0];
                                else *d = C{v[0], v[1]};
                            }
                        }
                    }
                } else {
                    // without the fetched inputs; x_mid's (phase 1) takes the couplings to both
                    // neighbours, their t from the copies
                    for (int id = lane; id < nc * nr; id += 32) {
                        const int i = c0 + id % nc, j = id / nc;
                        const int64_t g = g0 + i;
                        C v = zero_c<C>();
                        if (g < P.n) {
                            v = from_c128<C>(s_in[j][g]);
                            const double2* tw = s_in[j] + ((int64_t)VS_W - in_slot) * js.n;
                            for (int e = P.Lptr[g]; e < P.Lptr[g + 1]; ++e) {
                                const C a = Lval[e];
                                const int c = P.Lcol[e];
                                const C t = phase ? from_c128<C>(tw[c < T ? g0 - T + c : g0 + c]) : vprev[j * T + c];
                                v.x -= a.x * t.x - a.y * t.y;
                                v.y -= a.x * t.y + a.y * t.x;
                            }
                        }
                        sbuf[j * T + i] = v;
                    }
                }
                __syncwarp();
            }
            const C* rhs = fwd ? sbuf : vprev;
            for (int rs = r0; ONE ? rs == r0 : rs < r1; rs += SR, ++chunk) {
                C* rbuf = red + (chunk & 1) * RW * R * SR;
                if constexpr (!ONE) {
                    if (rs > r0) bounded([&] { return mbar_try_wait(&full[slot], spar); }, 2);
                    L = layout(min(SR, r1 - rs));
                    // many rows a CTA: the matrices bound the step, not its chain
                    if (!fwd) fetch_t(g0 + rs, L.rows);
                }
                const int CP = 1 << L.lgc;
                Rt acc[R][2];
#pragma unroll
                for (int j = 0; j < R; ++j) acc[j][0] = acc[j][1] = Rt(0);
                if (L.on) {
                    const VT* Mrow = reinterpret_cast<const VT*>(stage + (slot * SR + L.r) * TP);
                    int u = u0 + L.cp;
                    if constexpr (NC == 1) {
                        const VT* X = reinterpret_cast<const VT*>(rhs);  // unit u of job j at X[j * U + u]
                        // packed FP32 pairs, pa_j += (m.x, m.x) * (x.x, x.y) and
                        // pb_j += (m.y, m.y) * (x.x, x.y), so that m x = (pa.x - pb.y, pa.y + pb.x):
                        // two paired FMAs per complex product instead of four scalar ones
                        float2 pa[R], pb[R];
#pragma unroll
                        for (int j = 0; j < R; ++j) pa[j] = pb[j] = make_float2(0.f, 0.f);
                        auto units = [&](auto un) {
                            constexpr int N = decltype(un)::value;
                            VT mv[N], xv[N][R];
#pragma unroll
                            for (int i = 0; i < N; ++i) {
                                mv[i] = Mrow[u + i * CP];
#pragma unroll
                                for (int j = 0; j < R; ++j) xv[i][j] = X[j * U + u + i * CP];
                            }
#pragma unroll
                            for (int i = 0; i < N; ++i)
#pragma unroll
                                for (int e = 0; e < VN; ++e) {
                                    const C m = Vec16<C>::get(mv[i], e);
                                    const float2 mr = make_float2(m.x, m.x), mi = make_float2(m.y, m.y);
#pragma unroll
                                    for (int j = 0; j < R; ++j) {
                                        const C x = Vec16<C>::get(xv[i][j], e);
                                        const float2 xx = make_float2(x.x, x.y);
                                        pa[j] = __ffma2_rn(mr, xx, pa[j]);
                                        pb[j] = __ffma2_rn(mi, xx, pb[j]);
                                    }
                                }
                            u += N * CP;
                        };
                        if constexpr (R == 1)
                            while (u + 3 * CP < u1) units(std::integral_constant<int, 4>{});
                        if constexpr (R <= 2)
                            while (u + CP < u1) units(std::integral_constant<int, 2>{});
                        while (u < u1) units(std::integral_constant<int, 1>{});
#pragma unroll
                        for (int j = 0; j < R; ++j) {
                            acc[j][0] = pa[j].x - pb[j].y;
                            acc[j][1] = pa[j].y + pb[j].x;
                        }
                    } else {
                        for (; u < u1; u += CP) {
                            const C m = Mrow[u];
#pragma unroll
                            for (int j = 0; j < R; ++j) {
                                const C x = rhs[j * T + u];
                                acc[j][0] = fma(m.x, x.x, acc[j][0]);
                                acc[j][1] = fma(m.x, x.y, acc[j][1]);
                                acc[j][0] = fma(-m.y, x.y, acc[j][0]);
                                acc[j][1] = fma(m.y, x.x, acc[j][1]);
                            }
                        }
                    }
                }
                // Sum the column phases of each row: while a lane holds several jobs it keeps
                // half of them and trades the other half with its partner, so that the
                // stages cost R/2 + R/4 + ... sums instead of R each.
                int jb = 0, width = R, dup = 0;
                int cpart = -1;  // the component a lane has kept
#pragma unroll
                for (int st = 0; st < 5; ++st) {
                    if (st >= L.lgc) break;
                    const int mask = 1 << (L.lg + L.lgc - 1 - st);
                    const int w = R >> st;  // constant after unrolling
                    if (w > 1) {
                        const bool upper = (lane & mask) != 0;
#pragma unroll
                        for (int j = 0; j < R / 2; ++j)
                            if (j < w / 2) {
#pragma unroll
                                for (int v = 0; v < 2; ++v) {
                                    const Rt give = upper ? acc[j][v] : acc[j + w / 2][v];
                                    const Rt keep = upper ? acc[j + w / 2][v] : acc[j][v];
                                    acc[j][v] = keep + __shfl_xor_sync(0xffffffffu, give, mask);
                                }
                            }
                        if (upper) jb += w / 2;
                        width = w / 2;
                    } else if (NC == 2 && (st == 0 || (R >> (st - 1)) > 1)) {
                        // complex128: then a component, an FP64 addition less a stage
                        const bool upper = (lane & mask) != 0;
                        const Rt give = upper ? acc[0][0] : acc[0][1];
                        const Rt keep = upper ? acc[0][1] : acc[0][0];
                        acc[0][0] = keep + __shfl_xor_sync(0xffffffffu, give, mask);
                        cpart = upper ? 1 : 0;
                    } else {
#pragma unroll
                        for (int v = 0; v < V; ++v) acc[0][v] += __shfl_xor_sync(0xffffffffu, acc[0][v], mask);
                        dup |= mask;
                    }
                }
                if constexpr (!ONE) {
                    if (!fwd) {
                        copies_done();
                        __syncwarp();
                    }
                }
                if (L.on && (lane & dup) == 0) {
                    const double2* tch = tpf + (ONE ? cur * R * SR : 0) + L.r;
#pragma unroll
                    for (int j = 0; j < R; ++j) {
                        if (j < width && jb + j < nr) {
                            if (!fwd && jb + j == warp) {  // R <= 8 jobs: one a warp
                                if constexpr (!(ONE && R == 1)) in_t = from_c128<C>(tch[(jb + j) * SR]);
                                acc[j][0] -= NC == 2 && cpart == 1 ? in_t.y : in_t.x;
                                if (NC == 1 || cpart < 0) acc[j][1] -= in_t.y;
                            }
                            C* d = rbuf + ((jb + j) * SR + L.r) * RW + warp;
                            if (NC == 1 || cpart < 0) *d = C{acc[j][0], acc[j][1]};
                            else reinterpret_cast<Rt*>(d)[cpart] = acc[j][0];
                        }
                    }
                }
                consumer_sync();  // partial sums written; the stage is consumed
                if (tid == 0) mbar_arrive(&empty[slot]);
                const bool failed = failed_flag(&s_fail);
                const int nel = nr << L.lg;  // (row, job) pairs, rows padded to a power of two
                const Rt sgn = fwd ? Rt(1) : Rt(-1);
                auto finished = [&](const C v, int r, int j) {
                    if (failed) return;
                    if (!last) {
                        const uint32_t off = (uint32_t)(((cur * R + j) * T + rs + r) * (int)sizeof(C));
                        const uint32_t boff = (uint32_t)(cur * (int)sizeof(uint64_t));
                        if (dst < Cact) st_async_c(rvec[0] + off, v, rbar[0] + boff);
                        if (dst + DSTEP < Cact) st_async_c(rvec[1] + off, v, rbar[1] + boff);
                        if constexpr (DSTEP < 8)
                            for (int qq = dst + 2 * DSTEP; qq < Cact; qq += DSTEP)
                                st_async_c(mapa_u32(vbuf, qq) + off, v, mapa_u32(vbar, qq) + boff);
                    } else if (dst == 0 && g0 + rs + r < P.n) {
                        // the last vector; x_mid is every side's, side 0 stores it
                        const int64_t g = g0 + rs + r;
                        if (phase == 0 || b > 0 || side == 0) s_out[j][g] = to_c128(v);
                        // t_{mid±1}: the copy that launch 1 reads
                        if (phase == 0) s_out[j][g + ((int64_t)VS_W - out_slot) * js.n] = to_c128(v);
                    }
                };
                if constexpr (EVERY) {
                    for (int e = lane; e < nel; e += 32) {
                        const int r = R == 1 ? e : e & ((1 << L.lg) - 1), j = R == 1 ? 0 : e >> L.lg;
                        if (r >= L.rows) continue;
                        const C* pr = rbuf + (j * SR + r) * RW;
                        C p[CL_WARPS];
#pragma unroll
                        for (int w = 0; w < CL_WARPS; ++w) p[w] = pr[w];
#pragma unroll
                        for (int h = CL_WARPS / 2; h > 0; h /= 2)
#pragma unroll
                            for (int w = 0; w < h; ++w) {
                                p[w].x += p[w + h].x;
                                p[w].y += p[w + h].y;
                            }
                        finished(C{sgn * p[0].x, sgn * p[0].y}, r, j);
                    }
                } else {
                    constexpr int PARTS = LPE / NC;
                    const int comp = NC == 2 ? tid % 2 : 0, part = (tid % LPE) / NC;
                    for (int e = tid / LPE; (e & ~(32 / LPE - 1)) < nel; e += CL_WARPS * 32 / LPE) {
                        const int r = e & ((1 << L.lg) - 1), j = e >> L.lg;
                        const bool in = r < L.rows && j < nr;
                        const int at = (in ? j * SR + r : 0) * RW + part;
                        C v;
                        if constexpr (NC == 2) {
                            const double* pr = reinterpret_cast<const double*>(rbuf + at) + comp;
                            double a = pr[0];
#pragma unroll
                            for (int w = PARTS; w < CL_WARPS; w += PARTS) a += pr[2 * w];
#pragma unroll
                            for (int m = NC; m < LPE; m *= 2) a += __shfl_xor_sync(0xffffffffu, a, m);
                            if (!fwd) a = -a;
                            const double o = __shfl_xor_sync(0xffffffffu, a, 1);
                            v.x = comp ? o : a;
                            v.y = comp ? a : o;
                        } else {
                            const C* pr = rbuf + at;
                            v = pr[0];
#pragma unroll
                            for (int w = PARTS; w < CL_WARPS; w += PARTS) {
                                v.x += pr[w].x;
                                v.y += pr[w].y;
                            }
#pragma unroll
                            for (int m = 1; m < LPE; m *= 2) {
                                v.x += __shfl_xor_sync(0xffffffffu, v.x, m);
                                v.y += __shfl_xor_sync(0xffffffffu, v.y, m);
                            }
                            v = C{sgn * v.x, sgn * v.y};
                        }
                        if (in) finished(v, r, j);
                    }
                }
                if (++slot == NS) {
                    slot = 0;
                    spar ^= 1;
                }
                if (rs != r0) continue;
                // Once a step, while its rows are on their way: the previous vector's rows of
                // this CTA go to memory.  (That vector stays until the peers have our next rows.)
                if (b > 0 && !failed && (phase == 0 || b > 1 || side == 0)) {
                    const int64_t gp = g0 - (int64_t)dir * T + r0;
                    for (int i = (CL_WARPS - 1 - warp) * 32 + lane; i < myrows; i += CL_WARPS * 32)
                        if (gp + i < P.n)
                            for (int j = 0; j < nr; ++j) s_out[j][gp + i] = to_c128(vprev[j * T + r0 + i]);
                }
            }
            if (b > 0 && prv == 2) vpar ^= 1;
            prv = cur;
            cur = cur == 2 ? 0 : cur + 1;
        }
    }
    // the cluster barrier keeps every CTA's shared memory alive until all peers
    // have finished sending into it
    cl.sync();
}

// ---------------------------------------------------------------------------
namespace {

struct Plan {
    int R = 1, SR = 1, NS = 3, TP = 1;
    int pf = 0;  // the right-hand sides' inputs are fetched ahead
    size_t smem = 0;
};

// Row stride (complex values) of a stage in shared memory: a whole number of
// 16-byte units, and an odd one, so that the 16-byte loads of 8 consecutive
// rows at the same column fall in distinct bank groups.
int padded_row(int T, size_t cs) {
    int TP = T;
    while ((TP * cs) % 16 != 0 || ((TP * cs / 16) & 1) == 0) ++TP;
    return TP;
}

// the chain's vectors and the inputs fetched ahead
size_t vec_smem(int R, int T, size_t cs, bool pf) {
    return (size_t)4 * R * T * cs +
           (pf ? (size_t)T * (2 * R * sizeof(double2) + 2 * NE * (cs + sizeof(int)) + 8 * sizeof(int)) : 0);
}

// a stage row of R right-hand sides: partial sums, fetched t
size_t row_smem(int R, size_t cs) { return (size_t)2 * RW * R * cs + 3 * R * sizeof(double2); }

size_t plan_smem(const Plan& p, int T, size_t cs) {
    return (size_t)p.NS * p.SR * p.TP * cs + vec_smem(p.R, T, cs, p.pf) + p.SR * row_smem(p.R, cs) +
           (2 * p.NS + 3) * sizeof(uint64_t) + 32;
}

// Stage height for a CTA of Tc rows: each chunk of `rows` rows occupies the
// lanes as rows x column phases with rows padded to a power of two, so the
// estimate charges the padded rows' multiply-adds plus a fixed cost per chunk: its
// waits, barrier and sums.  Clocks: complex128 64 an FP64 instruction on each
// scheduler; complex64 measured at T = 200 on CTAs of 100 and 200 rows (16 and 25 rows
// a chunk with eight right-hand sides: 1,790 and 3,110; 16 and 20 with one: 880 and
// 1,100).
int choose_rows(int Tc, int SRmax, int T, size_t cs, int R) {
    const int VN = (int)(16 / cs);
    const bool dbl = cs == 16;
    const int Uw = cdiv_up(T / VN, CL_WARPS);
    const double per_unit = dbl ? R * 4 * 2 * 64.0 : R * VN * 14.0;
    const double per_chunk = dbl ? 4000.0 : (R <= 2 ? 700.0 : 250.0);
    int best = SRmax;
    double best_c = 1e300;
    for (int SR = 1; SR <= SRmax; ++SR) {
        double c = 0.0;
        for (int a = 0; a < Tc; a += SR) {
            const int rows = std::min(SR, Tc - a);
            int SRp = 1;
            while (SRp < rows) SRp <<= 1;
            const int CP = 32 / SRp;
            c += (double)((Uw + CP - 1) / CP) * per_unit + per_chunk;
        }
        if (c < best_c) {
            best_c = c;
            best = SR;
        }
    }
    return best;
}

// The plan of R right-hand sides for CTAs of Tc rows in `budget` bytes of shared
// memory: stage height, and whether inputs are fetched ahead.  That shortens the
// chain; where its shared memory would cut a CTA's rows into more chunks, the
// multiply-adds bound the step, not the chain (complex128, T = 200, eight
// right-hand sides on a cluster of 16: stages of 3 rows instead of 9).
bool make_plan(int T, size_t cs, int R, int Tc, Plan& p, size_t budget = 220 * 1024) {
    p.R = R;
    p.NS = 3;
    p.TP = padded_row(T, cs);
    auto height = [&](bool pf) {
        const size_t vec = vec_smem(R, T, cs, pf) + 112;
        if (vec >= budget) return 0;
        const int most = (int)std::min<size_t>(32, (budget - vec) / ((size_t)p.NS * p.TP * cs + row_smem(R, cs)));
        return most < 1 ? 0 : choose_rows(Tc, most, T, cs, R);
    };
    p.SR = height(false);
    p.pf = T <= PF_T && p.SR >= 1 && height(true) == p.SR;
    p.smem = plan_smem(p, T, cs);
    return p.SR >= 1;
}

// Largest R (right-hand sides per pass), at most want_R, whose stages fit.
int choose_R(int T, size_t cs, int want_R) {
    Plan p;
    for (int R : {8, 4, 2, 1})
        if ((R <= want_R || R == 1) && make_plan(T, cs, R, T, p)) return R;
    return 0;
}

template <class C, int R, int MINB> void set_smem_attr(size_t smem) {
    static size_t attr_set = 0;  // per instantiation
    static bool nonportable = false;
    auto both = [](auto&& f) {
        f(k_block_solve_cl<C, R, MINB, true, 0>);
        f(k_block_solve_cl<C, R, MINB, true, 1>);
        f(k_block_solve_cl<C, R, MINB, false, 0>);
        f(k_block_solve_cl<C, R, MINB, false, 1>);
    };
    if (!nonportable) {
        // clusters of up to 16 CTAs (beyond the portable 8) for launches of few groups
        // (where that is refused, the occupancy query reports no room for them)
        both([](auto* k) {
            if (cudaFuncSetAttribute(k, cudaFuncAttributeNonPortableClusterSizeAllowed, 1) != cudaSuccess)
                (void)cudaGetLastError();
        });
        nonportable = true;
    }
    if (smem > attr_set) {
        both([&](auto* k) {
            SIM_CUDA(cudaFuncSetAttribute(k, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)smem));
        });
        attr_set = smem;
    }
}

cudaLaunchConfig_t cluster_config(int ngroups, int Ccl, size_t smem, cudaStream_t st, cudaLaunchAttribute* attr) {
    cudaLaunchConfig_t cfg = {};
    cfg.gridDim = dim3(ngroups * Ccl);
    cfg.blockDim = dim3(CL_THREADS);
    cfg.dynamicSmemBytes = smem;
    cfg.stream = st;
    attr[0].id = cudaLaunchAttributeClusterDimension;
    attr[0].val.clusterDim.x = Ccl;
    attr[0].val.clusterDim.y = 1;
    attr[0].val.clusterDim.z = 1;
    cfg.attrs = attr;
    cfg.numAttrs = 1;
    return cfg;
}

// How many clusters of Ccl CTAs with `smem` bytes each the GPU holds at once
// (the CUDA occupancy query: clusters are placed within a GPC, so this is not
// simply SMs / Ccl).  Cached per (instantiation, Ccl, smem).
template <class C, int R, int MINB> int max_active_clusters(int Ccl, size_t smem) {
    static std::map<std::pair<int, size_t>, int> cache;
    const auto key = std::make_pair(Ccl, smem);
    const auto it = cache.find(key);
    if (it != cache.end()) return it->second;
    set_smem_attr<C, R, MINB>(smem);
    cudaLaunchAttribute attr[1];
    const cudaLaunchConfig_t cfg = cluster_config(1, Ccl, smem, nullptr, attr);
    int n = 0;
    if (cudaOccupancyMaxActiveClusters(&n, k_block_solve_cl<C, R, MINB, true, 0>, &cfg) != cudaSuccess) {
        (void)cudaGetLastError();
        n = 0;
    }
    cache[key] = n;
    return n;
}

template <class C, int R, int MINB>
void launch_cl(const Pencil& P, const JobSpace& js, int in_slot, int out_slot, void* const* fptrs, const Groups& groups,
               int ngroups, int Ccl, const Plan& pl, int* d_err, cudaStream_t st) {
    set_smem_attr<C, R, MINB>(pl.smem);
    cudaLaunchAttribute attr[2];
    cudaLaunchConfig_t cfg = cluster_config(ngroups * (P.mid + 1 < P.nb ? 2 : 1), Ccl, pl.smem, st, attr);
    // launch 1 may start before launch 0 has ended (griddepcontrol in the kernel)
    attr[1].id = cudaLaunchAttributeProgrammaticStreamSerialization;
    attr[1].val.programmaticStreamSerializationAllowed = 1;
    auto launch = [&](auto* kernel, bool after) {
        cfg.numAttrs = after ? 2 : 1;
        SIM_CUDA(cudaLaunchKernelEx(&cfg, kernel, P, js, in_slot, out_slot, fptrs, groups, pl.SR, pl.NS, pl.TP, pl.pf, d_err));
        SIM_LAUNCH_CHECK();
    };
    if (cdiv_up(P.T, Ccl) <= pl.SR) {  // every CTA's rows in one chunk
        if (P.mid > 0) launch(k_block_solve_cl<C, R, MINB, true, 0>, false);
        launch(k_block_solve_cl<C, R, MINB, true, 1>, P.mid > 0);
    } else {
        if (P.mid > 0) launch(k_block_solve_cl<C, R, MINB, false, 0>, false);
        launch(k_block_solve_cl<C, R, MINB, false, 1>, P.mid > 0);
    }
}

// Launch shape: CTAs per group (cluster size), CTAs per SM, and the plan.
struct Shape {
    int Ccl = 1, minb = 1;
    Plan pl;
};

// The shape of a launch of ng clusters: every cluster in one wave if the GPU holds
// that many clusters, and then the largest cluster (the most SMs, the fewest
// rows per CTA on the chain's critical path); cluster sizes need not be powers
// of two.  Two CTAs per SM are considered for single right-hand sides in
// complex64, whose plan then fits in half of an SM's shared memory.
template <class C, int R>
Shape choose_shape(const Pencil& P, size_t cs, int ng) {
    Shape best;
    double best_cost = 1e300;
    const int cmax = std::min(16, P.T);
    for (int minb = 1; minb <= 2; ++minb) {
        if (minb == 2 && !(R == 1 && sizeof(C) == 8)) continue;
        for (int c = 1; c <= cmax; ++c) {
            Plan q;
            if (!make_plan(P.T, cs, R, cdiv_up(P.T, c), q, minb == 2 ? 110 * 1024 : 220 * 1024)) continue;
            int maxc = 0;
            if constexpr (R == 1 && sizeof(C) == 8)
                maxc = minb == 1 ? max_active_clusters<C, R, 1>(c, q.smem) : max_active_clusters<C, R, 2>(c, q.smem);
            else
                maxc = max_active_clusters<C, R, 1>(c, q.smem);
            if (maxc <= 0) continue;
            const int waves = (ng + maxc - 1) / maxc;
            // waves first, then the fewest rows per CTA, then one CTA per SM
            const double cost = waves * 1e6 + (double)((P.T + c - 1) / c) * 10.0 + minb;
            if (cost < best_cost) {
                best_cost = cost;
                best.Ccl = c;
                best.minb = minb;
                best.pl = q;
            }
        }
    }
    if (best_cost == 1e300) {  // no occupancy answer: one CTA per group
        best.Ccl = 1;
        best.minb = 1;
        make_plan(P.T, cs, R, P.T, best.pl);
    }
    return best;
}

int* g_grp = nullptr;
int g_grp_cap = 0;
// pinned staging for the group table: a pageable upload would synchronise the stream
int* g_grp_h[2] = {nullptr, nullptr};
cudaEvent_t g_grp_ev[2] = {nullptr, nullptr};
int g_grp_h_cap = 0;
int g_grp_flip = 0;

}  // namespace

bool block_solve_cluster(const Pencil& P, int precision, const JobSpace& js, const std::vector<int>& active,
                         int in_slot, int out_slot, const double2* d_sigma, void* const* d_factor_ptrs,
                         cudaStream_t st) {
    if (active.empty()) return true;
    const size_t cs = precision == SIM_FP64 ? sizeof(double2) : sizeof(float2);
    if ((P.T * cs) % 16 != 0) return false;
    // group active jobs that share a shift (consecutive in the active list)
    std::vector<std::vector<int>> groups;
    int maxr = 1;
    for (size_t i = 0; i < active.size(); ++i) {
        const int j = active[i];
        if (!groups.empty() && js.h_jobshift[groups.back().back()] == js.h_jobshift[j] && groups.back().size() < 8)
            groups.back().push_back(j);
        else
            groups.push_back({j});
        maxr = std::max<int>(maxr, (int)groups.back().size());
    }
    const int R = choose_R(P.T, cs, maxr);
    if (R == 0) return false;
    // split groups larger than the plan's R
    std::vector<std::vector<int>> gs;
    for (auto& g : groups)
        for (size_t a = 0; a < g.size(); a += R) gs.emplace_back(g.begin() + a, g.begin() + std::min(g.size(), a + R));
    const int ng = (int)gs.size();
    const int nclusters = ng * (P.mid + 1 < P.nb ? 2 : 1);  // a cluster per side
    std::vector<int> flat((size_t)ng * R, -1);
    for (int g = 0; g < ng; ++g)
        for (size_t j = 0; j < gs[g].size(); ++j) flat[(size_t)g * R + j] = gs[g][j];
    Groups table;
    table.far = nullptr;
    if ((int)flat.size() <= Groups::MAX && js.J <= 32767) {
        std::copy(flat.begin(), flat.end(), table.near);
    } else {
        if ((int)flat.size() > g_grp_cap) {
            if (g_grp) {
                SIM_CUDA(cudaStreamSynchronize(st));
                cudaFree(g_grp);
            }
            g_grp_cap = (int)flat.size() * 2;
            SIM_CUDA(cudaMalloc(&g_grp, sizeof(int) * g_grp_cap * 2));
        }
        if ((int)flat.size() > g_grp_h_cap) {
            for (int b = 0; b < 2; ++b) {
                if (g_grp_ev[b]) SIM_CUDA(cudaEventSynchronize(g_grp_ev[b]));
                if (g_grp_h[b]) cudaFreeHost(g_grp_h[b]);
                SIM_CUDA(cudaMallocHost(&g_grp_h[b], sizeof(int) * flat.size() * 2));
                if (!g_grp_ev[b]) SIM_CUDA(cudaEventCreateWithFlags(&g_grp_ev[b], cudaEventDisableTiming));
            }
            g_grp_h_cap = (int)flat.size() * 2;
        }
        const int fb = g_grp_flip;
        g_grp_flip ^= 1;
        SIM_CUDA(cudaEventSynchronize(g_grp_ev[fb]));  // the copy that last used this buffer is done
        std::copy(flat.begin(), flat.end(), g_grp_h[fb]);
        table.far = g_grp + (size_t)fb * g_grp_cap;
        SIM_CUDA(cudaMemcpyAsync(const_cast<int*>(table.far), g_grp_h[fb], sizeof(int) * flat.size(), cudaMemcpyHostToDevice, st));
        SIM_CUDA(cudaEventRecord(g_grp_ev[fb], st));
    }
    Shape sh;
    if (precision == SIM_FP64) {
        if (R == 8) sh = choose_shape<double2, 8>(P, cs, nclusters);
        else if (R == 4) sh = choose_shape<double2, 4>(P, cs, nclusters);
        else if (R == 2) sh = choose_shape<double2, 2>(P, cs, nclusters);
        else sh = choose_shape<double2, 1>(P, cs, nclusters);
    } else {
        if (R == 8) sh = choose_shape<float2, 8>(P, cs, nclusters);
        else if (R == 4) sh = choose_shape<float2, 4>(P, cs, nclusters);
        else if (R == 2) sh = choose_shape<float2, 2>(P, cs, nclusters);
        else sh = choose_shape<float2, 1>(P, cs, nclusters);
    }
    const int Ccl = sh.Ccl;
    const Plan& pl = sh.pl;
    const double TT = (double)P.T * P.T, blocks = 2.0 * P.nb - 1.0;
    // instrumentation also files each launch under its shape (right-hand sides
    // per pass, CTAs per group), e.g. "block_solve_r8_c2"
    char shape[40];
    snprintf(shape, sizeof shape, "block_solve_r%d_c%d%s", pl.R, Ccl, sh.minb == 2 ? "x2" : "");
    kprof_begin("block_solve", st);
    kprof_begin(shape, st);
#define SIM_LAUNCH_R(CT, RR, MB) \
    launch_cl<CT, RR, MB>(P, js, in_slot, out_slot, d_factor_ptrs, table, ng, Ccl, pl, js.host->err, st)
    if (precision == SIM_FP64) {
        if (pl.R == 8) SIM_LAUNCH_R(double2, 8, 1);
        else if (pl.R == 4) SIM_LAUNCH_R(double2, 4, 1);
        else if (pl.R == 2) SIM_LAUNCH_R(double2, 2, 1);
        else SIM_LAUNCH_R(double2, 1, 1);
    } else {
        if (pl.R == 8) SIM_LAUNCH_R(float2, 8, 1);
        else if (pl.R == 4) SIM_LAUNCH_R(float2, 4, 1);
        else if (pl.R == 2) SIM_LAUNCH_R(float2, 2, 1);
        else if (sh.minb == 2) SIM_LAUNCH_R(float2, 1, 2);
        else SIM_LAUNCH_R(float2, 1, 1);
    }
#undef SIM_LAUNCH_R
    // algorithmic bytes: each group reads the factor once, and 4 vectors per job
    const double alg_bytes = ng * blocks * TT * cs + (double)active.size() * 4.0 * P.n * sizeof(double2);
    const double alg_flops = (double)active.size() * 8.0 * blocks * TT;
    kprof_end(shape, st, alg_bytes, alg_flops);
    kprof_end("block_solve", st, alg_bytes, alg_flops);
    return true;
}

void block_solve_check(JobHost& host) {
    const int code = host.err ? *(volatile int*)host.err : 0;
    if (code == 0) return;
    *host.err = 0;
    throw CudaError{cudaErrorLaunchTimeout, "block solve: a wait on an mbarrier ran out (code " + std::to_string(code) + ")"};
}

}  // namespace sim
