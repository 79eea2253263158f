// Solve phase on the GPU: the nonlinear AMLI-cycle (paper Alg. 2) with nonlinear PCG on the
// coarse levels (Alg. 1), the quadtree-coloured Gauss-Seidel smoother (Sec. 4.5), implicit
// prolongation / restriction (Sec. 4.3), and the outer Krylov iteration (Alg. 1 on the
// finest level, flexible CG with full A-orthogonalisation).
//
// Execution. One application of the preconditioner B^_fine is a fixed program of ops (see
// cycle_ops.cuh) over device-resident data; every scalar stays on the device. It runs as a
// sequence of two kinds of launches. The fine levels' ops between two visits of the coarse levels
// are one launch of a persistent cooperative kernel (one CTA per SM): the CTAs execute each op
// row-parallel and meet at a bounded grid barrier before the next. The coarse levels (pure
// latency) run in the shared memory of a thread-block cluster (cluster_tail.cuh), a launch per
// visit; of a small quadtree all levels do, and an application is that one launch. The outer
// Krylov update is four small kernels per iteration; the host reads one residual per iteration.
#include <algorithm>
#include <cmath>
#include <cstdlib>
#include <cstring>
#include <type_traits>

#include "cluster_tail.cuh"
#include "cycle_ops.cuh"

namespace amg {

template <class T>
using GLev = LevelDev<T, kBig>;           // level in HBM

// persistent kernel CTA size (one CTA per SM): the FP64 cycle runs with fewer threads and
// twice the registers each, as its ops at the 64-register cap of 1024 threads spill
constexpr int kPThreads = 1024;
constexpr int kPThreads64 = 512;
template <class T>
constexpr int cycle_threads() { return sizeof(T) == 8 ? kPThreads64 : kPThreads; }
// coarse levels of at least this many rows restrict in two grid-wide passes (OP_RESID,
// OP_GATHER): their rows' children lie in different colours, far apart in HBM, and the
// one-pass form's four-lane gathers read scattered slots
constexpr int kSplitRestrictRows = 524288;


constexpr int kTprofCount = 16 * kMaxLevels;  // cluster's profile slots: 16 op kinds per level

template <class T>
struct CycleArgs {
    const GLev<T> *tab;
    const Op *prog;
    int nlev;
    int k0, k1;                  // this launch's ops
    unsigned long long bar_base; // arrivals at the barrier counter before this launch
    double *partials;            // [2][4][gridDim]
    unsigned long long *bar;     // barrier counter (zeroed before every application)
    int *err;
    unsigned long long *ts;      // per-op end timestamps (profiling) or null
    // host-set barrier fault (amg_debug_barrier_fault): wait limit of every grid barrier, and
    // arrivals the first barrier waits for beyond the grid's (0: none)
    unsigned long long bar_limit_ns;
    int bar_extra;
    // the finest level's input and output vectors when not the table's (FGMRES basis vectors)
    T *rhs0, *e0;
    // the CTAs lend their dynamic shared memory to the big blocks' sweeps; the warp-sized
    // ones go to warps [0, big_wwarps) with big_wslice bytes each (0: to every warp, from
    // global memory)
    int big_smem, big_wwarps;
    unsigned big_wslice;
};

// ---------------------------------------------------------------------------------------
// standalone executor (diagnostic path: amg_apply_cycle on coarse levels, amg_smooth)
template <class T>
__global__ void __launch_bounds__(kRedThreads) k_op(const GLev<T> *__restrict__ tab, Op op,
                                                    RedCtx rc) {
    run_op<GLev<T>, RM_LASTBLOCK>(tab, op, rc, blockIdx.x * blockDim.x + threadIdx.x,
                                  gridDim.x * blockDim.x);
}

// ---------------------------------------------------------------------------------------
// persistent cycle kernel
// sum the per-CTA partials of the previous op (every CTA, identical order) into sc; one
// warp per value, in FP64 for the FP64 cycle and in FP32 for the FP32 cycle (whose per-CTA
// partials are FP32 sums)
template <class T, class TAB>
__device__ __forceinline__ void finalize(const CycleArgs<T> &a, const TAB *tab, const Op &op) {
    const int k = (int)threadIdx.x >> 5, lane = threadIdx.x & 31;
    if (k < op.fin_n) {  // a warp per value
        const int G = gridDim.x;
        double *sc = tab[op.fin_level].sc;
        const double *part = a.partials + ((size_t)op.fin_pb * 4 + k) * G;
        double y;
        if constexpr (sizeof(T) == 4) {
            float x = 0.f;
            for (int b = lane; b < G; b += 32) x += (float)__ldcg(&part[b]);
#pragma unroll
            for (int o = 16; o > 0; o >>= 1) x += __shfl_down_sync(0xffffffffu, x, o);
            y = (double)x;
        } else {
            y = 0.0;
            for (int b = lane; b < G; b += 32) y += __ldcg(&part[b]);
            y = warp_sum(y);
        }
        if (lane == 0 && op.fin_dst[k] >= 0) sc[op.fin_dst[k]] = y;
    }
    __syncthreads();
}

// ops [k0, k1) of an application's program. B: kCoop, kBig (LevelDev)
extern __shared__ __align__(16) unsigned char amg_smem[];

template <class T, int B>
__global__ void __launch_bounds__(cycle_threads<T>(), 1) k_cycle(CycleArgs<T> a) {
    using GL = LevelDev<T, B>;  // the same layout as GLev<T>
    __shared__ GL gtab[kMaxLevels];
    __shared__ unsigned long long target;
    __shared__ int abort_flag;
    if (threadIdx.x == 0) {
        // bar_extra > 0 only under a host-set barrier fault
        target = a.bar_base + (unsigned long long)a.bar_extra;
        abort_flag = ld_volatile_int(a.err) & kErrTimeout;  // of an earlier launch
    }
    {  // the level table, read by every op, lives in shared memory
        const int words = a.nlev * (int)(sizeof(GL) / sizeof(int));
        for (int i = threadIdx.x; i < words; i += blockDim.x)
            ((int *)gtab)[i] = ((const int *)a.tab)[i];
    }
    __syncthreads();
    if (abort_flag) return;
    asm volatile("griddepcontrol.launch_dependents;");  // they wait for the end of this launch
    if (threadIdx.x == 0) {
        if (a.rhs0) gtab[0].rhs = a.rhs0;
        if (a.e0) gtab[0].e = a.e0;
    }
    // the op descriptors pass through shared memory: a few threads fetch the next one while
    // the CTA waits at the barrier, and every thread reads its fields from there (a per-thread
    // copy would cost every thread a 72-byte global load and a local-memory round trip)
    __shared__ Op sop[2];
    constexpr int kOpWords = (int)(sizeof(Op) / sizeof(int));
    if (threadIdx.x < kOpWords)
        ((int *)&sop[a.k0 & 1])[threadIdx.x] = ((const int *)(a.prog + a.k0))[threadIdx.x];
    __syncthreads();
    // rows go to warps in 32-row chunks with the CTA index fastest, so an op over a few
    // thousand rows (the coarse grid-wide levels) spreads over every SM instead of filling the
    // first few CTAs; a warp's rows stay consecutive (coalesced slots, lane = row mod 32)
    const int gtid = (((int)threadIdx.x >> 5) * (int)gridDim.x + (int)blockIdx.x) * 32 +
                     ((int)threadIdx.x & 31);
    const int gnth = gridDim.x * blockDim.x;
    const RedCtx rc{a.partials, nullptr};
    BigScratch sc;
    if ((B & kBig) && a.big_smem) {
        unsigned dyn;
        asm("mov.u32 %0, %%dynamic_smem_size;" : "=r"(dyn));
        sc.p = amg_smem;
        sc.bytes = dyn;
        sc.wwarps = a.big_wwarps;
        sc.wslice = a.big_wslice;
    }
    RowAhead<GL> held;
    op_ahead(gtab[sop[a.k0 & 1].level], sop[a.k0 & 1], gtid, gnth, sc, held);
    for (int k = a.k0; k < a.k1; k++) {
        const Op &op = sop[k & 1];
        // the next descriptor into the other buffer (last read by op k-1), issued before op k
        // runs: a load still in flight at the barrier would delay its release fence
        if (threadIdx.x < kOpWords && k + 1 < a.k1)
            ((int *)&sop[(k + 1) & 1])[threadIdx.x] = ((const int *)(a.prog + k + 1))[threadIdx.x];
        if (op.fin_pb >= 0) finalize(a, gtab, op);
        if (op_has_ahead(gtab[op.level], op, gnth))
            run_op_held<GL, RM_PARTIAL>(gtab[op.level], op, rc, gtid, gnth, BlockGroup{}, sc, held);
        else if (op.kind != OP_NOP)
            run_op<GL, RM_PARTIAL>(gtab, op, rc, gtid, gnth, sc);
        // the end of the launch orders its last op before whatever follows on the stream
        const bool last = k + 1 == a.k1;
        const Op &nx = sop[(k + 1) & 1];
        if (!last && !grid_barrier(a.bar, a.err, target, abort_flag, a.bar_limit_ns,
                                   [&] { op_ahead(gtab[nx.level], nx, gtid, gnth, sc, held); }))
            break;
        if (a.ts && blockIdx.x == 0 && threadIdx.x == 0) a.ts[k] = global_ns();
    }
}

__global__ void k_timestamp(unsigned long long *t) { *t = global_ns(); }

// ---------------------------------------------------------------------------------------
template <class P>
__device__ __forceinline__ void asm_keep(P &p) {
    asm volatile("" : "+l"(p) : : "memory");
}
// Launches that overlap the end of the kernel before them (programmatic dependent launch).
// follow(...) comes first in such a kernel: it lets the next one be launched and waits until
// the kernel before it has ended and its writes can be seen. Every kernel of a chain does so, so
// one that has ended has all before it ended. The pointers pass through it because loads through
// const __restrict__ pointers may otherwise be moved above the wait. With these launches for the
// outer kernels of flexible CG and for the cluster's kernel a solve takes, FP64: 34^2 nodes 702
// -> 644 us, 257^2 6.30 -> 6.20 ms, 1025^2 37.9 -> 37.3 ms. FGMRES's kernels keep the plain
// launch (129^3 nodes 25.8 -> 26.1 ms with it), and so do the grid's (no gain on top).
template <class... P>
__device__ __forceinline__ void follow(P &...p) {
    asm volatile("griddepcontrol.launch_dependents;");
    asm volatile("griddepcontrol.wait;" ::: "memory");
    (asm_keep(p), ...);
}
// a launch that need not wait for the end of the kernel before it
template <class... P, class... A>
void launch_following(void (*kernel)(P...), int grid, int block, cudaStream_t s, A... args) {
    cudaLaunchConfig_t cfg = {};
    cfg.gridDim = dim3(grid);
    cfg.blockDim = dim3(block);
    cfg.stream = s;
    cudaLaunchAttribute attr;
    attr.id = cudaLaunchAttributeProgrammaticStreamSerialization;
    attr.val.programmaticStreamSerializationAllowed = 1;
    cfg.attrs = &attr;
    cfg.numAttrs = 1;
    AMG_CUDA(cudaLaunchKernelEx(&cfg, kernel, P(args)...));
}

// ---------------------------------------------------------------------------------------
// outer Krylov kernels (FP64, pi order)
__global__ void k_gather(int n, const int *__restrict__ idx, const double *__restrict__ src,
                         double *__restrict__ dst) {
    int p = blockIdx.x * blockDim.x + threadIdx.x;
    if (p < n) dst[p] = src[idx[p]];
}

__global__ void k_scatter(int n, const int *__restrict__ idx, const double *__restrict__ src,
                          double *__restrict__ dst) {
    int p = blockIdx.x * blockDim.x + threadIdx.x;
    if (p < n) dst[idx[p]] = src[p];
}

// 1 / a_ii of every row (slot 0 of the sliced ELL holds the diagonal)
template <class T>
__global__ void k_inv_diag(int n, const int *__restrict__ sl, const double *__restrict__ val,
                           T *__restrict__ dinv) {
    int i = blockIdx.x * blockDim.x + threadIdx.x;
    if (i < n) dinv[i] = (T)(1.0 / val[sl[i >> 5] + (i & 31)]);
}

template <class A, class B>
__global__ void k_convert(int n, const A *__restrict__ src, B *__restrict__ dst) {
    int i = blockIdx.x * blockDim.x + threadIdx.x;
    if (i < n) dst[i] = (B)src[i];
}

// (v, v) -> out
__global__ void __launch_bounds__(kRedThreads) k_norm2(int n, const double *__restrict__ v,
                                                       double *out, RedCtx rc) {
    double a[1] = {0.0};
    for (int i = blockIdx.x * blockDim.x + threadIdx.x; i < n; i += gridDim.x * blockDim.x)
        a[0] += v[i] * v[i];
    double *o[1] = {out};
    reduce_store<1, RM_LASTBLOCK, double>(a, o, rc, 0, BlockGroup{});
}

// t = b - A x, (t, t) -> out
__global__ void __launch_bounds__(kRedThreads) k_true_residual(GLev<double> L,
                                                               const double *__restrict__ b,
                                                               const double *__restrict__ x,
                                                               double *__restrict__ t,
                                                               double *out, RedCtx rc) {
    double a[1] = {0.0};
    for (int i = blockIdx.x * blockDim.x + threadIdx.x; i < L.n; i += gridDim.x * blockDim.x) {
        double ri = row_residual(L, i, b, x);
        t[i] = ri;
        a[0] += ri * ri;
    }
    double *o[1] = {out};
    reduce_store<1, RM_LASTBLOCK, double>(a, o, rc, 0, BlockGroup{});
}

// outer scalars: osc[OS_BB] = (b,b), osc[OS_RR] = (r,r), osc[OS_STOP] = breakdown flag,
// osc[OS_RP] = (r, p_i), osc[OS_TT] = (t, t), osc[OS_ERR] = the cycle's error flag (copied here by
// an iteration's last kernel: one read back per iteration), osc[OS_ZQ + j] = (z, A p_j);
// (p_j, A p_j) in opq
enum : int { OS_BB = 0, OS_RR = 1, OS_STOP = 2, OS_RP = 4, OS_TT = 5, OS_ERR = 7, OS_ZQ = 8 };

// Dots of w with the basis vectors V[0..m), kDotChunk vectors per sweep over the rows: each
// thread keeps one grid-stride partial sum per vector (in row order), each block reduces them
// vector by vector, and the last block to finish sums the block partials in block order.
constexpr int kDotChunk = 8;

// partial sums of a[0..M) over the block into partials[(c0 + i) gridDim.x + block], i < M
template <int M>
__device__ __forceinline__ void mdot_block_sum(double (&a)[M], int c0, double *partials) {
    constexpr int P = M > 4 ? 8 : M > 2 ? 4 : M;
    __shared__ double part[8][kRedThreads / 32];
    const int lane = threadIdx.x & 31, w = threadIdx.x >> 5;
    double k[P];
#pragma unroll
    for (int i = 0; i < P; i++) k[i] = i < M ? a[i < M ? i : 0] : 0.0;
    const double y = warp_sums<P>(k);
    const int v = lane / (32 / P);  // the value this lane ends with
    if ((lane & (32 / P - 1)) == 0 && v < M) part[v][w] = y;
    __syncthreads();
    if (w < M) {  // a warp per value
        double y = lane < kRedThreads / 32 ? part[w][lane] : 0.0;
#pragma unroll
        for (int o = kRedThreads / 64; o > 0; o >>= 1) y += __shfl_down_sync(0xffffffffu, y, o);
        if (lane == 0) partials[(size_t)(c0 + w) * gridDim.x + blockIdx.x] = y;
    }
    __syncthreads();  // `part` is reused by the next chunk
}

// dots of w with V[c0 .. c0 + M). M is exact: an FP64 instruction that is predicated off takes
// its 64 cycles all the same, and these kernels are bound by the FP64 pipe (2.0M rows, one
// vector: 35 us with eight predicated products per row, 10 with one; eight vectors: 37)
template <int M>
__device__ __forceinline__ void mdot_exact(int n, const double *__restrict__ w,
                                           double *const *__restrict__ V, int c0, double *partials) {
    const double *vp[M];
    double a[M];
#pragma unroll
    for (int i = 0; i < M; i++) {
        vp[i] = V[c0 + i];
        a[i] = 0.0;
    }
    for (int k = blockIdx.x * blockDim.x + threadIdx.x; k < n; k += gridDim.x * blockDim.x) {
        const double wk = w[k];
#pragma unroll
        for (int i = 0; i < M; i++) a[i] += wk * vp[i][k];
    }
    mdot_block_sum<M>(a, c0, partials);
}
__device__ __forceinline__ void mdot_chunk(int n, const double *__restrict__ w,
                                           double *const *__restrict__ V, int c0, int mc,
                                           double *partials) {
    switch (mc) {
        case 1: mdot_exact<1>(n, w, V, c0, partials); break;
        case 2: mdot_exact<2>(n, w, V, c0, partials); break;
        case 3: mdot_exact<3>(n, w, V, c0, partials); break;
        case 4: mdot_exact<4>(n, w, V, c0, partials); break;
        case 5: mdot_exact<5>(n, w, V, c0, partials); break;
        case 6: mdot_exact<6>(n, w, V, c0, partials); break;
        case 7: mdot_exact<7>(n, w, V, c0, partials); break;
        default: mdot_exact<8>(n, w, V, c0, partials); break;
    }
}

// x - sum_{i < m} c[i] V[i][k], in order; four vectors' loads at a time
__device__ __forceinline__ double minus_combination(double x, int k, double *const *__restrict__ V, int m,
                                                    const double *__restrict__ c) {
    int i = 0;
    for (; i + 4 <= m; i += 4) {
        const double v0 = V[i][k], v1 = V[i + 1][k], v2 = V[i + 2][k], v3 = V[i + 3][k];
        x -= c[i] * v0;
        x -= c[i + 1] * v1;
        x -= c[i + 2] * v2;
        x -= c[i + 3] * v3;
    }
    for (; i < m; i++) x -= c[i] * V[i][k];
    return x;
}

__device__ __forceinline__ void mdot_finish(int m, double *out, const RedCtx &rc) {
    __shared__ bool last;
    if (threadIdx.x == 0) {
        __threadfence();
        unsigned t = atomicAdd(rc.counter, 1u);
        last = (t == gridDim.x - 1);
    }
    __syncthreads();
    if (!last) return;
    __threadfence();
    // vector i by warp i mod (warps): each sum in the same order as one warp summing them all
    const int lane = threadIdx.x & 31, wid = threadIdx.x >> 5, nw = blockDim.x >> 5;
    for (int i = wid; i < m; i += nw) {
        double y = 0.0;
        for (int b = lane; b < (int)gridDim.x; b += 32)
            y += __ldcg(&rc.partials[(size_t)i * gridDim.x + b]);
        y = warp_sum(y);
        if (lane == 0) out[i] = y;
    }
    __syncthreads();  // every warp's partial reads before the counter is re-armed
    if (threadIdx.x == 0) *rc.counter = 0u;
}

// (z, q_j) for all j < it: each block loops over j; the last block reduces every j
__global__ void __launch_bounds__(kRedThreads, 4)
    k_outer_multidot(int n, const double *__restrict__ z, double *const *__restrict__ Q,
                     int it, double *osc, RedCtx rc) {
    follow(z, Q, osc);
    for (int c0 = 0; c0 < it; c0 += kDotChunk)
        mdot_chunk(n, z, Q, c0, min(kDotChunk, it - c0), rc.partials);
    mdot_finish(it, osc + OS_ZQ, rc);
}

// p_it = z - sum_j (z, q_j) / (p_j, q_j) p_j   (Alg. 1 step 2 on the finest level)
// The coefficients are divided once per block (FP64 division is a long instruction sequence
// on this GPU), the same values as dividing per row.
constexpr int kOrthCoef = 256;

__global__ void k_outer_orth(int n, const double *__restrict__ z, double *const *__restrict__ P,
                             int it, const double *__restrict__ osc,
                             const double *__restrict__ opq) {
    __shared__ double cf[kOrthCoef];
    follow(z, P, osc, opq);
    for (int j = threadIdx.x; j < it && j < kOrthCoef; j += blockDim.x)
        cf[j] = -osc[OS_ZQ + j] / opq[j];
    __syncthreads();
    double *p = P[it];
    for (int i = blockIdx.x * blockDim.x + threadIdx.x; i < n; i += gridDim.x * blockDim.x) {
        double acc = z[i];
        int j = 0;
        for (; j + 4 <= it && j + 4 <= kOrthCoef; j += 4) {  // four vectors' loads at a time
            const double v0 = P[j][i], v1 = P[j + 1][i], v2 = P[j + 2][i], v3 = P[j + 3][i];
            acc += cf[j] * v0;
            acc += cf[j + 1] * v1;
            acc += cf[j + 2] * v2;
            acc += cf[j + 3] * v3;
        }
        for (; j < it; j++)
            acc += (j < kOrthCoef ? cf[j] : -osc[OS_ZQ + j] / opq[j]) * P[j][i];
        p[i] = acc;
    }
}

// q = A p, (p, q) -> opq[it], (r, p) -> osc[RP]
__global__ void __launch_bounds__(kRedThreads) k_outer_spmv_dot(GLev<double> L,
                                                                double *const *__restrict__ P,
                                                                double *const *__restrict__ Q,
                                                                int it,
                                                                const double *__restrict__ r,
                                                                double *osc, double *opq,
                                                                RedCtx rc) {
    follow(P, Q, r, osc, opq);
    const double *p = P[it];
    double *q = Q[it];
    double v[2] = {0.0, 0.0};
    for (int row = blockIdx.x * blockDim.x + threadIdx.x; row < L.n; row += gridDim.x * blockDim.x) {
        int base, width;
        row_span(L, row, base, width);  // computed, not loaded, for uniform slices
        const double acc = row_dot(L, base, 0, width, p);
        q[row] = acc;
        v[0] += p[row] * acc;
        v[1] += r[row] * p[row];
    }
    double *out[2] = {&opq[it], &osc[OS_RP]};
    reduce_store<2, RM_LASTBLOCK, double>(v, out, rc, 0, BlockGroup{});
}

// alpha = (r, p) / (p, Ap); x += alpha p; r -= alpha q; (r, r)
__global__ void __launch_bounds__(kRedThreads) k_outer_update(int n, double *const *__restrict__ P,
                                                              double *const *__restrict__ Q,
                                                              int it, double *__restrict__ x,
                                                              double *__restrict__ r, double *osc,
                                                              const double *__restrict__ opq,
                                                              const int *err, RedCtx rc) {
    follow(P, Q, x, r, osc, opq);
    const double pq = opq[it];
    const bool bad = !(pq > 0.0) || !isfinite(pq);
    __shared__ double alpha_s;  // one FP64 division per block, not per thread
    if (threadIdx.x == 0) alpha_s = bad ? 0.0 : osc[OS_RP] / pq;
    __syncthreads();
    const double alpha = alpha_s;
    const double *p = P[it];
    const double *q = Q[it];
    double v[1] = {0.0};
    for (int i = blockIdx.x * blockDim.x + threadIdx.x; i < n; i += gridDim.x * blockDim.x) {
        x[i] += alpha * p[i];
        double rn = r[i] - alpha * q[i];
        r[i] = rn;
        v[0] += rn * rn;
    }
    double *out[1] = {&osc[OS_RR]};
    reduce_store<1, RM_LASTBLOCK, double>(v, out, rc, 0, BlockGroup{});
    if (blockIdx.x == 0 && threadIdx.x == 0) {
        if (bad) osc[OS_STOP] = 1.0;
        osc[OS_ERR] = (double)*err;
    }
}

// ---------------------------------------------------------------------------------------
// FGMRES kernels (FP64, pi order); V and Z are arrays of vector pointers
// w = A z
__global__ void k_spmv(GLev<double> L, const double *__restrict__ z, double *__restrict__ w) {
    for (int row = blockIdx.x * blockDim.x + threadIdx.x; row < L.n; row += gridDim.x * blockDim.x) {
        int base, width;
        row_span(L, row, base, width);
        w[row] = row_dot(L, base, 0, width, z);
    }
}

// out[i] = (w, V[i]) for i < m
__global__ void __launch_bounds__(kRedThreads, 4) k_mdot(int n, const double *__restrict__ w,
                                                      double *const *__restrict__ V, int m,
                                                      double *out, RedCtx rc) {
    for (int c0 = 0; c0 < m; c0 += kDotChunk)
        mdot_chunk(n, w, V, c0, min(kDotChunk, m - c0), rc.partials);
    mdot_finish(m, out, rc);
}

// The second Gram-Schmidt pass's dots fused with the first pass's subtraction (both are
// row-local): w -= sum_i c[i] V[i], then out[i] = (w, V[i]) for i < m. Each row's new w is
// written by the thread that reads it again in the later chunks.
__global__ void __launch_bounds__(kRedThreads, 4) k_orth_mdot(int n, double *__restrict__ w,
                                                           double *const *__restrict__ V, int m,
                                                           const double *__restrict__ c,
                                                           double *out, RedCtx rc) {
    for (int k = blockIdx.x * blockDim.x + threadIdx.x; k < n; k += gridDim.x * blockDim.x) {
        w[k] = minus_combination(w[k], k, V, m, c);
    }
    for (int c0 = 0; c0 < m; c0 += kDotChunk)
        mdot_chunk(n, w, V, c0, min(kDotChunk, m - c0), rc.partials);
    mdot_finish(m, out, rc);
}

// w -= sum_i c[i] V[i]; (w, w) -> *nrm2
__global__ void __launch_bounds__(kRedThreads) k_orth_sub(int n, double *__restrict__ w,
                                                          double *const *__restrict__ V, int m,
                                                          const double *__restrict__ c,
                                                          double *nrm2, const int *err,
                                                          double *err_out, RedCtx rc) {
    double a[1] = {0.0};
    for (int k = blockIdx.x * blockDim.x + threadIdx.x; k < n; k += gridDim.x * blockDim.x) {
        const double x = minus_combination(w[k], k, V, m, c);
        w[k] = x;
        a[0] += x * x;
    }
    double *o[1] = {nrm2};
    reduce_store<1, RM_LASTBLOCK, double>(a, o, rc, 0, BlockGroup{});
    if (blockIdx.x == 0 && threadIdx.x == 0) *err_out = (double)*err;
}

// v = w * s
__global__ void k_scale(int n, const double *__restrict__ w, double s, double *__restrict__ v) {
    for (int k = blockIdx.x * blockDim.x + threadIdx.x; k < n; k += gridDim.x * blockDim.x) v[k] = w[k] * s;
}

// x += sum_j y[j] Z[j]
__global__ void k_lincomb(int n, double *__restrict__ x, double *const *__restrict__ Z, int m,
                          const double *__restrict__ y) {
    for (int k = blockIdx.x * blockDim.x + threadIdx.x; k < n; k += gridDim.x * blockDim.x) {
        double acc = x[k];
        for (int j = 0; j < m; j++) acc += y[j] * Z[j][k];
        x[k] = acc;
    }
}

// =======================================================================================
// diagnostics: per-kernel timing and algorithmic bytes
thread_local int64_t g_launches = 0;

enum : int { K_CYCLE = OP_NKINDS, K_OUTER_MULTIDOT, K_OUTER_ORTH, K_OUTER_SPMV_DOT, K_OUTER_UPDATE,
             K_TRUE_RESIDUAL, K_FGMRES_SPMV, K_FGMRES_MDOT, K_FGMRES_ORTH, K_NUM };
constexpr int K_IN_CYCLE = 100;  // + op kind: an op timed inside the persistent kernel
constexpr int K_IN_TAIL = 200;   // + op kind: an op timed inside the cluster (CTA 0's clock)

const char *kernel_name(int kind) {
    static const char *names[K_NUM] = {"zero", "gs_colour", "resid_restrict", "prolong_correct",
                                       "coarse_solve", "alg1_multidot", "alg1_orth",
                                       "alg1_spmv_dot", "alg1_update", "tail_cta", "barrier_only",
                                       "gs_first_colour", "residual", "restrict_gather",
                                       "cycle_persistent", "outer_multidot", "outer_orth",
                                       "outer_spmv_dot", "outer_update", "true_residual",
                                       "fgmres_spmv", "fgmres_mdot", "fgmres_orth_sub"};
    static const char *incycle[OP_NKINDS] = {"in_cycle:zero", "in_cycle:gs_colour",
                                             "in_cycle:resid_restrict", "in_cycle:prolong_correct",
                                             "in_cycle:coarse_solve", "in_cycle:alg1_multidot",
                                             "in_cycle:alg1_orth", "in_cycle:alg1_spmv_dot",
                                             "in_cycle:alg1_update", "in_cycle:tail_cta",
                                             "in_cycle:barrier_only", "in_cycle:gs_first_colour",
                                             "in_cycle:residual", "in_cycle:restrict_gather"};
    static const char *intail[OP_NKINDS] = {"in_tail:zero", "in_tail:gs_colour",
                                            "in_tail:resid_restrict", "in_tail:prolong_correct",
                                            "in_tail:coarse_solve", "in_tail:alg1_multidot",
                                            "in_tail:alg1_orth", "in_tail:alg1_spmv_dot",
                                            "in_tail:alg1_update", "in_tail:?", "in_tail:?",
                                            "in_tail:gs_first_colour", "in_tail:residual",
                                            "in_tail:restrict_gather"};
    if (kind >= K_IN_CYCLE && kind < K_IN_CYCLE + OP_NKINDS) return incycle[kind - K_IN_CYCLE];
    if (kind >= K_IN_TAIL && kind < K_IN_TAIL + OP_NKINDS) return intail[kind - K_IN_TAIL];
    return (kind >= 0 && kind < K_NUM) ? names[kind] : "unknown";
}

struct Profiler {
    struct Rec {
        int kind, level;
        double bytes;
        cudaEvent_t a, b;
    };
    bool on = false;
    bool tail_ops = false;  // also time every step inside the cluster
    std::vector<Rec> pending;
    struct Acc {
        int64_t launches = 0;
        double ms = 0, bytes = 0;
    };
    std::vector<std::pair<std::pair<int, int>, Acc>> acc;

    Acc &slot(int kind, int level) {
        for (auto &e : acc)
            if (e.first.first == kind && e.first.second == level) return e.second;
        acc.push_back({{kind, level}, Acc()});
        return acc.back().second;
    }
    void add(int kind, int level, double ms, double bytes, int64_t launches = 1) {
        Acc &a = slot(kind, level);
        a.launches += launches;
        a.ms += ms;
        a.bytes += bytes;
    }
    Rec begin(int kind, int level, double bytes, cudaStream_t s) {
        Rec r{kind, level, bytes, nullptr, nullptr};
        AMG_CUDA(cudaEventCreate(&r.a));
        AMG_CUDA(cudaEventCreate(&r.b));
        AMG_CUDA(cudaEventRecord(r.a, s));
        return r;
    }
    void end(Rec &r, cudaStream_t s) {
        AMG_CUDA(cudaEventRecord(r.b, s));
        pending.push_back(r);
    }
    void harvest() {
        for (auto &r : pending) {
            float ms = 0.f;
            if (cudaEventElapsedTime(&ms, r.a, r.b) == cudaSuccess) add(r.kind, r.level, ms, r.bytes);
            else cudaGetLastError();
            cudaEventDestroy(r.a);
            cudaEventDestroy(r.b);
        }
        pending.clear();
    }
    ~Profiler() {
        for (auto &r : pending) {
            cudaEventDestroy(r.a);
            cudaEventDestroy(r.b);
        }
    }
};

void profiler_enable(amg_hierarchy *h, int mode) {
    if (!h->prof) h->prof = new Profiler();
    h->prof->on = mode != 0;
    h->prof->tail_ops = mode == 1;
    h->prof->acc.clear();
}

void profiler_free(amg_hierarchy *h) {
    delete h->prof;
    h->prof = nullptr;
}

int profiler_read(const amg_hierarchy *h, int cap, int32_t *kind, int32_t *level,
                  int64_t *launches, double *ms, double *bytes) {
    if (!h->prof) return 0;
    int k = 0;
    for (auto &e : h->prof->acc) {
        if (k >= cap) break;
        if (kind) kind[k] = e.first.first;
        if (level) level[k] = e.first.second;
        if (launches) launches[k] = e.second.launches;
        if (ms) ms[k] = e.second.ms;
        if (bytes) bytes[k] = e.second.bytes;
        k++;
    }
    return (int)h->prof->acc.size();
}

static bool profiling(const amg_hierarchy *h) { return h->prof && h->prof->on; }

// algorithmic bytes of one op: every array the op must touch, once, at its width
// (w = value width, 4-byte column indices; padding of the sliced ELL is not counted)
static double op_bytes(const amg_hierarchy *h, const Op &op, int w) {
    const Level &lv = h->lev[op.level];
    const double n = lv.n, nnz = (double)lv.A.stored;
    const double nn = op.level + 1 < h->nlev ? h->lev[op.level + 1].n : 0;
    switch (op.kind) {
        case OP_ZERO: return w * n;
        case OP_GS_FIRST: return w * n + 2.0 * w * (op.i1 - op.i0);
        case OP_GS: {
            const std::vector<int> &ranges = op.level == 0 ? lv.color_blocks : lv.color_rows;
            int c = 0;
            while (c + 1 < (int)ranges.size() && ranges[c] != op.i0) c++;
            double rows = lv.color_rows[c + 1] - lv.color_rows[c];
            double e = c < (int)lv.color_nnz.size() ? (double)lv.color_nnz[c] : 0;
            double blocks = op.i1 - op.i0;
            return e * (4 + w) + rows * 3.0 * w + (op.level == 0 ? 4.0 * blocks : 0.0);
        }
        case OP_RESTRICT:
            return nnz * (4 + w) + 2.0 * w * n + w * nn + (op.level == 0 ? 4.0 * nn : 16.0 * nn);
        // the two passes of a split restriction: the restriction's bytes, shared out (the
        // intermediate residual vector is the split's own traffic, not the method's)
        case OP_RESID: return nnz * (4 + w) + 2.0 * w * n;
        case OP_GATHER: return w * nn + 16.0 * nn;
        case OP_PROLONG: return 2.0 * w * n + 4.0 * n + w * nn;
        case OP_COARSE: return w * n * n + 2.0 * w * n;
        case OP_MULTIDOT: return w * n * (1 + op.step);
        case OP_ORTH: return w * n * (2 + op.step);
        case OP_SPMV_DOT: return nnz * (4 + w) + 3.0 * w * n;
        case OP_UPDATE: return (op.step == 0 ? 2.0 : 3.0) * w * n + (op.last ? 0.0 : 3.0 * w * n);
    }
    return 0;
}

// =======================================================================================
// host side
struct EngineBase {
    Op *prog = nullptr;
    int nops = 0;
    int grid = 0;
    size_t smem = 0;   // of the cycle kernel (big blocks)
    int form = 0;  // the cycle kernel's instance (kCoop, kBig)
    int big_smem = 0;  // the CTAs sweep the big blocks in their shared memory
    int big_wwarps = 0;  // warps of a CTA with a slice for the warp-sized blocks
    unsigned big_wslice = 0;
    ClLayout cl{};                   // the cluster's levels (cl.tl = nlev: none)
    unsigned char *cl_image = nullptr;
    std::vector<Op> hprog, htail;
    double tail_bytes = 0, cycle_bytes = 0;
    unsigned long long *ts = nullptr;
    unsigned long long *tprof = nullptr;
};

namespace {

template <class T>
Vecs<T> &vecs(Level &lv);
template <>
Vecs<double> &vecs<double>(Level &lv) { return lv.v64; }
template <>
Vecs<float> &vecs<float>(Level &lv) { return lv.v32; }

int red_grid(int64_t n) {
    return (int)std::min<int64_t>(kRedBlocks, std::max<int64_t>(1, (n + kRedThreads - 1) / kRedThreads));
}

size_t align16(size_t b) { return (b + 15) & ~(size_t)15; }


// finest-level blocks of six or more rows on average (the octree's 2x2x2-node aggregates):
// the lane-parallel block smoother (op_gs_blocks_coop) and restriction. Smaller blocks (a few
// rows, as on a quadtree with several nodes per cell) keep one thread per block: with
// kBlockLanes lanes each, most lanes would idle and the sweep would need more passes.
bool coop_blocks(const Level &lv) {
    return lv.nblocks > 0 && 6 * (int64_t)lv.nblocks <= (int64_t)lv.n;
}

bool is_reduction(const Op &op) {
    return op.kind == OP_MULTIDOT || op.kind == OP_SPMV_DOT || (op.kind == OP_UPDATE && !op.last);
}

// Walks Alg. 2 / Alg. 1 from a level and appends the ops to a program. The recursion stops
// at `stop_level`, where one OP_TAIL stands for B~ of that level (the cycle's program), or
// continues to the coarsest level (traffic accounting, standalone execution).
struct Builder {
    amg_hierarchy *h;
    std::vector<Op> *out;
    int stop_level;  // >= nlev: never stop

    static Op mk(int kind, int level) {
        Op o;
        std::memset(&o, 0, sizeof o);
        o.kind = kind;
        o.level = level;
        o.red_pb = -1;
        o.fin_pb = -1;
        for (int k = 0; k < 4; k++) o.fin_dst[k] = -1;
        return o;
    }
    void emit(const Op &o) { out->push_back(o); }

    // first non-empty colour of level l (its point-GS first colour), [r0, r1)
    void first_colour(int l, int &r0, int &r1) const {
        const std::vector<int> &ranges = h->lev[l].color_rows;
        const int nc = (int)ranges.size() - 1;
        int c0 = 0;
        while (c0 < nc && ranges[c0 + 1] == ranges[c0]) c0++;
        r0 = c0 < nc ? ranges[c0] : 0;
        r1 = c0 < nc ? ranges[c0 + 1] : 0;
    }
    // does B~_l start with the point-GS first colour of B^_l (step 0) in this program?
    bool starts_with_first_colour(int l) const {
        return l >= 1 && l < h->nlev && l != stop_level && !h->lev[l].coarsest;
    }

    // the big blocks of colour c on the finest level go to whole CTAs (grid-wide programs)
    void big_range(int l, int c, Op &g) const {
        const Level &lv = h->lev[l];
        if (l != 0 || lv.nbig == 0) return;
        g.bb0 = lv.color_big[c];
        g.bbc = lv.color_bigc[c];
        g.bb1 = lv.color_big[c + 1];
    }

    // z = B^_l [f] (Alg. 2). first_done: the first colour of the pre-smoothing was already
    // done by the op before (a fused RESTRICT or UPDATE)
    void bhat(int l, int fsel, int zsel, bool first_done = false) {
        Level &lv = h->lev[l];
        const std::vector<int> &ranges = (l == 0) ? lv.color_blocks : lv.color_rows;
        const int nc = (int)ranges.size() - 1;
        int c0 = 0;  // pre-smoothing u1 = R_k f from zero, colours ascending
        if (l == 0) {
            Op z = mk(OP_ZERO, l);
            z.usel = zsel;
            emit(z);
        } else {  // first non-empty colour fused with the zero fill (point smoother)
            while (c0 < nc && ranges[c0 + 1] == ranges[c0]) c0++;
            if (!first_done) {
                Op g = mk(OP_GS_FIRST, l);
                g.i0 = c0 < nc ? ranges[c0] : 0;
                g.i1 = c0 < nc ? ranges[c0 + 1] : 0;
                g.fsel = fsel;
                g.usel = zsel;
                emit(g);
            }
            c0++;
        }
        // the first sweep's remaining colours, then nu_pre - 1 further forward sweeps
        for (int sw = 0; sw < h->opt.nu_pre; sw++)
            for (int c = sw == 0 ? c0 : 0; c < nc; c++) {
                if (ranges[c + 1] == ranges[c]) continue;
                Op g = mk(OP_GS, l);
                g.i0 = ranges[c];
                g.i1 = ranges[c + 1];
                g.fsel = fsel;
                g.usel = zsel;
                big_range(l, c, g);
                emit(g);
            }
        Op rs = mk(OP_RESTRICT, l);  // next.rhs = P^t (f - A u1)
        rs.fsel = fsel;
        rs.usel = zsel;
        if (l == 0 && lv.nbig > 0) rs.bb1 = lv.nbig;  // every big block, by whole CTAs
        const bool fuse = starts_with_first_colour(l + 1);
        if (fuse) {  // and the next level's first colour from zero
            rs.fuse = 1;
            first_colour(l + 1, rs.f0, rs.f1);
        }
        if (l >= 1 && lv.n >= kSplitRestrictRows) {
            // a large coarse level: the residual row by row into q_step, then the children
            // sums (coalesced slots instead of a gather over four colours' rows)
            Op rr = mk(OP_RESID, l);
            rr.fsel = fsel;
            rr.usel = zsel;
            rr.step = zsel - V_P0;
            emit(rr);
            rs.kind = OP_GATHER;
            rs.step = zsel - V_P0;
        }
        emit(rs);
        btilde(l + 1, fuse);         // next.e = B~_{k-1}[next.rhs]
        Op pr = mk(OP_PROLONG, l);   // u2 = u1 + P e
        pr.usel = zsel;
        emit(pr);
        for (int sw = 0; sw < h->opt.nu_post; sw++)  // post-smoothing: colours descending
            for (int c = nc - 1; c >= 0; c--) {
                if (ranges[c + 1] == ranges[c]) continue;
                Op g = mk(OP_GS, l);
                g.i0 = ranges[c];
                g.i1 = ranges[c + 1];
                g.backward = 1;
                g.fsel = fsel;
                g.usel = zsel;
                big_range(l, c, g);
                emit(g);
            }
    }

    // e = B~_l [rhs] (Alg. 1 with kcycle_n steps; exact on the coarsest level). first_done:
    // step 0's first colour was done by the restriction into this level
    void btilde(int l, bool first_done = false) {
        if (l == stop_level) {
            emit(mk(OP_TAIL, l));
            return;
        }
        Level &lv = h->lev[l];
        if (lv.coarsest) {
            emit(mk(OP_COARSE, l));
            return;
        }
        const int n = h->opt.kcycle_n;
        for (int i = 0; i < n; i++) {
            bhat(l, i == 0 ? V_RHS : V_R, V_P0 + i, i == 0 ? first_done : true);
            if (i > 0) {
                Op md = mk(OP_MULTIDOT, l);
                md.step = i;
                emit(md);
                Op ot = mk(OP_ORTH, l);
                ot.step = i;
                emit(ot);
            }
            Op sd = mk(OP_SPMV_DOT, l);
            sd.step = i;
            emit(sd);
            Op up = mk(OP_UPDATE, l);
            up.step = i;
            up.last = (i == n - 1);
            if (!up.last) {  // and the next step's first colour from zero, on r_{i+1}
                up.fuse = 1;
                first_colour(l, up.f0, up.f1);
            }
            emit(up);
        }
    }
};

// persistent program: reductions leave partials in alternating buffers; the next op sums
// them into the level's scalars
void annotate_reductions(std::vector<Op> &prog) {
    std::vector<Op> out;
    int pb = 0;
    bool pending = false;
    Op pend{};
    auto attach = [&](Op &op) {
        op.fin_pb = pend.red_pb;
        op.fin_level = pend.level;
        if (pend.kind == OP_MULTIDOT) {
            op.fin_n = pend.step;
            for (int j = 0; j < pend.step; j++) op.fin_dst[j] = SC_ZQ0 + j;
        } else if (pend.kind == OP_SPMV_DOT) {
            op.fin_n = 2;
            op.fin_dst[0] = SC_PQ0 + pend.step;
            op.fin_dst[1] = SC_RP0 + pend.step;
        } else {
            op.fin_n = 1;
            op.fin_dst[0] = SC_RR0 + pend.step;
        }
    };
    for (Op op : prog) {
        if (pending) {
            attach(op);
            pending = false;
        }
        if (is_reduction(op)) {
            op.red_pb = pb;
            pb ^= 1;
            pending = true;
            pend = op;
        }
        out.push_back(op);
    }
    if (pending) {
        Op nop = Builder::mk(OP_NOP, pend.level);
        attach(nop);
        out.push_back(nop);
    }
    prog.swap(out);
}

template <class T>
void table_image(amg_hierarchy *h, std::vector<GLev<T>> &tab) {
    tab.assign(h->nlev, GLev<T>());
    for (int l = 0; l < h->nlev; l++) {
        Level &lv = h->lev[l];
        GLev<T> &d = tab[l];
        std::memset(&d, 0, sizeof d);
        d.n = lv.n;
        d.fine = (l == 0) ? 1 : 0;
        // blocks of several rows (octree aggregates): a lane per row (op_gs_blocks_coop)
        d.bg = (l == 0 && coop_blocks(lv)) ? kBlockLanes : 0;
        d.w = lv.A.uw;
        d.sl = lv.A.sl_ptr;
        d.col = lv.A.col;
        if constexpr (sizeof(T) == 8) d.val = (const T *)lv.A.val;
        else d.val = (const T *)lv.A.val32;
        if constexpr (sizeof(T) == 8) d.dinv = (const T *)lv.dinv64;
        else d.dinv = (const T *)lv.dinv32;
        d.bptr = lv.bptr;
        d.big = (l == 0) ? lv.big_dev : nullptr;
        d.parent = lv.parent;
        d.children = (l + 1 < h->nlev) ? h->lev[l + 1].children : nullptr;
        d.children2 = (l + 1 < h->nlev) ? h->lev[l + 1].children2 : nullptr;
        d.Ainv = lv.Ainv;
        d.Ainv2 = lv.Ainv32;
        Vecs<T> &v = vecs<T>(lv);
        d.rhs = v.rhs;
        d.e = v.e;
        d.r = v.r;
        for (int i = 0; i < kMaxKcycle; i++) {
            d.p[i] = v.p[i];
            d.q[i] = v.q[i];
        }
        d.sc = lv.sc;
        d.nnext = (l + 1 < h->nlev) ? h->lev[l + 1].n : 0;
    }
}

template <class T>
void fill_tables(amg_hierarchy *h) {
    std::vector<GLev<T>> tab;
    table_image<T>(h, tab);
    void *&dst = (sizeof(T) == 8) ? h->lev_tab64 : h->lev_tab32;
    if (!dst) dst = halloc<GLev<T>>(h, h->nlev);
    AMG_CUDA(cudaMemcpyAsync(dst, tab.data(), sizeof(GLev<T>) * h->nlev, cudaMemcpyHostToDevice,
                             h->stream));
}

template <class T>
const GLev<T> *dtab(amg_hierarchy *h) {
    return (const GLev<T> *)((sizeof(T) == 8) ? h->lev_tab64 : h->lev_tab32);
}

// widest slice (slots per row) of each level, from its slice pointers
std::vector<int> slice_widths(amg_hierarchy *h) {
    std::vector<int> w(h->nlev, 0);
    std::vector<std::vector<int>> sl(h->nlev);
    bool read = false;
    for (int l = 0; l < h->nlev; l++) {
        const Sell &A = h->lev[l].A;
        if (A.uw > 0) {  // one width, known here
            w[l] = A.uw;
            continue;
        }
        sl[l].resize(A.nslices + 1);
        AMG_CUDA(cudaMemcpyAsync(sl[l].data(), A.sl_ptr, sizeof(int) * sl[l].size(),
                                 cudaMemcpyDeviceToHost, h->stream));
        read = true;
    }
    if (read) AMG_CUDA(cudaStreamSynchronize(h->stream));
    for (int l = 0; l < h->nlev; l++)
        for (size_t k = 0; k + 1 < sl[l].size(); k++)
            w[l] = std::max(w[l], (sl[l][k + 1] - sl[l][k]) / kSliceH);
    return w;
}

template <class T>
EngineBase *&engine_slot(amg_hierarchy *h) {
    return (sizeof(T) == 8) ? h->eng64 : h->eng32;
}

template <class T>
void *cycle_kernel(int B) {
    switch (B) {
        case 0: return (void *)k_cycle<T, 0>;
        case kCoop: return (void *)k_cycle<T, kCoop>;
        case kBig: return (void *)k_cycle<T, kBig>;
        default: return (void *)k_cycle<T, kCoop | kBig>;
    }
}

// ---------------------------------------------------------------------------------------
// the cluster's levels (cluster_tail.cuh)

// one candidate: swept levels [tl, tl + nsp), the dense level after them
struct ClPlan {
    ClLayout y;
    std::vector<ClColor> geo;           // the strips of every swept level
    std::vector<unsigned char> tables;  // [kClRanks][table_bytes]: the head of every image
    int table_bytes = 0;
};

// strip r's rows of colour c (the finest level: of its blocks, hb = their first rows)
int2 cl_own_rows(const ClSrc &S, const std::vector<int> &hb, int r, int c) {
    const ClSrc &B = S.bptr ? (&S)[1] : S;  // the next level: its rows are the blocks
    const int len = B.cr[c + 1] - B.cr[c];
    const int a = B.cr[c] + cl_part(len, r), b = B.cr[c] + cl_part(len, r + 1);
    return S.bptr ? make_int2(hb[a], hb[b]) : make_int2(a, b);
}

// Layout and tables for the swept levels G.lv[s0 ..] (hierarchy levels level0 ..) and the dense
// level after them, or false if they do not fit `budget` bytes of shared memory. win: their
// windows; xchild: [2][nlv], by the next level's kind (swept, dense); fo: owner of each row of
// the dense level; sparse: M alone and the sparse A after it.
template <class T>
bool cluster_plan(const ClSrcs &G, const std::vector<int2> &win, const std::vector<int> &xchild, int nlv,
                  const int *fo, const std::vector<int> &hb, const std::vector<int> &widths, int s0, int level0,
                  bool dense, bool sparse, int nch, const amg_options &opt, long budget, ClPlan &P) {
    constexpr int vb = (int)sizeof(T), NR = kClRanks;
    ClLayout &y = P.y;
    std::memset(&y, 0, sizeof y);
    y.nsp = G.nsp - s0;
    y.tl = level0;
    y.dense = dense;
    y.kc = opt.kcycle_n;
    y.nu_pre = opt.nu_pre;
    y.nu_post = opt.nu_post;
    const ClSrc &D = G.lv[G.nsp];
    y.nd = D.n;
    y.ch = (((D.n + NR - 1) / NR) + 3) & ~3;
    y.stride = NR * y.ch;
    auto win_of = [&](int a, int r, int c) {
        return win[cl_win(s0 + a, r, c)];
    };
    auto own_of = [&](const ClSrc &S, int r, int c) { return cl_own_rows(S, hb, r, c); };
    // the strips: windows, bytes exchanged, neighbours
    P.geo.assign((size_t)std::max(1, y.nsp) * NR * kClColors, ClColor{});
    auto geo = [&](int a, int r, int c) -> ClColor & { return P.geo[cl_win(a, r, c)]; };
    std::vector<std::vector<ClHead>> head(y.nsp, std::vector<ClHead>(NR));
    std::vector<std::vector<std::vector<int>>> expect(y.nsp);
    std::vector<int> c_first(y.nsp, 0);
    std::vector<std::vector<int>> peers(NR);
    std::vector<std::vector<char>> is_peer(NR, std::vector<char>(NR, 0));
    std::vector<size_t> max_own(y.nsp + 1, 1), max_win(y.nsp, 1), over(y.nsp, 0);
    for (int a = 0; a < y.nsp; a++) {
        const ClSrc &S = G.lv[s0 + a];
        ClLev &L = y.lv[a];
        L.level = level0 + a;
        L.ncol = S.ncol;
        L.w = std::max(1, widths[level0 + a]);
        // Lanes per row: as few as take its slots, eight each. FP64: one instruction of a warp
        // takes 64 cycles, of each of nw warps at once 19 nw (measured, whatever the lanes do),
        // so rows are split further where their warps still run side by side: the sum over a
        // step's colours (the largest one's rows) and its two products with all own rows
        L.lg = -1;
        double best = 0;
        int rows = 1, all = 0, colours = 0;
        for (int c = 0; c < S.ncol; c++) {
            const int len = (S.cr[c + 1] - S.cr[c] + NR - 1) / NR;
            rows = std::max(rows, len);
            all += len;
            colours += S.cr[c + 1] > S.cr[c] ? 2 : 0;
        }
        for (int lg = 0; lg <= 2; lg++) {
            int ns = 2;  // 2, 4 or 8
            while (ns << lg < L.w - 1 && ns <= kClSlots) ns *= 2;
            if (ns > kClSlots) continue;
            auto fp64 = [&](int r, int instr) {
                const int t = r << lg, full = t / kClThreads, rest = (t % kClThreads + 31) / 32;
                return (full * 19.0 * kClWarps + (rest ? std::max(64, 19 * rest) : 0)) * instr + 70.0 * lg;
            };
            if (S.bptr && lg > 0) continue;  // a block is one lane's
            const double cost = vb == 8 ? colours * fp64(rows, ns + lg + 2) + 2 * fp64(all, ns + lg + 3) : lg;
            if (L.lg >= 0 && cost >= best) continue;
            L.lg = lg;
            L.ns = vb == 8 ? ns : kClSlots;
            best = cost;
        }
        if (L.lg < 0) return false;
        L.nch = nch;
        int cf = -1, cl = 0;
        for (int c = 0; c < S.ncol; c++)
            if (S.cr[c + 1] > S.cr[c]) {
                if (cf < 0) cf = c;
                cl = c;
            }
        cf = std::max(cf, 0);
        for (int r = 0; r < NR; r++) {
            ClHead &h = head[a][r];
            std::memset(&h, 0, sizeof h);
            for (int c = 0; c < S.ncol; c++) {
                const int2 o = own_of(S, r, c), w = win_of(a, r, c);
                ClColor &C = geo(a, r, c);
                C.cnt = o.y - o.x;
                C.m0 = h.nown;
                C.seg0 = h.nwin;
                C.seglen = w.y - w.x;
                C.li0 = h.nwin + o.x - w.x;
                C.g0 = o.x;
                h.nown += C.cnt;
                h.nwin += C.seglen;
            }
            if (h.nwin * vb > 65535) return false;  // 16-bit byte offsets
            h.fc0 = geo(a, r, cf).m0;
            h.fcn = S.bptr ? 0 : geo(a, r, cf).cnt;
            c_first[a] = cf;
            h.fs0 = geo(a, r, cf).seg0;
            h.fs1 = h.fs0 + (S.bptr ? 0 : geo(a, r, cf).seglen);
            h.ls0 = geo(a, r, cl).seg0;
            h.ls1 = h.ls0 + (S.bptr ? 0 : geo(a, r, cl).seglen);
            max_own[a] = std::max(max_own[a], (size_t)h.nown);
            max_win[a] = std::max(max_win[a], (size_t)h.nwin);
        }
        expect[a].assign(NR, std::vector<int>(S.ncol, 0));
        for (int r = 0; r < NR; r++) {
            size_t all = 0;
            for (int c = 0; c < S.ncol; c++) {
                const int2 o = own_of(S, r, c);
                int holders = 0;  // strips that hold some of these rows
                size_t rows = 0;
                for (int d = 0; d < NR; d++) {
                    if (d == r) continue;
                    const int2 w = win_of(a, d, c);
                    const int lo = std::max(o.x, w.x), hi = std::min(o.y, w.y);
                    if (lo >= hi) continue;
                    expect[a][d][c] += (hi - lo) * vb;
                    head[a][d].expect_all += (hi - lo) * vb;
                    is_peer[r][d] = is_peer[d][r] = 1;
                    holders++;
                    rows += hi - lo;
                }
                if (holders > 2) all += rows;  // may need the list of further destinations
            }
            over[a] = std::max(over[a], all);
        }
    }
    for (int r = 0; r < NR; r++)
        for (int d = 0; d < NR; d++)
            if (is_peer[r][d]) peers[r].push_back(d);
    // the dense level's rows, each with its first child
    std::vector<std::vector<unsigned short>> down(NR);
    for (int i = 0; i < D.n && y.nsp > 0; i++) down[fo[i]].push_back((unsigned short)i);
    for (int r = 0; r < NR; r++) max_own[y.nsp] = std::max(max_own[y.nsp], down[r].size());
    for (int a = 0; a < y.nsp; a++)
        for (int r = 0; r < NR; r++) head[a][r].fexp = G.lv[s0 + a].bptr ? 0 : expect[a][r][c_first[a]];
    // the sweeps of every strip: before the restriction (the first colour is done by the step
    // before) and after the correction
    auto lists = [&](int a, int r, std::vector<ClOp> &pre, std::vector<ClOp> &post) {
        const ClLev &L = y.lv[a];
        const ClSrc &S = G.lv[s0 + a];
        pre.clear();
        post.clear();
        auto colour = [&](int c) {
            if (S.bptr) {  // own blocks, numbered colour by colour
                int b0 = 0;
                const ClSrc &B = G.lv[s0 + a + 1];
                auto blocks = [&](int k) {
                    const int len = B.cr[k + 1] - B.cr[k];
                    return cl_part(len, r + 1) - cl_part(len, r);
                };
                for (int k = 0; k < c; k++) b0 += blocks(k);
                return ClOp{b0, blocks(c), expect[a][r][c], 0};
            }
            const ClColor &C = geo(a, r, c);
            return ClOp{C.m0 << L.lg, C.cnt << L.lg, expect[a][r][c], 0};
        };
        for (int sw = 0; sw < y.nu_pre; sw++)
            for (int c = 0; c < S.ncol; c++)
                if (S.cr[c + 1] > S.cr[c] && (sw > 0 || c > c_first[a] || S.bptr)) pre.push_back(colour(c));
        for (int sw = 0; sw < y.nu_post; sw++)
            for (int c = S.ncol - 1; c >= 0; c--)
                if (S.cr[c + 1] > S.cr[c]) post.push_back(colour(c));
    };
    size_t off = 0;
    auto take = [&](size_t bytes) {
        const int o = (int)off;
        off += align16(bytes);
        return o;
    };
    y.dhead = take(sizeof(int));
    y.down = take(sizeof(short) * max_own[y.nsp]);
    y.peers = take(sizeof(int) * (NR + 1));
    y.levels = take(sizeof(ClLev) * y.nsp);
    std::vector<ClOp> pre, post;
    for (int a = 0; a < y.nsp; a++) {
        ClLev &L = y.lv[a];
        lists(a, 0, pre, post);  // the same length in every strip
        L.npre = (int)pre.size();
        L.npost = (int)post.size();
        L.head = take(sizeof(ClHead));
        L.pre = take(sizeof(ClOp) * std::max<size_t>(1, pre.size()));
        L.post = take(sizeof(ClOp) * post.size());
    }
    P.table_bytes = (int)off;
    for (int a = 0; a < y.nsp; a++) {
        ClLev &L = y.lv[a];
        L.R = (int)max_own[a] << L.lg;
        L.nact = std::min(kClWarps, (L.R + 31) / 32);
        L.Rn = (int)max_own[a + 1];
        const bool fine = G.lv[s0 + a].bptr != nullptr;
        L.kind = fine ? 2 : xchild[(a + 1 < y.nsp ? 0 : 1) * nlv + s0 + a];
        L.over = take(sizeof(unsigned) * over[a]);
        L.val = take((size_t)L.ns * L.R * vb);
        L.col = take((size_t)kClSlots * L.R * 2);
        L.diag = take(max_own[a] * vb);
        L.dinv = take(max_own[a] * vb);
        L.own = take(2 * max_own[a]);
        L.dst = take(sizeof(uint4) * max_own[a]);
        L.parent = take(2 * max_win[a]);
        if (fine) L.blk = take(2 * ((size_t)L.Rn + 1));
        else L.child = take(2 * (size_t)nch * L.Rn);
    }
    y.top = take(sizeof(int) * max_own[0]);
    // dense level: FP32 M's high parts and A M (unless the product with A is sparse), M's low parts; FP64
    // M. Without it, the coarsest inverse, in FP32 its two parts
    const size_t rows_bytes = (size_t)y.ch * y.stride * vb;
    y.mat = take((dense && !sparse ? 2 : 1) * rows_bytes);
    if (vb == 4) y.mat_lo = take(rows_bytes);
    size_t beyond = 0;
    if (dense && sparse) {
        y.aw = widths[level0 + y.nsp];
        const size_t val_bytes = align16((size_t)y.aw * y.ch * vb), col_bytes = align16((size_t)y.aw * y.ch * 2);
        if (vb == 4) beyond = val_bytes + col_bytes;
        y.aval = vb == 4 ? (int)off : take(val_bytes);
        y.acol = vb == 4 ? (int)(off + val_bytes) : take(col_bytes);
    }
    y.image_bytes = (int)off;
    y.image_stride = (int)(off + beyond);
    for (int a = 0; a < y.nsp; a++) {
        ClLev &L = y.lv[a];
        const size_t b = max_win[a] * vb;
        const bool fine = G.lv[s0 + a].bptr != nullptr;  // B^_0 alone: no Alg. 1
        L.rhs = take(max_own[a] * vb);
        if (!fine) {
            L.r = take(max_own[a] * vb);
            L.e = take(b);
        }
        for (int k = 0; k < (fine ? 1 : y.kc); k++) {
            L.p[k] = take(b);
            L.q[k] = take(b);
        }
    }
    const size_t len = (size_t)y.stride * vb;
    y.F = take(len);
    y.E = take(len);
    y.out = take((size_t)2 * y.ch * vb);
    y.stage = take(max_own[y.nsp] * vb);
    if (dense) {
        y.Rv = y.F;  // r_{i+1} over r_i
        for (int k = 0; k < y.kc; k++) {
            y.P[k] = take(len);
            y.Q[k] = take(len);
        }
    }
    y.bytes = (int)off;
    if ((long)off > budget) return false;
    P.tables.assign((size_t)NR * P.table_bytes, 0);
    for (int r = 0; r < NR; r++) {
        unsigned char *im = P.tables.data() + (size_t)r * P.table_bytes;
        auto put = [&](int o, const void *p, size_t b) { if (b) std::memcpy(im + o, p, b); };
        const int nd = (int)down[r].size(), np = (int)peers[r].size();
        put(y.dhead, &nd, sizeof nd);
        put(y.down, down[r].data(), 2 * down[r].size());
        put(y.peers, &np, sizeof np);
        put(y.levels, y.lv, sizeof(ClLev) * y.nsp);
        put(y.peers + (int)sizeof(int), peers[r].data(), sizeof(int) * peers[r].size());
        for (int a = 0; a < y.nsp; a++) {
            lists(a, r, pre, post);
            put(y.lv[a].head, &head[a][r], sizeof(ClHead));
            put(y.lv[a].pre, pre.data(), sizeof(ClOp) * pre.size());
            put(y.lv[a].post, post.data(), sizeof(ClOp) * post.size());
        }
    }
    return true;
}

template <class T>
void *cluster_kernel() {
    return (void *)k_cluster_tail<T>;
}

// Launch of the cluster with `smem` bytes per CTA; attr: two attributes of the caller's. Its image
// may come in while the launch before it ends.
cudaLaunchConfig_t cluster_config(size_t smem, cudaStream_t s, cudaLaunchAttribute *attr) {
    cudaLaunchConfig_t cfg;
    std::memset(&cfg, 0, sizeof cfg);
    cfg.gridDim = dim3(kClRanks);
    cfg.blockDim = dim3(kClThreads);
    cfg.dynamicSmemBytes = smem;
    cfg.stream = s;
    attr[0].id = cudaLaunchAttributeClusterDimension;
    attr[0].val.clusterDim.x = kClRanks;
    attr[0].val.clusterDim.y = 1;
    attr[0].val.clusterDim.z = 1;
    attr[1].id = cudaLaunchAttributeProgrammaticStreamSerialization;
    attr[1].val.programmaticStreamSerializationAllowed = 1;
    cfg.attrs = attr;
    cfg.numAttrs = 2;
    return cfg;
}

// Can the device (or the part of it this process has) hold a cluster of 16 CTAs, one per SM?
// That takes 16 SMs of one GPC; without them every level runs on the grid.
template <class T>
bool cluster_fits(size_t smem, cudaStream_t s) {
    if (fault_no_cluster()) return false;
    cudaLaunchAttribute attr[2];
    const cudaLaunchConfig_t cfg = cluster_config(smem, s, attr);
    int clusters = 0;
    if (cudaFuncSetAttribute(cluster_kernel<T>(), cudaFuncAttributeMaxDynamicSharedMemorySize, (int)smem) == cudaSuccess &&
        cudaFuncSetAttribute(cluster_kernel<T>(), cudaFuncAttributeNonPortableClusterSizeAllowed, 1) == cudaSuccess &&
        cudaOccupancyMaxActiveClusters(&clusters, cluster_kernel<T>(), &cfg) == cudaSuccess)
        return clusters > 0;
    cudaGetLastError();
    return false;
}

// Chooses the cluster's levels (the finest level from which everything fits) and builds their
// image. E->cl.tl = nlev if there are none: every level runs on the grid.
template <class T>
void build_cluster(amg_hierarchy *h, EngineBase *E, int optin) {
    cudaStream_t s = h->stream;
    const int nlev = h->nlev;
    std::memset(&E->cl, 0, sizeof E->cl);
    E->cl.tl = nlev;
    cudaFuncAttributes fa;
    AMG_CUDA(cudaFuncGetAttributes(&fa, cluster_kernel<T>()));
    const long budget = (long)optin - (long)fa.sharedSizeBytes;
    if (!cluster_fits<T>((size_t)budget, s)) return;
    const std::vector<int> widths = slice_widths(h);
    auto sweepable = [&](int l) {
        const Level &lv = h->lev[l];
        return lv.n <= kClRowsMax && (int)lv.color_rows.size() - 1 <= kClColors && !lv.coarsest;
    };
    auto source = [&](int l, bool ranges) {
        ClSrc S;
        std::memset(&S, 0, sizeof S);
        const Level &lv = h->lev[l];
        S.n = lv.n;
        S.sl = lv.A.sl_ptr;
        S.col = lv.A.col;
        S.parent = lv.parent;
        S.ch = l + 1 < nlev ? h->lev[l + 1].children : nullptr;
        S.ch2 = l + 1 < nlev ? h->lev[l + 1].children2 : nullptr;
        S.val64 = lv.A.val;
        S.val32 = lv.A.val32;
        S.bptr = l == 0 ? lv.bptr : nullptr;
        S.ncol = ranges ? (int)lv.color_rows.size() - 1 : 1;
        if (ranges)
            for (int c = 0; c <= S.ncol; c++) S.cr[c] = lv.color_rows[c];
        else
            S.cr[1] = lv.n;
        return S;
    };
    // the dense level is the one above the coarsest (M, A M) or the coarsest (its inverse);
    // windows are found for every level that may be swept
    const int last = nlev - 2;  // the coarsest level that is swept or dense
    if (last < 0) return;
    int first = last + 1;
    while (first - 1 >= 1 && sweepable(first - 1) && last + 1 - (first - 1) <= kClLevels) first--;
    // the finest level too, a small quadtree's: then an application is one launch (a block is one
    // lane's: not big ones, nor an octree's). 65^2 nodes, FP64: 211 -> 153 us per application, 34^2
    // nodes: a solve 901 -> 667 us. Blocks of 6 to 16 rows too, although the grid has a lane per
    // row for them (kCoop): per application, FP64 (FP32), 90^2 nodes over 32^2 cells 185 (145) us
    // with the finest level on the grid, 145 (106) here; 45^2 over 16^2: 153 (125), 115 (90);
    // 100^2 over 32^2: 202 (149), 159 (109)
    if (first == 1 && sweepable(0) && last + 1 <= kClLevels && h->dim == 2 && h->lev[0].nbig == 0 &&
        (int)h->lev[0].color_blocks.size() == (int)h->lev[0].color_rows.size())
        first = 0;
    if (first > last) return;
    const int nch = h->dim == 3 ? 8 : 4;
    ClSrcs G;
    std::memset(&G, 0, sizeof G);
    G.nsp = last + 1 - first;
    for (int a = 0; a < G.nsp; a++) G.lv[a] = source(first + a, true);
    // the coarsest level is not smoothed; its colours only cut it into strips
    const bool crr = (int)h->lev[nlev - 1].color_rows.size() - 1 <= kClColors &&
                     h->lev[nlev - 1].color_rows.size() > 1;
    G.lv[G.nsp] = source(nlev - 1, crr);
    std::vector<int> hb;  // the finest level's blocks
    if (first == 0) {
        hb.resize(h->lev[1].n + 1);
        AMG_CUDA(cudaMemcpyAsync(hb.data(), h->lev[0].bptr, sizeof(int) * hb.size(), cudaMemcpyDeviceToHost, s));
        AMG_CUDA(cudaStreamSynchronize(s));
    }
    const size_t words = (size_t)G.nsp * kClRanks * kClColors;
    std::vector<int2> win(3 * words);
    for (int a = 0; a < G.nsp; a++)
        for (int r = 0; r < kClRanks; r++)
            for (int c = 0; c < kClColors; c++) {
                const size_t o = cl_win(a, r, c);
                win[o] = c < G.lv[a].ncol ? cl_own_rows(G.lv[a], hb, r, c) : make_int2(0, 0);
                win[words + o] = win[2 * words + o] = make_int2(INT32_MAX, 0);
            }
    const int nc = h->lev[nlev - 1].n, nfo = nc + (G.nsp > 1 ? h->lev[last].n : 0);
    Scratch tmp(s);
    int2 *dwin = tmp.get<int2>(3 * words);
    int *dfo = tmp.get<int>(nfo);
    AMG_CUDA(cudaMemcpyAsync(dwin, win.data(), sizeof(int2) * win.size(), cudaMemcpyHostToDevice, s));
    k_cl_windows<<<dim3(nblocks_for(G.lv[0].n, 256), G.nsp), 256, 0, s>>>(G, dwin, dwin + words, words, dfo);
    AMG_LAUNCH_CHECK();
    k_cl_parents<<<1, 1024, 0, s>>>(G, dwin, dwin + words, words);
    AMG_LAUNCH_CHECK();
    std::vector<int> fo(nfo);
    AMG_CUDA(cudaMemcpyAsync(win.data(), dwin, sizeof(int2) * win.size(), cudaMemcpyDeviceToHost, s));
    AMG_CUDA(cudaMemcpyAsync(fo.data(), dfo, sizeof(int) * nfo, cudaMemcpyDeviceToHost, s));
    AMG_CUDA(cudaStreamSynchronize(s));
    std::vector<int> xchild(2 * G.nsp, 0);
    for (int kind = 0; kind < 2; kind++)
        for (int a = 0; a < G.nsp; a++)
            for (size_t k = 0; k < (size_t)kClRanks * kClColors; k++) {
                const int2 w = win[(1 + kind) * words + cl_win(a, 0, 0) + k];
                if (w.x < w.y) xchild[kind * G.nsp + a] = 1;
            }
    // the finest start that fits; with the dense matrices if that start allows them
    ClSrcs GD = G;  // dense level = the last swept one
    GD.nsp = G.nsp - 1;
    const bool can_dense = last >= 1 && h->lev[last].n <= kClDenseMax;
    ClPlan P;
    bool ok = false;
    int s0 = 0;
    for (; s0 < G.nsp; s0++) {
        for (int sparse = sizeof(T) == 8; !ok && can_dense && sparse < 2; sparse++)
            ok = cluster_plan<T>(GD, win, xchild, G.nsp, fo.data() + nc, hb, widths, s0, first + s0, true, sparse != 0,
                                 nch, h->opt, budget, P);
        if (!ok)
            ok = cluster_plan<T>(G, win, xchild, G.nsp, fo.data(), hb, widths, s0, first + s0, false, false, nch,
                                 h->opt, budget, P);
        if (ok) break;
    }
    if (!ok) return;
    ClLayout &y = P.y;
    ClSrcs &U = y.dense ? GD : G;
    if (s0 > 0) {
        for (int a = 0; a + s0 <= U.nsp; a++) U.lv[a] = U.lv[a + s0];
        U.nsp -= s0;
    }
    E->cl_image = halloc<unsigned char>(h, (size_t)kClRanks * y.image_stride);
    AMG_CUDA(cudaMemsetAsync(E->cl_image, 0, (size_t)kClRanks * y.image_stride, s));
    AMG_CUDA(cudaMemcpy2DAsync(E->cl_image, y.image_stride, P.tables.data(), P.table_bytes, P.table_bytes,
                               kClRanks, cudaMemcpyHostToDevice, s));
    const Level &C = h->lev[nlev - 1];
    ClColor *geo = tmp.get<ClColor>(P.geo.size());
    int *over_n = tmp.get<int>(kClLevels * kClRanks);
    AMG_CUDA(cudaMemcpyAsync(geo, P.geo.data(), sizeof(ClColor) * P.geo.size(), cudaMemcpyHostToDevice, s));
    AMG_CUDA(cudaMemsetAsync(over_n, 0, sizeof(int) * kClLevels * kClRanks, s));
    k_cl_image<T><<<dim3(4, kClRanks, y.nsp + 1), 256, 0, s>>>(U, y, E->cl_image, geo, over_n, C.Ainv, C.Ainv32);
    AMG_LAUNCH_CHECK();
    if (y.dense) {
        const size_t smem = sizeof(double) * (3 * (size_t)y.nd + 2 * (size_t)C.n);
        k_dense_cycle<T><<<y.nd, 128, smem, s>>>(U.lv[U.nsp], y, E->cl_image, C.Ainv, C.n);
        AMG_LAUNCH_CHECK();
    }
    AMG_CUDA(cudaStreamSynchronize(s));  // P's tables are locals
    E->cl = y;
}

template <class T>
void build_engine(amg_hierarchy *h) {
    EngineBase *&slot = engine_slot<T>(h);
    if (slot) return;
    // kept only when complete (an allocation can fail part-way)
    struct Holder {
        EngineBase *p = new EngineBase();
        ~Holder() { delete p; }
    } hold;
    EngineBase *E = hold.p;
    cudaStream_t s = h->stream;
    int dev = h->device, optin = 0, nsm = 0;
    AMG_CUDA(cudaDeviceGetAttribute(&optin, cudaDevAttrMaxSharedMemoryPerBlockOptin, dev));
    AMG_CUDA(cudaDeviceGetAttribute(&nsm, cudaDevAttrMultiProcessorCount, dev));
    E->form = (coop_blocks(h->lev[0]) ? kCoop : 0) | (h->lev[0].nbig > 0 ? kBig : 0);
    build_cluster<T>(h, E, optin);
    const int tl = E->cl.tl;
    Builder b{h, &E->hprog, tl};
    if (tl == 0) b.emit(Builder::mk(OP_TAIL, 0));  // the whole application
    else b.bhat(0, V_RHS, V_E);
    annotate_reductions(E->hprog);
    if (tl < h->nlev) {
        Builder bt{h, &E->htail, h->nlev + 1};  // the cluster's ops (traffic accounting only)
        if (tl == 0) bt.bhat(0, V_RHS, V_E);
        else bt.btilde(tl);
    }
    for (const Op &op : E->htail) E->tail_bytes += op_bytes(h, op, sizeof(T));
    for (const Op &op : E->hprog)
        E->cycle_bytes += (op.kind == OP_TAIL) ? E->tail_bytes
                          : (op.kind == OP_NOP) ? 0.0 : op_bytes(h, op, sizeof(T));
    E->nops = (int)E->hprog.size();
    E->prog = halloc<Op>(h, E->hprog.size());
    AMG_CUDA(cudaMemcpyAsync(E->prog, E->hprog.data(), sizeof(Op) * E->hprog.size(),
                             cudaMemcpyHostToDevice, s));
    // Big blocks: swept in the CTAs' shared memory. A CTA-sized block needs as much as the
    // largest one that fits on the device; the warp-sized ones get a slice each on as many
    // warps per CTA as the most of them in one colour need (a block that does not fit takes
    // the global-memory sweep; the forward and backward schedules each count).
    void *kern = cycle_kernel<T>(E->form);
    cudaFuncAttributes fa;
    AMG_CUDA(cudaFuncGetAttributes(&fa, kern));
    const size_t static_smem = fa.sharedSizeBytes;
    if (h->lev[0].nbig > 0) {
        const Level &F0 = h->lev[0];
        const int vsel = sizeof(T) == 8;
        const size_t avail = (size_t)std::max<long>(0, (long)optin - (long)static_smem - 1024);
        size_t big = 0;
        for (size_t need : F0.big_smem[vsel])
            if (need > 0 && need <= avail) big = std::max(big, need);
        const size_t wneed = F0.big_smem_warp[vsel];
        int wtasks = 0;  // warp-sized blocks of the fullest colour
        for (size_t c = 0; c < F0.color_bigc.size(); c++)
            wtasks = std::max(wtasks, F0.color_bigc[c] - F0.color_big[c]);
        if (wneed > 0 && wneed <= avail && wtasks > 0) {
            const int per_cta = (wtasks + nsm - 1) / nsm;
            E->big_wwarps = std::min({cycle_threads<T>() / 32, per_cta, (int)(avail / wneed)});
            E->big_wslice = (unsigned)wneed;
        }
        const size_t smem = std::max(big, (size_t)E->big_wwarps * E->big_wslice);
        if (smem > 0) {
            E->big_smem = 1;
            E->smem = smem;
        }
    }
    // the kernel's dynamic shared-memory limit is a property of the function, shared by every
    // hierarchy of the process: set it to the device maximum (never lower it below what
    // another hierarchy's launches use); each launch passes its own size
    AMG_CUDA(cudaFuncSetAttribute(kern, cudaFuncAttributeMaxDynamicSharedMemorySize,
                                  (int)std::max<long>(0, (long)optin - (long)static_smem)));
    int per_sm = 0;
    AMG_CUDA(cudaOccupancyMaxActiveBlocksPerMultiprocessor(&per_sm, kern, cycle_threads<T>(),
                                                           E->smem));
    if (per_sm < 1) throw Error{AMG_ERR_CUDA, "persistent cycle kernel cannot be resident"};
    E->grid = nsm;  // one CTA per SM (co-resident: cooperative launch)
    E->ts = halloc<unsigned long long>(h, E->hprog.size() + 1);
    E->tprof = halloc<unsigned long long>(h, 2 * kTprofCount);
    AMG_CUDA(cudaMemsetAsync(E->tprof, 0, 2 * kTprofCount * sizeof(unsigned long long), s));
    slot = E;
    hold.p = nullptr;
}


template <class T>
void alloc_vecs(amg_hierarchy *h) {
    for (int l = 0; l < h->nlev; l++) {
        Level &lv = h->lev[l];
        Vecs<T> &v = vecs<T>(lv);
        int n = lv.n;
        if (l > 0) {
            if (!v.rhs) v.rhs = halloc<T>(h, n);
            if (!v.e) v.e = halloc<T>(h, n);
        }
        if (l > 0 && !lv.coarsest) {
            if (!v.r) v.r = halloc<T>(h, n);
            for (int i = 0; i < h->opt.kcycle_n; i++) {
                if (!v.p[i]) v.p[i] = halloc<T>(h, n);
                if (!v.q[i]) v.q[i] = halloc<T>(h, n);
            }
        }
    }
}

void ensure_fp32(amg_hierarchy *h) {
    if (h->fp32_ready) return;
    cudaStream_t s = h->stream;
    // every step keeps what an earlier, failed attempt already allocated (an allocation can
    // fail part-way; the next solve then completes the set)
    for (int l = 0; l < h->nlev; l++) {
        Level &lv = h->lev[l];
        if (lv.A.val32) continue;
        float *v = halloc<float>(h, lv.A.padded);
        k_convert<double, float><<<nblocks_for(lv.A.padded, 256), 256, 0, s>>>(
            (int)lv.A.padded, lv.A.val, v);
        AMG_LAUNCH_CHECK();
        lv.A.val32 = v;
    }
    for (int l = 0; l < h->nlev; l++) {
        Level &lv = h->lev[l];
        if (lv.dinv32) continue;
        float *d = halloc<float>(h, lv.n);
        k_inv_diag<float><<<nblocks_for(lv.n, 256), 256, 0, s>>>(lv.n, lv.A.sl_ptr, lv.A.val, d);
        AMG_LAUNCH_CHECK();
        lv.dinv32 = d;
    }
    alloc_vecs<float>(h);
    if (!h->r32) h->r32 = halloc<float>(h, h->N);
    if (!h->z32) h->z32 = halloc<float>(h, h->N);
    h->lev[0].v32.rhs = h->r32;
    h->lev[0].v32.e = h->z32;
    fill_tables<float>(h);
    build_engine<float>(h);
    h->fp32_ready = true;
}

// one application: z = B^_0 [r] on level 0's table buffers. The program runs as launches of
// the persistent kernel over the ops between the cluster's levels, and of the cluster kernel
// for these
template <class T>
void launch_cycle(amg_hierarchy *h, T *rhs0 = nullptr, T *e0 = nullptr) {
    // hierarchies of a batched setup get their single-system engine on first use
    if (!engine_slot<T>(h)) build_engine<T>(h);
    EngineBase *E = engine_slot<T>(h);
    cudaStream_t s = h->stream;
    const bool prof = profiling(h);
    CycleArgs<T> a;
    a.tab = dtab<T>(h);
    a.rhs0 = rhs0;
    a.e0 = e0;
    a.prog = E->prog;
    a.nlev = h->nlev;
    a.partials = h->cyc_partials;
    a.bar = h->bar;
    a.err = h->err_flag;
    a.bar_limit_ns = h->dbg_bar_limit_ns > 0 ? (unsigned long long)h->dbg_bar_limit_ns
                                             : kBarrierLimitNs;
    a.bar_extra = h->dbg_bar_extra;
    a.big_smem = E->big_smem;
    a.big_wwarps = E->big_wwarps;
    a.big_wslice = E->big_wslice;
    if (E->cl.tl > 0) AMG_CUDA(cudaMemsetAsync(h->bar, 0, sizeof(unsigned long long), s));
    a.ts = prof ? E->ts + 1 : nullptr;
    Profiler::Rec rec{};
    if (prof) {
        k_timestamp<<<1, 1, 0, s>>>(E->ts);
        AMG_LAUNCH_CHECK();
        rec = h->prof->begin(K_CYCLE, 0, E->cycle_bytes, s);
    }
    ClArgs<T> ca;
    cudaLaunchConfig_t cfg;
    cudaLaunchAttribute attr[2];
    if (E->cl.tl < h->nlev) {
        const Vecs<T> &v = vecs<T>(h->lev[E->cl.tl]);
        ca.y = E->cl;
        ca.image = E->cl_image;
        ca.rhs = E->cl.tl == 0 && rhs0 ? rhs0 : v.rhs;
        ca.e = E->cl.tl == 0 && e0 ? e0 : v.e;
        ca.err = h->err_flag;
        ca.limit_ns = a.bar_limit_ns;
        ca.extra = h->dbg_bar_extra;
        ca.tprof = (prof && h->prof->tail_ops) ? E->tprof : nullptr;
        cfg = cluster_config((size_t)E->cl.bytes, s, attr);
    }
    unsigned long long bars = 0;  // barriers of the launches so far
    for (int k = 0; k < E->nops;) {
        if (E->hprog[k].kind == OP_TAIL) {
            ca.ts = prof ? a.ts + k : nullptr;
            void *args[] = {&ca};
            AMG_CUDA(cudaLaunchKernelExC(&cfg, cluster_kernel<T>(), args));
            AMG_LAUNCH_CHECK();
            k++;
            continue;
        }
        a.k0 = k;
        while (k < E->nops && E->hprog[k].kind != OP_TAIL) k++;
        a.k1 = k;
        a.bar_base = bars * (unsigned long long)E->grid;
        bars += (unsigned long long)(a.k1 - a.k0 - 1);
        void *args[] = {&a};
        AMG_CUDA(cudaLaunchCooperativeKernel(cycle_kernel<T>(E->form), dim3(E->grid),
                                             dim3(cycle_threads<T>()), args, E->smem, s));
        AMG_LAUNCH_CHECK();
    }
    if (prof) h->prof->end(rec, s);
}

// per-op durations of the last profiled launch, from the in-kernel timestamps (each op's
// time includes the grid barrier that ends it)
template <class T>
void harvest_cycle_timestamps(amg_hierarchy *h) {
    EngineBase *E = engine_slot<T>(h);
    std::vector<unsigned long long> t(E->hprog.size() + 1);
    AMG_CUDA(cudaMemcpy(t.data(), E->ts, sizeof(unsigned long long) * t.size(),
                        cudaMemcpyDeviceToHost));
    for (size_t k = 0; k < E->hprog.size(); k++) {
        const Op &op = E->hprog[k];
        double ms = (double)(t[k + 1] - t[k]) * 1e-6;
        double bytes = (op.kind == OP_TAIL) ? E->tail_bytes
                       : (op.kind == OP_NOP) ? 0.0 : op_bytes(h, op, sizeof(T));
        h->prof->add(K_IN_CYCLE + op.kind, op.level, ms, bytes);
    }
    // inside the cluster: SM cycles per op kind and level, reported at the nominal clock
    std::vector<unsigned long long> tp(2 * kTprofCount);
    AMG_CUDA(cudaMemcpy(tp.data(), E->tprof, sizeof(unsigned long long) * tp.size(),
                        cudaMemcpyDeviceToHost));
    AMG_CUDA(cudaMemset(E->tprof, 0, sizeof(unsigned long long) * tp.size()));
    int khz = 0;
    AMG_CUDA(cudaDeviceGetAttribute(&khz, cudaDevAttrClockRate, h->device));
    for (int slot = 0; slot < kTprofCount; slot++)
        if (tp[kTprofCount + slot])
            h->prof->add(K_IN_TAIL + (slot & 15), slot / 16, (double)tp[slot] / khz, 0.0,
                         (int64_t)tp[kTprofCount + slot]);
}

// standalone execution of B^_l (diagnostic path): one kernel per op, every level in HBM
template <class T>
void run_standalone(amg_hierarchy *h, int l, int fsel, int zsel) {
    cudaStream_t s = h->stream;
    std::vector<Op> prog;
    Builder b{h, &prog, h->nlev + 1};
    b.bhat(l, fsel, zsel);
    RedCtx rc{h->red_partials, h->red_counter};
    for (const Op &op : prog) {
        const Level &lv = h->lev[op.level];
        int grid;
        switch (op.kind) {
            case OP_GS: grid = nblocks_for(op.i1 - op.i0, kRedThreads); break;
            case OP_RESTRICT: grid = nblocks_for(h->lev[op.level + 1].n, kRedThreads); break;
            case OP_COARSE: grid = 1; break;
            case OP_MULTIDOT:
            case OP_SPMV_DOT:
            case OP_UPDATE: grid = red_grid(lv.n); break;
            default: grid = nblocks_for(lv.n, kRedThreads);
        }
        k_op<T><<<grid, kRedThreads, 0, s>>>(dtab<T>(h), op, rc);
        AMG_LAUNCH_CHECK();
    }
}

}  // namespace

// the cycle's level copies in its precision (FP32 copies are made once, on first use)
void prepare_cycle(amg_hierarchy *h) {
    if (h->opt.cycle_prec != AMG_FP32 || h->fp32_ready) return;
    if (h->nlev > 1) {
        ensure_fp32(h);
        return;
    }
    // one level: the cycle is the exact solve (high/low float inverse) on FP32 vectors
    h->r32 = halloc<float>(h, h->N);
    h->z32 = halloc<float>(h, h->N);
    h->lev[0].v32.rhs = h->r32;
    h->lev[0].v32.e = h->z32;
    fill_tables<float>(h);
    h->fp32_ready = true;
}

// device level table of the cycle precision (LevelDev<T>[nlev])
const void *level_table(const amg_hierarchy *h, bool fp32) {
    return fp32 ? h->lev_tab32 : h->lev_tab64;
}

void allocate_solve_workspace(amg_hierarchy *h) {
    const int n = (int)h->N;
    h->red_partials = halloc<double>(h, (size_t)kRedBlocks * std::max(8, h->opt.max_iters + 8));
    h->red_counter = halloc<unsigned int>(h, 1);
    AMG_CUDA(cudaMemsetAsync(h->red_counter, 0, sizeof(unsigned int), h->stream));
    h->cyc_partials = halloc<double>(h, 2 * 4 * 1024);
    h->bar = halloc<unsigned long long>(h, 32);
    AMG_CUDA(cudaMemsetAsync(h->bar, 0, 32 * sizeof(unsigned long long), h->stream));
    alloc_vecs<double>(h);
    // level-0 cycle input / output are the outer solver's r and z
    h->xo = halloc<double>(h, n);
    h->ro = halloc<double>(h, n);
    h->zo = halloc<double>(h, n);
    h->to = halloc<double>(h, n);
    h->bo = halloc<double>(h, n);
    h->lev[0].v64.rhs = h->ro;
    h->lev[0].v64.e = h->zo;
    h->osc = halloc<double>(h, outer_scalar_count(h->opt.max_iters));
    h->dP = halloc<double *>(h, h->opt.max_iters);
    h->dQ = halloc<double *>(h, h->opt.max_iters);
    ensure_pinned(h);
    for (int l = 0; l < h->nlev; l++) {
        Level &lv = h->lev[l];
        lv.dinv64 = halloc<double>(h, lv.n);
        k_inv_diag<double><<<nblocks_for(lv.n, 256), 256, 0, h->stream>>>(lv.n, lv.A.sl_ptr, lv.A.val,
                                                                          lv.dinv64);
        AMG_LAUNCH_CHECK();
    }
    fill_tables<double>(h);
    // the FP64 cycle's engine now; an FP32-cycle hierarchy builds its FP32 engine on its first
    // solve (ensure_fp32), and an FP64 one only if the FP64 cycle is ever launched
    if (h->nlev > 1 && h->opt.cycle_prec != AMG_FP32) build_engine<double>(h);
}

int bounds_flags_solve() { return bounds_flag_read_clear(); }

size_t outer_scalar_count(int max_iters) { return OS_ZQ + 2 * (size_t)max_iters + 8; }

void ensure_pinned(amg_hierarchy *h) {
    if (!h->h_pinned)
        AMG_CUDA(cudaMallocHost(&h->h_pinned, (64 + 2 * (size_t)h->opt.max_iters) * sizeof(double)));
}

double cycle_application_bytes(amg_hierarchy *h, int value_bytes) {
    std::vector<Op> prog;
    Builder b{h, &prog, h->nlev + 1};  // every level's ops, down to the coarsest
    b.bhat(0, V_RHS, V_E);
    double s = 0.0;
    for (const Op &op : prog)
        if (op.kind != OP_NOP) s += op_bytes(h, op, value_bytes);
    return s;
}

size_t level_table_image(amg_hierarchy *h, bool fp32, std::vector<unsigned char> &out) {
    auto put = [&](const auto &tab) {
        const size_t b = sizeof(tab[0]) * tab.size();
        out.resize(b);
        std::memcpy(out.data(), tab.data(), b);
        return b;
    };
    if (fp32) {
        std::vector<GLev<float>> tab;
        table_image<float>(h, tab);
        return put(tab);
    }
    std::vector<GLev<double>> tab;
    table_image<double>(h, tab);
    return put(tab);
}

int first_cluster_level(const amg_hierarchy *h) {
    const EngineBase *E = h->opt.cycle_prec == AMG_FP32 ? h->eng32 : h->eng64;
    return E ? E->cl.tl : -1;
}

void free_engines(amg_hierarchy *h) {
    delete h->eng64;
    delete h->eng32;
    h->eng64 = h->eng32 = nullptr;
}

int ensure_directions(amg_hierarchy *h, int count) {
    const int n = (int)h->N;
    const int chunk = 16;
    int old = (int)h->P.size();
    if (count <= old) return old;
    int target = std::min(h->opt.max_iters, ((count + chunk - 1) / chunk) * chunk);
    // the new P and Q vectors in one allocation (each 256-byte aligned); if it fails, P and
    // Q keep their length
    const size_t stride = ((size_t)n + 31) & ~(size_t)31, m = (size_t)(target - old);
    double *slab = halloc<double>(h, 2 * m * stride);
    for (size_t j = 0; j < m; j++) {
        h->P.push_back(slab + j * stride);
        h->Q.push_back(slab + (m + j) * stride);
    }
    AMG_CUDA(cudaMemcpyAsync(h->dP, h->P.data(), sizeof(double *) * target, cudaMemcpyHostToDevice,
                             h->stream));
    AMG_CUDA(cudaMemcpyAsync(h->dQ, h->Q.data(), sizeof(double *) * target, cudaMemcpyHostToDevice,
                             h->stream));
    AMG_CUDA(cudaStreamSynchronize(h->stream));  // the tables are copied from host vectors
    return target;
}

static GLev<double> fine_view(amg_hierarchy *h) {
    GLev<double> L;
    std::memset(&L, 0, sizeof L);
    Level &lv = h->lev[0];
    L.n = lv.n;
    L.w = lv.A.uw;
    L.sl = lv.A.sl_ptr;
    L.col = lv.A.col;
    L.val = lv.A.val;
    return L;
}

// the error flag of the cycle's kernels, read by the caller
static void raise_device_error(amg_hierarchy *h, int err) {
    if (err & kErrTimeout) {
        // the kernels ended early: clear the flag and the barrier state for the next launch
        AMG_CUDA(cudaMemsetAsync(h->err_flag, 0, sizeof(int), h->stream));
        AMG_CUDA(cudaMemsetAsync(h->bar, 0, sizeof(unsigned long long), h->stream));
        AMG_CUDA(cudaStreamSynchronize(h->stream));
        throw Error{AMG_ERR_TIMEOUT, "a wait inside the cycle (grid barrier or cluster exchange) timed out"};
    }
}

static void check_device_error(amg_hierarchy *h) {
    int err = 0;
    AMG_CUDA(cudaMemcpyAsync(&err, h->err_flag, sizeof(int), cudaMemcpyDeviceToHost, h->stream));
    AMG_CUDA(cudaStreamSynchronize(h->stream));
    raise_device_error(h, err);
}

// one application of B^_0 to h->ro (FP64) into h->zo (FP64)
// out = B^_0 [in] (FP64 vectors; in = h->ro, out = h->zo unless given: the FGMRES basis
// passes its vectors directly)
static void apply_preconditioner(amg_hierarchy *h, const double *in = nullptr,
                                 double *out = nullptr) {
    cudaStream_t s = h->stream;
    const int n = (int)h->N;
    if (!in) in = h->ro;
    if (!out) out = h->zo;
    if (h->nlev == 1) {  // exact solve on the only level (table vectors ro -> zo)
        if (in != h->ro)
            AMG_CUDA(cudaMemcpyAsync(h->ro, in, sizeof(double) * n, cudaMemcpyDeviceToDevice, s));
        Op op = Builder::mk(OP_COARSE, 0);
        RedCtx rc{h->red_partials, h->red_counter};
        k_op<double><<<1, kRedThreads, 0, s>>>(dtab<double>(h), op, rc);
        AMG_LAUNCH_CHECK();
        if (out != h->zo)
            AMG_CUDA(cudaMemcpyAsync(out, h->zo, sizeof(double) * n, cudaMemcpyDeviceToDevice, s));
        return;
    }
    if (h->opt.cycle_prec == AMG_FP32) {
        k_convert<double, float><<<nblocks_for(n, 256), 256, 0, s>>>(n, in, h->r32);
        AMG_LAUNCH_CHECK();
        launch_cycle<float>(h);
        k_convert<float, double><<<nblocks_for(n, 256), 256, 0, s>>>(n, h->z32, out);
        AMG_LAUNCH_CHECK();
    } else {
        launch_cycle<double>(h, const_cast<double *>(in), out);
    }
}

static int solve_fgmres(amg_hierarchy *h, const double *b_nat, double tol, double *x_nat,
                        int *iters, double *relres);

int solve(amg_hierarchy *h, const double *b_nat, double tol, double *x_nat, int *iters,
          double *relres) {
    ensure_pinned(h);  // a hierarchy of the batched setup allocates it here
    if (h->opt.outer == AMG_OUTER_FGMRES) return solve_fgmres(h, b_nat, tol, x_nat, iters, relres);
    cudaStream_t s = h->stream;
    const int n = (int)h->N;
    const int maxit = h->opt.max_iters;
    Level &F = h->lev[0];
    RedCtx rc{h->red_partials, h->red_counter};
    const bool prof = profiling(h);
    if (h->opt.cycle_prec == AMG_FP32 && h->nlev > 1) ensure_fp32(h);
    // x = 0, r = b (pi order)
    k_gather<<<nblocks_for(n, 256), 256, 0, s>>>(n, F.nat, b_nat, h->bo);
    AMG_LAUNCH_CHECK();
    AMG_CUDA(cudaMemcpyAsync(h->ro, h->bo, sizeof(double) * n, cudaMemcpyDeviceToDevice, s));
    AMG_CUDA(cudaMemsetAsync(h->xo, 0, sizeof(double) * n, s));
    AMG_CUDA(cudaMemsetAsync(h->osc, 0, sizeof(double) * 8, s));
    k_norm2<<<red_grid(n), kRedThreads, 0, s>>>(n, h->bo, h->osc + OS_BB, rc);
    AMG_LAUNCH_CHECK();
    AMG_CUDA(cudaMemcpyAsync(h->h_pinned, h->osc, sizeof(double) * 8, cudaMemcpyDeviceToHost, s));
    AMG_CUDA(cudaStreamSynchronize(s));
    const double bn = std::sqrt(h->h_pinned[OS_BB]);
    int status = AMG_ERR_NOT_CONVERGED;
    int it = 0;
    double rel = 1.0;
    if (!std::isfinite(bn)) throw Error{AMG_ERR_INVALID_ARG, "non-finite right-hand side"};
    if (bn == 0.0) {
        status = AMG_OK;
        rel = 0.0;
    } else {
        double *opq = h->osc + OS_ZQ + maxit;
        GLev<double> Lf = fine_view(h);
        const double nd = n, nnz = (double)F.A.stored;
        for (it = 0; it < maxit;) {
            ensure_directions(h, it + 1);
            apply_preconditioner(h);  // zo = B^[ro]
            Profiler::Rec rec{};
            if (prof) rec = h->prof->begin(K_OUTER_MULTIDOT, 0, 8.0 * nd * (1 + it), s);
            launch_following(k_outer_multidot, red_grid(n), kRedThreads, s, n, h->zo, h->dQ, it, h->osc, rc);
            AMG_LAUNCH_CHECK();
            if (prof) h->prof->end(rec, s);
            if (prof) rec = h->prof->begin(K_OUTER_ORTH, 0, 8.0 * nd * (2 + it), s);
            launch_following(k_outer_orth, nblocks_for(n, 256), 256, s, n, h->zo, h->dP, it, h->osc, opq);
            AMG_LAUNCH_CHECK();
            if (prof) h->prof->end(rec, s);
            if (prof) rec = h->prof->begin(K_OUTER_SPMV_DOT, 0, 12.0 * nnz + 24.0 * nd, s);
            launch_following(k_outer_spmv_dot, red_grid(n), kRedThreads, s, Lf, h->dP, h->dQ, it, h->ro,
                                                                 h->osc, opq, rc);
            AMG_LAUNCH_CHECK();
            if (prof) h->prof->end(rec, s);
            if (prof) rec = h->prof->begin(K_OUTER_UPDATE, 0, 48.0 * nd, s);
            launch_following(k_outer_update, red_grid(n), kRedThreads, s, n, h->dP, h->dQ, it, h->xo,
                                                               h->ro, h->osc, opq,
                                                               h->err_flag, rc);
            AMG_LAUNCH_CHECK();
            if (prof) h->prof->end(rec, s);
            AMG_CUDA(cudaMemcpyAsync(h->h_pinned, h->osc, sizeof(double) * 8,
                                     cudaMemcpyDeviceToHost, s));
            AMG_CUDA(cudaStreamSynchronize(s));
            if (h->nlev > 1) raise_device_error(h, (int)h->h_pinned[OS_ERR]);
            if (prof) {
                h->prof->harvest();
                if (h->nlev > 1) {
                    if (h->opt.cycle_prec == AMG_FP32) harvest_cycle_timestamps<float>(h);
                    else harvest_cycle_timestamps<double>(h);
                }
            }
            it++;
            if (h->h_pinned[OS_STOP] != 0.0) {
                status = AMG_ERR_BREAKDOWN;
                break;
            }
            rel = std::sqrt(h->h_pinned[OS_RR]) / bn;
            if (!std::isfinite(rel)) {
                status = AMG_ERR_BREAKDOWN;
                break;
            }
            if (rel <= tol) {
                k_true_residual<<<red_grid(n), kRedThreads, 0, s>>>(Lf, h->bo, h->xo, h->to,
                                                                    h->osc + OS_TT, rc);
                AMG_LAUNCH_CHECK();
                AMG_CUDA(cudaMemcpyAsync(h->h_pinned, h->osc, sizeof(double) * 8,
                                         cudaMemcpyDeviceToHost, s));
                AMG_CUDA(cudaStreamSynchronize(s));
                rel = std::sqrt(h->h_pinned[OS_TT]) / bn;
                if (rel <= tol) {
                    status = AMG_OK;
                    break;
                }
                AMG_CUDA(cudaMemcpyAsync(h->ro, h->to, sizeof(double) * n, cudaMemcpyDeviceToDevice, s));
            }
        }
        if (status != AMG_OK) {
            k_true_residual<<<red_grid(n), kRedThreads, 0, s>>>(Lf, h->bo, h->xo, h->to,
                                                                h->osc + OS_TT, rc);
            AMG_LAUNCH_CHECK();
            AMG_CUDA(cudaMemcpyAsync(h->h_pinned, h->osc, sizeof(double) * 8,
                                     cudaMemcpyDeviceToHost, s));
            AMG_CUDA(cudaStreamSynchronize(s));
            rel = std::sqrt(h->h_pinned[OS_TT]) / bn;
        }
    }
    k_scatter<<<nblocks_for(n, 256), 256, 0, s>>>(n, F.nat, h->xo, x_nat);
    AMG_LAUNCH_CHECK();
    AMG_CUDA(cudaStreamSynchronize(s));
    if (iters) *iters = it;
    if (relres) *relres = rel;
    return status;
}


// Restarted flexible GMRES(m) (right preconditioning, FP64 basis and Hessenberg matrix,
// classical Gram-Schmidt applied twice): the outer iteration for a preconditioner that
// varies between applications (the nonlinear AMLI-cycle, in FP32 or FP64). The host keeps the
// (m+1) x m Hessenberg matrix and its Givens rotations; each iteration reads m+2 scalars.
static int solve_fgmres(amg_hierarchy *h, const double *b_nat, double tol, double *x_nat,
                        int *iters, double *relres) {
    cudaStream_t s = h->stream;
    const int n = (int)h->N;
    const int maxit = h->opt.max_iters;
    const int m = std::max(1, std::min(h->opt.fgmres_restart, maxit));
    Level &F = h->lev[0];
    RedCtx rc{h->red_partials, h->red_counter};
    if (h->opt.cycle_prec == AMG_FP32 && h->nlev > 1) ensure_fp32(h);
    // basis V[0..m], preconditioned directions Z[0..m-1] (the outer direction store)
    ensure_directions(h, std::min(maxit, std::max(2 * m + 1, 1)));
    if ((int)h->P.size() < 2 * m + 1) throw Error{AMG_ERR_UNSUPPORTED, "max_iters too small for the restart length"};
    double **dV = h->dP;          // V[i] = P[i], i <= m
    double **dZ = h->dP + m + 1;  // Z[j] = P[m + 1 + j]
    double *w = h->to;
    double *dh = h->osc + OS_ZQ;           // first pass's dots and the norm: m + 2 scalars
    double *dh2 = h->osc + OS_ZQ + m + 2;  // second pass's dots: m + 1 (maxit >= 2m + 1)
    GLev<double> Lf = fine_view(h);
    k_gather<<<nblocks_for(n, 256), 256, 0, s>>>(n, F.nat, b_nat, h->bo);
    AMG_LAUNCH_CHECK();
    AMG_CUDA(cudaMemsetAsync(h->xo, 0, sizeof(double) * n, s));
    k_norm2<<<red_grid(n), kRedThreads, 0, s>>>(n, h->bo, h->osc + OS_BB, rc);
    AMG_LAUNCH_CHECK();
    AMG_CUDA(cudaMemcpyAsync(h->h_pinned, h->osc, sizeof(double) * 8, cudaMemcpyDeviceToHost, s));
    AMG_CUDA(cudaStreamSynchronize(s));
    const double bn = std::sqrt(h->h_pinned[OS_BB]);
    if (!std::isfinite(bn)) throw Error{AMG_ERR_INVALID_ARG, "non-finite right-hand side"};
    int it = 0, status = AMG_ERR_NOT_CONVERGED;
    double rel = 1.0;
    const bool prof = profiling(h);
    const double nd = n, nnzf = (double)F.A.stored;
    std::vector<double> H((size_t)(m + 1) * m), cs(m), sn(m), g(m + 1), y(m);
    std::vector<double> hv(std::max(m + 2, 8));
    double *dy = h->osc + OS_ZQ + maxit + 4;  // coefficients for the update (m <= maxit)
    auto read_scalars = [&](const double *d, int count, double *out) {
        AMG_CUDA(cudaMemcpyAsync(h->h_pinned, d, sizeof(double) * count, cudaMemcpyDeviceToHost, s));
        AMG_CUDA(cudaStreamSynchronize(s));
        for (int k = 0; k < count; k++) out[k] = h->h_pinned[k];
    };
    if (bn == 0.0) {
        status = AMG_OK;
        rel = 0.0;
    }
    // r = b - A x (x = 0 at the start)
    AMG_CUDA(cudaMemcpyAsync(h->ro, h->bo, sizeof(double) * n, cudaMemcpyDeviceToDevice, s));
    double beta = bn;
    while (status != AMG_OK && it < maxit) {
        // V[0] = r / beta
        k_scale<<<nblocks_for(n, 256), 256, 0, s>>>(n, h->ro, 1.0 / beta, h->P[0]);
        AMG_LAUNCH_CHECK();
        std::fill(g.begin(), g.end(), 0.0);
        g[0] = beta;
        int j = 0;
        bool done = false;
        for (; j < m && it < maxit; j++) {
            // Z[j] = B^[V[j]]
            apply_preconditioner(h, h->P[j], h->P[m + 1 + j]);
            // w = A Z[j], orthogonalised twice against V[0..j]
            Profiler::Rec rec{};
            if (prof) rec = h->prof->begin(K_FGMRES_SPMV, 0, 12.0 * nnzf + 16.0 * nd, s);
            k_spmv<<<nblocks_for(n, 256), 256, 0, s>>>(Lf, h->P[m + 1 + j], w);
            AMG_LAUNCH_CHECK();
            if (prof) h->prof->end(rec, s);
            // classical Gram-Schmidt twice: h1 = V^t w, w -= V h1, h2 = V^t w, w -= V h2
            if (prof) rec = h->prof->begin(K_FGMRES_MDOT, 0, 8.0 * nd * (j + 2), s);
            k_mdot<<<red_grid(n), kRedThreads, 0, s>>>(n, w, dV, j + 1, dh, rc);
            AMG_LAUNCH_CHECK();
            if (prof) h->prof->end(rec, s);
            if (prof) rec = h->prof->begin(K_FGMRES_ORTH, 0, 8.0 * nd * (j + 3), s);
            k_orth_mdot<<<red_grid(n), kRedThreads, 0, s>>>(n, w, dV, j + 1, dh, dh2, rc);
            AMG_LAUNCH_CHECK();
            if (prof) h->prof->end(rec, s);
            if (prof) rec = h->prof->begin(K_FGMRES_ORTH, 0, 8.0 * nd * (j + 3), s);
            k_orth_sub<<<red_grid(n), kRedThreads, 0, s>>>(n, w, dV, j + 1, dh2, dh + j + 1, h->err_flag,
                                                          h->osc + OS_ERR, rc);
            AMG_LAUNCH_CHECK();
            if (prof) h->prof->end(rec, s);
            {  // the cycle's error flag, h1 and the norm, h2: one read back of [OS_ERR, dh2 + j + 1)
                const double *hp = h->h_pinned;
                AMG_CUDA(cudaMemcpyAsync(h->h_pinned, h->osc + OS_ERR, sizeof(double) * (1 + m + 2 + j + 1),
                                         cudaMemcpyDeviceToHost, s));
                AMG_CUDA(cudaStreamSynchronize(s));
                if (h->nlev > 1) raise_device_error(h, (int)hp[0]);
                for (int i = 0; i < j + 2; i++) hv[i] = hp[1 + i];
                for (int i = 0; i <= j; i++) H[(size_t)i * m + j] = (0.0 + hv[i]) + hp[1 + m + 2 + i];
            }
            if (prof) {
                h->prof->harvest();
                if (h->nlev > 1) {
                    if (h->opt.cycle_prec == AMG_FP32) harvest_cycle_timestamps<float>(h);
                    else harvest_cycle_timestamps<double>(h);
                }
            }
            it++;
            const double hn = std::sqrt(hv[j + 1]);
            H[(size_t)(j + 1) * m + j] = hn;
            // apply the previous rotations to column j, then a new one
            for (int i = 0; i < j; i++) {
                double a = H[(size_t)i * m + j], b2 = H[(size_t)(i + 1) * m + j];
                H[(size_t)i * m + j] = cs[i] * a + sn[i] * b2;
                H[(size_t)(i + 1) * m + j] = -sn[i] * a + cs[i] * b2;
            }
            double a = H[(size_t)j * m + j], b2 = H[(size_t)(j + 1) * m + j];
            double r = std::hypot(a, b2);
            if (!(r > 0.0) || !std::isfinite(r)) {
                status = AMG_ERR_BREAKDOWN;
                done = true;
                break;
            }
            cs[j] = a / r;
            sn[j] = b2 / r;
            H[(size_t)j * m + j] = r;
            H[(size_t)(j + 1) * m + j] = 0.0;
            g[j + 1] = -sn[j] * g[j];
            g[j] = cs[j] * g[j];
            rel = std::fabs(g[j + 1]) / bn;
            if (rel <= tol) {
                j++;
                done = true;
                break;
            }
            if (hn > 0.0) {
                k_scale<<<nblocks_for(n, 256), 256, 0, s>>>(n, w, 1.0 / hn, h->P[j + 1]);
                AMG_LAUNCH_CHECK();
            } else {  // exact solution in the Krylov space
                j++;
                done = true;
                break;
            }
        }
        const int k = std::min(j, m);
        // y = H(0:k,0:k)^{-1} g(0:k); x += Z y
        for (int i = k - 1; i >= 0; i--) {
            double acc = g[i];
            for (int l = i + 1; l < k; l++) acc -= H[(size_t)i * m + l] * y[l];
            y[i] = acc / H[(size_t)i * m + i];
        }
        if (k > 0) {
            std::memcpy(h->h_pinned, y.data(), sizeof(double) * k);
            AMG_CUDA(cudaMemcpyAsync(dy, h->h_pinned, sizeof(double) * k, cudaMemcpyHostToDevice, s));
            k_lincomb<<<nblocks_for(n, 256), 256, 0, s>>>(n, h->xo, dZ, k, dy);
            AMG_LAUNCH_CHECK();
        }
        // true residual r = b - A x
        k_true_residual<<<red_grid(n), kRedThreads, 0, s>>>(Lf, h->bo, h->xo, h->ro, h->osc + OS_TT, rc);
        AMG_LAUNCH_CHECK();
        read_scalars(h->osc, 8, hv.data());
        beta = std::sqrt(hv[OS_TT]);
        rel = beta / bn;
        if (rel <= tol) status = AMG_OK;
        else if (status == AMG_ERR_BREAKDOWN) break;
        (void)done;
    }
    k_scatter<<<nblocks_for(n, 256), 256, 0, s>>>(n, F.nat, h->xo, x_nat);
    AMG_LAUNCH_CHECK();
    AMG_CUDA(cudaStreamSynchronize(s));
    if (iters) *iters = it;
    if (relres) *relres = rel;
    return status;
}

// z = B^_level [f] in natural order (FP64). Level 0 runs the persistent kernel exactly as the
// solve does; coarser levels run the standalone executor (one kernel per op).
void apply_cycle_level(amg_hierarchy *h, int level, const double *f_nat, double *z_nat) {
    cudaStream_t s = h->stream;
    Level &lv = h->lev[level];
    const int n = lv.n;
    RedCtx rc{h->red_partials, h->red_counter};
    if (lv.coarsest) {
        double *fbuf = level == 0 ? h->ro : lv.v64.rhs;
        double *ebuf = level == 0 ? h->zo : lv.v64.e;
        k_gather<<<nblocks_for(n, 256), 256, 0, s>>>(n, lv.nat, f_nat, fbuf);
        AMG_LAUNCH_CHECK();
        Op op = Builder::mk(OP_COARSE, level);
        k_op<double><<<1, kRedThreads, 0, s>>>(dtab<double>(h), op, rc);
        AMG_LAUNCH_CHECK();
        k_scatter<<<nblocks_for(n, 256), 256, 0, s>>>(n, lv.nat, ebuf, z_nat);
        AMG_LAUNCH_CHECK();
        AMG_CUDA(cudaStreamSynchronize(s));
        return;
    }
    if (level == 0) {  // the solve's preconditioner, in the configured cycle precision
        if (h->opt.cycle_prec == AMG_FP32) ensure_fp32(h);
        k_gather<<<nblocks_for(n, 256), 256, 0, s>>>(n, lv.nat, f_nat, h->ro);
        AMG_LAUNCH_CHECK();
        apply_preconditioner(h);
        k_scatter<<<nblocks_for(n, 256), 256, 0, s>>>(n, lv.nat, h->zo, z_nat);
        AMG_LAUNCH_CHECK();
        AMG_CUDA(cudaStreamSynchronize(s));
        check_device_error(h);
        return;
    }
    k_gather<<<nblocks_for(n, 256), 256, 0, s>>>(n, lv.nat, f_nat, lv.v64.rhs);
    AMG_LAUNCH_CHECK();
    run_standalone<double>(h, level, V_RHS, V_P0);
    k_scatter<<<nblocks_for(n, 256), 256, 0, s>>>(n, lv.nat, lv.v64.p[0], z_nat);
    AMG_LAUNCH_CHECK();
    AMG_CUDA(cudaStreamSynchronize(s));
}

// one sweep of the coloured smoother on `level`, natural order in/out (FP64)
void smooth_level(amg_hierarchy *h, int level, int backward, const double *f_nat, double *u_nat) {
    cudaStream_t s = h->stream;
    Level &lv = h->lev[level];
    const int n = lv.n;
    double *fbuf = level == 0 ? h->ro : lv.v64.rhs;
    double *ubuf = level == 0 ? h->zo : lv.v64.e;
    k_gather<<<nblocks_for(n, 256), 256, 0, s>>>(n, lv.nat, f_nat, fbuf);
    k_gather<<<nblocks_for(n, 256), 256, 0, s>>>(n, lv.nat, u_nat, ubuf);
    AMG_LAUNCH_CHECK();
    const std::vector<int> &ranges = (level == 0) ? lv.color_blocks : lv.color_rows;
    const int nc = (int)ranges.size() - 1;
    RedCtx rc{h->red_partials, h->red_counter};
    for (int k = 0; k < nc; k++) {
        int c = backward ? nc - 1 - k : k;
        if (ranges[c + 1] == ranges[c]) continue;
        Op g = Builder::mk(OP_GS, level);
        g.i0 = ranges[c];
        g.i1 = ranges[c + 1];
        g.backward = backward;
        g.fsel = V_RHS;
        g.usel = V_E;
        Builder{h, nullptr, h->nlev}.big_range(level, c, g);
        k_op<double><<<nblocks_for(g.i1 - g.i0, kRedThreads), kRedThreads, 0, s>>>(dtab<double>(h), g, rc);
        AMG_LAUNCH_CHECK();
    }
    k_scatter<<<nblocks_for(n, 256), 256, 0, s>>>(n, lv.nat, ubuf, u_nat);
    AMG_LAUNCH_CHECK();
    AMG_CUDA(cudaStreamSynchronize(s));
}

}  // namespace amg
