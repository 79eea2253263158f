// The coarse levels of the AMLI-cycle in the shared memory of one thread-block cluster.
//
// B~_tl (Alg. 1 with Alg. 2 inside, down to the exact coarsest solve) is a chain of thousands
// of dependent steps over a few hundred to a few thousand rows each, so what bounds it is the
// latency of a step, not bytes or arithmetic. k_cluster_tail runs it on 16 CTAs of one cluster
// (the largest cluster the GPU takes): every level is cut into 16 strips, each CTA holds its
// strip's rows and vectors in its own shared memory with the neighbours' rows its rows read
// ("the window"), and after each step the new values go straight into the neighbours' windows
// (st.async, counted by an mbarrier on the receiving side): no round trip through L2, no
// grid-wide barrier, and a step waits for its neighbours only. Measured on GB300 in a loop of
// the primitive (SM cycles on top of the loop): values to two neighbours and the wait for
// theirs 390, a cluster-wide barrier 440 plus 570 for a load from a peer's shared memory, a
// grid barrier over L2 2,900.
//
// Colour c of a level is the contiguous row range [cr[c], cr[c+1]); CTA r owns its part
// [len r / 16, len (r+1) / 16). Rows of a colour ascend by cell, so a part is a strip of the
// auxiliary grid. CTA r's window of colour c is the smallest row interval that holds its own
// rows, the columns of its own rows, the rows whose columns its own rows are (both, so that
// the exchange is symmetric), the children of its own rows of the next level, and the parents
// of its window on the level above. The vectors that others read
// (z, e, the residual) are stored in window order, the others by own row.
//
// What keeps the steps in order without a cluster barrier. Neighbour exchanges are numbered;
// exchange k counts on mbarrier k mod 2. Each CTA sends every neighbour (the same set for all
// levels) a 4-byte token besides the rows of exchange k, and leaves exchange k when all tokens,
// rows and its own warps' arrivals have come in, so neighbours are at most one exchange
// apart. In exchange k a CTA writes rows of one colour (or one vector) into its neighbours'
// windows; a neighbour that still computes step k neither reads nor writes these: rows of one
// colour are not coupled, and the steps that fill a whole window (from zero, prolongation)
// leave out the colour that is exchanged next. One that still computes step k-1 can only be
// at rows it does not send here, which read nothing of this CTA's (symmetric windows).
// A token comes from the CTA's last warp and vouches for that warp alone; rows vouch for the warps
// that sent them. So a step that writes window entries which other CTAs own, and which a
// neighbour may send in the exchange after this one, has a CTA barrier before its arrival: the
// zeroed windows at the entry and before a level's first colour, the correction added on the
// finest level. (The checking build, -DAMG_BOUNDS_CHECK, keeps some warps of every step waiting
// for a few microseconds, another set each step, so that a missing one shows in the results.)
// Sums over the cluster and gathers to all CTAs count on two mbarriers of their own, by the same
// rule: every CTA sends something in each (its sums, its rows of a product, and in the gather into
// the dense level a token, as it may own no row there), so none is more than one behind. A CTA
// without rows on any level has no neighbours and is held to the others by these alone.
//
// The level above the coarsest: B^ there is linear (the coarsest solve is exact), so setup
// forms M = B^ and A M as dense matrices once (k_dense_cycle, FP64), each CTA keeps 1/16 of
// their rows, and one product with a residual gives p and A p of an Alg. 1 step; that replaces
// about 13 dependent steps. In FP32 M takes the coarsest inverse's place and is held like it, as a
// sum of two floats with a compensated product, so p is rounded once; A M is one float with a plain
// sum, as A itself is where a level is swept: its error against 64 bits is 5e-8 to 1e-7, of a
// product of A with the rounded p 1.3e-7 to 1.6e-6 (squares, disks, graded, cubes; random and smooth
// r), as |A M| |r| is 0.03 to 0.7 of |A| |p|. FP64 keeps M alone and multiplies by the sparse A
// after it (256 rows: a product with both is 4,900 cycles of the FP64 pipe, with M 2,450 and one
// more gather 600: 9.7 -> 8.8 us per visit, 9.1 with beta rounded once). So does FP32 where M's two
// parts fit but not A M beside them (512 rows); A's few rows per CTA are then read through L1. Where
// M does not fit, the level is swept like the others and the coarsest solve is the dense product.
#pragma once

#include <cstddef>
#include <cstring>
#include <type_traits>

#include "cycle_ops.cuh"

namespace amg {

constexpr int kClRanks = 16;       // CTAs of the cluster
constexpr int kClThreads = 256;
constexpr int kClWarps = kClThreads / 32;
constexpr int kClLevels = 8;       // swept levels at most
constexpr int kClColors = 32;      // colours of a swept level at most
constexpr int kClRowsMax = 20480;  // rows of a swept level at most (16-bit window indices)
constexpr int kClDenseMax = 512;   // rows of the dense level at most
constexpr int kClSlots = 8;        // off-diagonal slots a lane takes at most
constexpr unsigned kClNone = 0x7FFFFFFFu;  // no destination

// one colour of a sweep on one CTA's strip; a level's sweeps are lists of these
struct __align__(16) ClOp {
    int m0, cnt;       // own rows, times lanes per row
    int expect;        // bytes its window receives in the exchange
    int pad;
};
struct __align__(16) ClHead {  // of one level's strip
    int nown, nwin, expect_all, fexp;  // fexp: bytes of the first non-empty colour,
    int fc0, fcn, fs0, fs1;    //   its own rows [fc0, fc0 + fcn) and window [fs0, fs1)
    int ls0, ls1, pad[2];      // last non-empty colour: window
};
// one colour of one CTA's strip (setup of the image only)
struct ClColor {
    int li0, cnt;      // own rows: window index of the first, number
    int m0;            // its index among the own rows of all colours
    int seg0, seglen;  // the colour's window
    int g0;            // pi-row of the first own row
};

// a swept level: sizes, and byte offsets into the shared memory (the same in every CTA)
struct __align__(16) ClLev {
    int own, col, val, diag;   // constant image: own rows' window indices, matrix,
    int dinv, dst, over, head; //   1 / a_ii, destinations (and further ones), ClHead
    int lg, ns;        // log2 of the lanes per row; off-diagonal slots a lane takes (even)
    int R;             // stride of the matrix tables (largest strip's rows times lanes)
    int kind;          // 1: a child of an own next-level row may lie in another strip; 2: the
                       //   finest level (block smoother)
    int pre, post, npre, npost;  // sweeps (ClOp) and their lengths
    int parent, child, nch, Rn;  // maps; children per row of the next level's rows, stride
    int rhs, r, e, nact;       // vectors: by own row, by window index; warps with rows in sums
    int p[kMaxKcycle], q[kMaxKcycle];
    int level, ncol, w, blk;   // blk: finest level, first own row of each own block
};

struct ClLayout {
    int nsp;           // swept levels: tl .. tl + nsp - 1; the dense level follows
    int tl;
    int dense;         // 1: M and A M of the level above the coarsest, 0: coarsest inverse
    int kc, nu_pre, nu_post;
    int nd, ch, stride;  // dense level: rows, rows per CTA (multiple of 4), row stride
    int mat, mat_lo;     // M, FP32: then A M (or the inverse); FP32: M's (the inverse's) low parts
    int aw, aval, acol;  // > 0: M alone, and A's rows: slots per row, values, columns (FP32: in the
                         //   image beyond what is copied)
    int dhead, down;     // gather into the dense level: own rows (count; their pi-rows)
    int peers;           // neighbour CTAs: count, ranks
    int levels;          // lv[] (a copy in the image)
    int top;             // pi-rows of the top level's own rows
    int F, Rv, E, out, P[kMaxKcycle], Q[kMaxKcycle];  // dense level's vectors (every CTA: all)
    int stage;           // one value per own row of the dense level
    int image_bytes, image_stride, bytes;  // copied; one CTA's; shared memory
    ClLev lv[kClLevels];
};

template <class T>
struct ClArgs {
    ClLayout y;
    const unsigned char *image;  // [kClRanks][image_stride]
    const T *rhs;                // level tl, pi order
    T *e;
    int *err;
    unsigned long long limit_ns;
    int extra;                   // host-set fault: bytes the first wait expects too many
    unsigned long long *ts;      // end timestamp (profiling) or null
    unsigned long long *tprof;   // cycles and counts per (level, kind) or null
};

// ---------------------------------------------------------------------------------------
// cluster primitives
__device__ __forceinline__ uint32_t cl_smem(const void *p) {
    return (uint32_t)__cvta_generic_to_shared(p);
}
// shared memory by 32-bit address: a load is one instruction and an address one add (through
// generic pointers each address is a 64-bit sum)
__device__ __forceinline__ void cl_lds(uint32_t a, float &v) {
    asm volatile("ld.shared.f32 %0, [%1];" : "=f"(v) : "r"(a) : "memory");
}
__device__ __forceinline__ void cl_lds(uint32_t a, double &v) {
    asm volatile("ld.shared.f64 %0, [%1];" : "=d"(v) : "r"(a) : "memory");
}
__device__ __forceinline__ void cl_lds(uint32_t a, int &v) {
    asm volatile("ld.shared.s32 %0, [%1];" : "=r"(v) : "r"(a) : "memory");
}
__device__ __forceinline__ void cl_lds(uint32_t a, unsigned short &v) {
    asm volatile("ld.shared.u16 %0, [%1];" : "=h"(v) : "r"(a) : "memory");
}
__device__ __forceinline__ void cl_lds(uint32_t a, uint2 &v) {
    asm volatile("ld.shared.v2.u32 {%0, %1}, [%2];" : "=r"(v.x), "=r"(v.y) : "r"(a) : "memory");
}
__device__ __forceinline__ void cl_lds(uint32_t a, uint4 &v) {
    asm volatile("ld.shared.v4.u32 {%0, %1, %2, %3}, [%4];"
                 : "=r"(v.x), "=r"(v.y), "=r"(v.z), "=r"(v.w) : "r"(a) : "memory");
}
__device__ __forceinline__ void cl_lds(uint32_t a, float4 &v) {
    asm volatile("ld.shared.v4.f32 {%0, %1, %2, %3}, [%4];"
                 : "=f"(v.x), "=f"(v.y), "=f"(v.z), "=f"(v.w) : "r"(a) : "memory");
}
__device__ __forceinline__ void cl_lds(uint32_t a, double2 &v) {
    asm volatile("ld.shared.v2.f64 {%0, %1}, [%2];" : "=d"(v.x), "=d"(v.y) : "r"(a) : "memory");
}
template <class V>
__device__ __forceinline__ V cl_ld(uint32_t a) {
    V v;
    cl_lds(a, v);
    return v;
}
__device__ __forceinline__ void cl_st(uint32_t a, float v) {
    asm volatile("st.shared.f32 [%0], %1;" ::"r"(a), "f"(v) : "memory");
}
__device__ __forceinline__ void cl_st(uint32_t a, double v) {
    asm volatile("st.shared.f64 [%0], %1;" ::"r"(a), "d"(v) : "memory");
}
__device__ __forceinline__ uint32_t cl_map(uint32_t addr, int rank) {
    uint32_t o;
    asm("mapa.shared::cluster.u32 %0, %1, %2;" : "=r"(o) : "r"(addr), "r"(rank));
    return o;
}
__device__ __forceinline__ void cl_store(uint32_t a, float v, uint32_t mb) {
    asm volatile("st.async.shared::cluster.mbarrier::complete_tx::bytes.f32 [%0], %1, [%2];" ::"r"(a),
                 "f"(v), "r"(mb) : "memory");
}
__device__ __forceinline__ void cl_store(uint32_t a, double v, uint32_t mb) {
    asm volatile("st.async.shared::cluster.mbarrier::complete_tx::bytes.f64 [%0], %1, [%2];" ::"r"(a),
                 "d"(v), "r"(mb) : "memory");
}
// the same where `on` (no branch: a branch costs a warp as much as a few instructions)
__device__ __forceinline__ void cl_store_if(bool on, uint32_t a, float v, uint32_t mb) {
    asm volatile(
        "{\n.reg .pred p;\nsetp.ne.u32 p, %3, 0;\n"
        "@p st.async.shared::cluster.mbarrier::complete_tx::bytes.f32 [%0], %1, [%2];\n}" ::"r"(a),
        "f"(v), "r"(mb), "r"((unsigned)on) : "memory");
}
__device__ __forceinline__ void cl_store_if(bool on, uint32_t a, double v, uint32_t mb) {
    asm volatile(
        "{\n.reg .pred p;\nsetp.ne.u32 p, %3, 0;\n"
        "@p st.async.shared::cluster.mbarrier::complete_tx::bytes.f64 [%0], %1, [%2];\n}" ::"r"(a),
        "d"(v), "r"(mb), "r"((unsigned)on) : "memory");
}
__device__ __forceinline__ void cl_st_if(bool on, uint32_t a, float v) {
    asm volatile("{\n.reg .pred p;\nsetp.ne.u32 p, %2, 0;\n@p st.shared.f32 [%0], %1;\n}" ::"r"(a), "f"(v),
                 "r"((unsigned)on) : "memory");
}
__device__ __forceinline__ void cl_st_if(bool on, uint32_t a, double v) {
    asm volatile("{\n.reg .pred p;\nsetp.ne.u32 p, %2, 0;\n@p st.shared.f64 [%0], %1;\n}" ::"r"(a), "d"(v),
                 "r"((unsigned)on) : "memory");
}
__device__ __forceinline__ void cl_store16(uint32_t a, const float *v, uint32_t mb) {
    const float4 x = *reinterpret_cast<const float4 *>(v);
    asm volatile(
        "st.async.shared::cluster.mbarrier::complete_tx::bytes.v4.f32 [%0], {%1, %2, %3, %4}, [%5];" ::"r"(a),
        "f"(x.x), "f"(x.y), "f"(x.z), "f"(x.w), "r"(mb) : "memory");
}
__device__ __forceinline__ void cl_store16(uint32_t a, const double *v, uint32_t mb) {
    const double2 x = *reinterpret_cast<const double2 *>(v);
    asm volatile(
        "st.async.shared::cluster.mbarrier::complete_tx::bytes.v2.f64 [%0], {%1, %2}, [%3];" ::"r"(a),
        "d"(x.x), "d"(x.y), "r"(mb) : "memory");
}
__device__ __forceinline__ void cl_mb_init(uint32_t mb, int count) {
    asm volatile("mbarrier.init.shared::cta.b64 [%0], %1;" ::"r"(mb), "r"(count) : "memory");
}
__device__ __forceinline__ void cl_mb_arrive_if(bool on, uint32_t mb) {
    asm volatile("{\n.reg .pred p;\nsetp.ne.u32 p, %1, 0;\n@p mbarrier.arrive.shared::cta.b64 _, [%0];\n}" ::"r"(mb),
                 "r"((unsigned)on) : "memory");
}
__device__ __forceinline__ void cl_mb_expect_if(bool on, uint32_t mb, int bytes) {
    asm volatile(
        "{\n.reg .pred p;\nsetp.ne.u32 p, %2, 0;\n@p mbarrier.arrive.expect_tx.shared::cta.b64 _, [%0], %1;\n}" ::"r"(mb),
        "r"(bytes), "r"((unsigned)on) : "memory");
}
__device__ __forceinline__ void cl_mb_expect(uint32_t mb, int bytes) {
    asm volatile("mbarrier.arrive.expect_tx.shared::cta.b64 _, [%0], %1;" ::"r"(mb), "r"(bytes)
                 : "memory");
}
__device__ __forceinline__ bool cl_mb_try(uint32_t mb, unsigned parity) {
    unsigned ok;
    asm volatile(
        "{\n.reg .pred p;\n"
        "mbarrier.try_wait.parity.acquire.cluster.shared::cta.b64 p, [%1], %2;\n"
        "selp.u32 %0, 1, 0, p;\n}" : "=r"(ok) : "r"(mb), "r"(parity) : "memory");
    return ok != 0;
}
__device__ __forceinline__ void cl_sync_all() {
    asm volatile("barrier.cluster.arrive.release;\nbarrier.cluster.wait.acquire;" ::: "memory");
}

// bounded wait: after limit_ns (or once another thread of the CTA gave up) false
__device__ __noinline__ bool cl_wait_slow(uint32_t mb, unsigned parity, volatile int *gave_up,
                                          int *err, unsigned long long limit_ns) {
    const unsigned long long t0 = global_ns();
    for (;;) {
        for (int k = 0; k < 64; k++)
            if (cl_mb_try(mb, parity)) return true;
        if (*gave_up) return false;
        if (global_ns() - t0 > limit_ns) {
            atomicOr(err, kErrTimeout);
            *gave_up = 1;
            return false;
        }
    }
}

// A CTA of which a wait ran out, once every CTA has stopped sending: what was under way to its
// shared memory lands before it leaves. Its image is counted (again with a limit). The stores of
// an exchange that never completes are not; one takes about 400 cycles, so 100 us are ample.
__device__ __noinline__ void cl_drain(uint32_t image_mb) {
    const unsigned long long t0 = global_ns();
    while (!cl_mb_try(image_mb, 0) && global_ns() - t0 < kBarrierLimitNs) {}
    while (global_ns() - t0 < 100000) {}
}

// a / b out of line, for the rare case (the kernel's code is larger than an SM's instruction cache)
__device__ __noinline__ double cl_quotient(double a, double b) { return a / b; }

// At these sizes a step is a few dozen instructions per thread, each about 4-5 cycles after the
// one before, so what counts is the number of instructions between the end of one wait and
// the stores that end the next. A row's constants (its columns' addresses, values, 1 / a_ii,
// its destinations' addresses) are therefore read into registers before the wait of the step
// before it, so that only the gathers of z, f and the sum follow the wait; level constants
// stay in registers, stores are predicated rather than branched around. One Gauss-Seidel
// colour, exchange included: 0.59-0.80 us with each step's code in line and no read ahead,
// 1.1-1.5 us as an interpreter of ops with all bodies in one loop, 0.40 us in this form
// (FP64: 0.91-0.98 -> 0.63-0.75 us). All levels from 16,384 rows down, 2 Alg. 1 steps each,
// 1.05M unknowns, FP32: 127 us per visit (8 per application); on one CTA the levels from
// 4,096 rows down took 139-150 us (16 per application) and the level above 3.0 us per step.
extern __shared__ __align__(16) unsigned char cl_dyn[];

template <class T>
__global__ void __launch_bounds__(kClThreads, 1)
k_cluster_tail(const __grid_constant__ ClArgs<T> a) {
    constexpr bool F64 = sizeof(T) == 8;
    constexpr int NR = kClRanks;
    __shared__ __align__(8) unsigned long long mbs[5];   // neighbours x 2, all CTAs x 2, image
    __shared__ __align__(16) T red[2][NR * kClWarps][2]; // sums over the cluster: the warps'
    __shared__ T coef_s[6];
    __shared__ T pqs[kClLevels + 1][kMaxKcycle];         // (p_i, A p_i) of every level
    __shared__ T inv_s[F64 ? kClLevels + 1 : 1][kMaxKcycle][2];  // FP64: its reciprocal, two parts
    __shared__ int stops[kClLevels + 1][kMaxKcycle];     // Alg. 1 stopped at or before step i
    __shared__ int gave_up_s, token;
    volatile int *gave_up = &gave_up_s;
    const ClLayout &y = a.y;
    const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
    int rank;
    asm("mov.u32 %0, %%cluster_ctarank;" : "=r"(rank));
    const uint32_t mb0 = cl_smem(mbs), dyn = cl_smem(cl_dyn);
    if (tid == 0) {
        for (int k = 0; k < 4; k++) cl_mb_init(mb0 + 8 * k, kClWarps);
        cl_mb_init(mb0 + 32, 1);
        asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
        gave_up_s = 0;
        token = 0;
    }
    __syncthreads();
    if (tid == 0) {  // this CTA's constant image, one bulk copy
        cl_mb_expect(mb0 + 32, y.image_bytes);
        asm volatile(
            "cp.async.bulk.shared::cluster.global.mbarrier::complete_tx::bytes [%0], [%1], %2, [%3];" ::"r"(dyn),
            "l"(a.image + (size_t)rank * y.image_stride), "r"(y.image_bytes), "r"(mb0 + 32)
            : "memory");
    }
    cl_sync_all();  // every CTA's mbarriers are ready
    bool alive = cl_mb_try(mb0 + 32, 0) || cl_wait_slow(mb0 + 32, 0, gave_up, a.err, kBarrierLimitNs);
    // launched before the end of the kernel before it (its writes can be seen from here on);
    // nothing above depends on that one, and the one after this waits in the same way
    asm volatile("griddepcontrol.launch_dependents;");
    asm volatile("griddepcontrol.wait;" ::: "memory");
    if (!__syncthreads_and(alive)) {  // no image: the others give up at their first exchange
        cl_sync_all();
        cl_drain(mb0 + 32);
        return;
    }
    // after an error of an earlier launch of this application the steps run without exchanges
    alive = !(ld_volatile_int(a.err) & kErrTimeout);
    unsigned kn = 0, ka = 0;  // exchanges so far: neighbours, all CTAs
    int extra = a.extra;
    auto at = [&](int off) { return cl_dyn + off; };
    const ClLev *lvs = (const ClLev *)at(y.levels);
    auto vec = [&](int off) { return (T *)(cl_dyn + off); };
    const int npeer = ((const int *)at(y.peers))[0];
    // a token for every neighbour: lane p of the last warp
    const bool has_peer = warp == kClWarps - 1 && lane < npeer;
    const int peer = has_peer ? ((const int *)at(y.peers))[1 + lane] : 0;
    const uint32_t peer_tok = cl_map(cl_smem(&token), peer), peer_mb = cl_map(mb0, peer);
    long long tp0 = 0;
    const bool mark_on = a.tprof && rank == 0 && tid == 0;
    // profiling: cycles and count per (level, kind); in global memory, as 1.3 KB of shared memory can
    // cost a level its place (97^2 nodes, kcycle_n = 4, FP64: 644 -> 1,079 us per application)
    if (mark_on) tp0 = clock64();
    auto mark = [&](int slot_level, int kind) {
        if (!mark_on) return;
        const long long t1 = clock64();
        const int slot = 16 * (y.tl + slot_level) + kind;
        atomicAdd(&a.tprof[slot], (unsigned long long)(t1 - tp0));
        atomicAdd(&a.tprof[16 * kMaxLevels + slot], 1ull);
        tp0 = t1;
    };
    // this CTA's arrivals at mbarrier mb, which counts its warps and `bytes` of stores (the last
    // warp, which seldom has rows, announces them)
    auto arrive = [&](uint32_t mb, int bytes) {
        __syncwarp();
        const bool one = alive && lane == 0;
        cl_mb_expect_if(one && warp == kClWarps - 1, mb, bytes + extra);
        cl_mb_arrive_if(one && warp != kClWarps - 1, mb);
        extra = 0;
    };
    auto wait = [&](uint32_t mb, unsigned k) {
        if (alive && !cl_mb_try(mb, (k >> 1) & 1))
            alive = cl_wait_slow(mb, (k >> 1) & 1, gave_up, a.err, a.limit_ns);
    };
    // neighbour exchange kn: this CTA's end of its stores; `bytes` of rows come in
    auto arrive_n = [&](int bytes) {
        const uint32_t par = 8 * (kn & 1);
        cl_store_if(has_peer && alive, peer_tok, 0.f, peer_mb + par);
        arrive(mb0 + par, bytes + 4 * npeer);
    };
    auto wait_n = [&]() {
        wait(mb0 + 8 * (kn & 1), kn);
        kn++;
    };
    auto mb_a = [&]() { return mb0 + 16 + 8 * (ka & 1); };
    auto wait_a = [&]() {
        wait(mb_a(), ka);
        ka++;
    };

    int lv = 0;                    // current swept level
    unsigned long long steps = 0;  // Alg. 1 step of every swept level, 4 bits each
    // the destinations as addresses: (place, mbarrier) of two, mapped once
    for (int l = 0; l < y.nsp; l++) {
        int last = 0;  // (index checks: the level's last window vector)
#ifdef AMG_BOUNDS_CHECK
        last = lvs[l].e;
        for (int k = 0; k < kMaxKcycle; k++) last = max(last, max(lvs[l].p[k], lvs[l].q[k]));
#endif
        uint4 *d = (uint4 *)at(lvs[l].dst);
        const int nown = ((const ClHead *)at(lvs[l].head))->nown;
#pragma unroll 1
        for (int m = tid; m < nown; m += kClThreads) {
            uint4 q = d[m];
            auto place = [&](unsigned &p, unsigned &b) {
                if (p >> 31 || p == kClNone) return;  // further ones: stays as it is
                if (!idx_ok((int)(p >> 16), NR) || !idx_ok(last + (int)(p & 0xFFFFu), y.bytes)) {
                    p = kClNone;
                    return;
                }
                b = cl_map(mb0, (int)(p >> 16));
                p = cl_map(dyn, (int)(p >> 16)) + (p & 0xFFFFu);
            };
            place(q.x, q.y);
            place(q.z, q.w);
            d[m] = q;
        }
    }
    __syncthreads();
    // ---- the level's constants ----------------------------------------------------------
    // (in registers: every wait and store makes the compiler read shared memory again)
    uint4 lt0{}, lt1{}, lt2{};  // ClLev: own, col, val, diag | dinv, dst, over, head | lg, ns, R, kind
    uint4 h0{}, h1{};           // ClHead: nown, nwin, expect_all, fexp | fc0, fcn, fs0, fs1
    uint32_t lvb = cl_smem(lvs);  // its ClLev
    auto bind = [&](int l) {
        lvb = cl_smem(&lvs[l]);
        lt0 = cl_ld<uint4>(lvb);
        lt1 = cl_ld<uint4>(lvb + 16);
        lt2 = cl_ld<uint4>(lvb + 32);
        h0 = cl_ld<uint4>(dyn + lt1.w);
        h1 = cl_ld<uint4>(dyn + lt1.w + 16);
    };
    auto field = [&](size_t off) { return cl_ld<int>(lvb + (uint32_t)off); };
#define CL_F(name) field(offsetof(ClLev, name))
    auto p_off = [&](int i) { return field(offsetof(ClLev, p) + 4 * i); };
    auto q_off = [&](int i) { return field(offsetof(ClLev, q) + 4 * i); };
    // ---- a row's constants ------------------------------------------------------------
    int mi = 0;                        // own row
    uint32_t lb = 0;                   // its byte offset in a window vector
    uint32_t d0 = 0, d1 = 0;           // its place in two strips' windows,
    uint32_t m0 = 0, m1 = 0;           //   their mbarriers of the exchange it is sent in
    bool to0 = false, to1 = false;     //   if any
    unsigned more = 0;                 // further ones: bit 31 and their list
    bool has = false, own = false;     // this lane has a row; is the one that stores it
    T dinv = 0, dg = 0, v[kClSlots];
    uint32_t za[kClSlots];             // addresses of its columns in z
#pragma unroll
    for (int k = 0; k < kClSlots; k++) {
        v[k] = T(0);
        za[k] = dyn;
    }
    // destinations of own row m (if on) for the vector at `off`, in neighbour exchange kx
    auto load_dst = [&](bool on, int m, int off, unsigned kx) {
        const uint4 q = cl_ld<uint4>(dyn + lt1.y + 16 * m);
        const uint32_t par = 8 * (kx & 1);
        on = on && alive;
        to0 = on && q.x != kClNone;
        to1 = on && (int)q.z >= 0 && q.z != kClNone;
        more = on && q.z >> 31 ? q.z : 0;
        d0 = q.x + (uint32_t)off;
        m0 = q.y + par;
        d1 = q.z + (uint32_t)off;
        m1 = q.w + par;
    };
    // row vr of rows [vr0, vr0 + cnt) (times lanes per row): this thread's; its products are
    // with the vector at zoff, its new value goes to the one at doff in exchange kx. A lane
    // without a row takes row 0 and stores nothing: no branches
    auto load_row = [&](int vr0, int vr, int cnt, int zoff, int doff, unsigned kx) {
        has = vr < cnt;
        const int o = has ? vr0 + vr : 0, m = o >> lt2.x;
        mi = m;
        own = has && (o & ((1 << lt2.x) - 1)) == 0;
        lb = cl_ld<unsigned short>(dyn + lt0.x + 2 * m);
        if (has && !idx_ok((int)lb, (int)sizeof(T) * (int)h0.y)) lb = 0;
        const uint4 c = cl_ld<uint4>(dyn + lt0.y + 16 * o);
        dg = cl_ld<T>(dyn + lt0.w + (int)sizeof(T) * m);
        if constexpr (!F64) {
            const float4 x0 = cl_ld<float4>(dyn + lt0.z + 16 * o),
                         x1 = cl_ld<float4>(dyn + lt0.z + 16 * ((int)lt2.z + o));
            v[0] = x0.x; v[1] = x0.y; v[2] = x0.z; v[3] = x0.w;
            v[4] = x1.x; v[5] = x1.y; v[6] = x1.z; v[7] = x1.w;
        } else {
#pragma unroll
            for (int k = 0; k < 4; k++)
                if (2 * k < (int)lt2.y) {
                    const double2 x = cl_ld<double2>(dyn + lt0.z + 16 * (k * (int)lt2.z + o));
                    v[2 * k] = x.x;
                    v[2 * k + 1] = x.y;
                }
        }
        const unsigned cw[4] = {c.x, c.y, c.z, c.w};
        const uint32_t zb = dyn + zoff;
#pragma unroll
        for (int k = 0; k < kClSlots; k++) za[k] = zb + ((k & 1) ? cw[k / 2] >> 16 : cw[k / 2] & 0xFFFFu);
        dinv = cl_ld<T>(dyn + lt1.x + (int)sizeof(T) * m);
        load_dst(own, m, doff, kx);
    };
    // Item `item` of [x0, x0 + cnt) of a sweep's colour: a row (times lanes), or on the finest level a
    // block, whose rows are taken in ascending (backward: descending) order: the first row is
    // read, `rest` more follow
    int rest = 0;
    auto load_item = [&](int x0, int item, int cnt, bool bwd, int blk, int zoff, unsigned kx) {
        if (blk == 0) {
            load_row(x0, item, cnt, zoff, zoff, kx);
            return;
        }
        const bool on = item < cnt;
        const uint32_t b = dyn + blk + 2 * (on ? x0 + item : 0);
        const int s = cl_ld<unsigned short>(b), e = cl_ld<unsigned short>(b + 2);
        rest = on ? e - s - 1 : 0;
        load_row(bwd ? e - 1 : s, 0, on, zoff, zoff, kx);
    };
    // off-diagonal part of the row's product with z, over its lanes
    auto gather = [&](int k) {
#ifdef AMG_BOUNDS_CHECK
        if (!idx_ok((int)(za[k] - dyn), y.bytes)) return T(0);
#endif
        return cl_ld<T>(za[k]);
    };
    auto row_dot = [&]() {
        T acc;
        if constexpr (!F64) {
            T x[kClSlots];
#pragma unroll
            for (int k = 0; k < kClSlots; k++) x[k] = gather(k);
            T s0 = v[0] * x[0], s1 = v[1] * x[1];
#pragma unroll
            for (int k = 2; k < kClSlots; k += 2) {
                s0 += v[k] * x[k];
                s1 += v[k + 1] * x[k + 1];
            }
            acc = s0 + s1;
        } else {
            // one FP64 instruction of a warp takes 64 cycles whatever its lanes do: no more of
            // them than the level's slots need
            acc = T(0);
            auto part = [&](auto k0, auto k1) {
                T x[kClSlots];
#pragma unroll
                for (int k = decltype(k0)::value; k < decltype(k1)::value; k++) x[k] = gather(k);
#pragma unroll
                for (int k = decltype(k0)::value; k < decltype(k1)::value; k++)
                    acc = k == 0 ? v[0] * x[0] : acc + v[k] * x[k];
            };
            using std::integral_constant;
            if (lt2.y > 4) part(integral_constant<int, 0>{}, integral_constant<int, 8>{});
            else if (lt2.y > 2) part(integral_constant<int, 0>{}, integral_constant<int, 4>{});
            else part(integral_constant<int, 0>{}, integral_constant<int, 2>{});
        }
        if (lt2.x > 0) {
            acc += __shfl_xor_sync(0xffffffffu, acc, 1);
            if (lt2.x > 1) acc += __shfl_xor_sync(0xffffffffu, acc, 2);
        }
        return acc;
    };
    // the row's new value to the strips that hold the row
    auto push = [&](int off, T u) {
        cl_store_if(to0, d0, u, m0);
        cl_store_if(to1, d1, u, m1);
        if (more) {
            const uint32_t par = 8 * (kn & 1);
            const unsigned *list = (const unsigned *)at(lt1.z) + (more & 0x7FFFFFFFu);
#pragma unroll 1
            for (unsigned d = *list; d != kClNone; d = *++list)
                if (idx_ok((int)(d >> 16), NR) && idx_ok(off + (int)(d & 0xFFFFu), y.bytes))
                    cl_store(cl_map(dyn + off + (d & 0xFFFFu), (int)(d >> 16)), u,
                         cl_map(mb0 + par, (int)(d >> 16)));
        }
    };
    // checking build: this warp is late now and then (chosen by CTA, warp and exchange)
    auto perhaps_late = [&] {
#ifdef AMG_BOUNDS_CHECK
        if ((5 * rank + 3 * warp + 7 * (int)(kn + ka)) % 11 < 4) __nanosleep(4000);
#endif
    };
    // z = 0 on the window, except the colour whose values come next
    auto zero_window = [&](uint32_t z) {  // of the level bound
        perhaps_late();
#pragma unroll 1
        for (unsigned k = tid; k < h0.y; k += kClThreads)
            if (k < h1.z || k >= h1.w) cl_st(z + (uint32_t)sizeof(T) * k, T(0));
    };
    // Gauss-Seidel sweeps over n colours; the first one's rows are loaded already. The rows of
    // the step after the sweep (all own rows of the level; sent, if at all, to the vector at
    // next_off in the next exchange) are loaded before its last wait.
    auto sweep = [&](int ops, int n, bool bwd, int foff, int zoff, int next_cnt, int next_off) {
        const uint32_t z = dyn + zoff, f = dyn + foff;
        const int blk = lt2.w == 2 ? CL_F(blk) : 0;
        uint4 op = cl_ld<uint4>(dyn + ops);  // a ClOp
#pragma unroll 1
        for (int k = 0; k < n; k++) {
            perhaps_late();
            auto relax = [&] {
                const T fi = cl_ld<T>(f + (uint32_t)sizeof(T) * mi);
                const T u = (fi - row_dot()) * dinv;
                push(zoff, u);
                cl_st_if(own, z + lb, u);
            };
            auto rest_of_block = [&] {
#pragma unroll 1
                for (; rest > 0; rest--) {
                    load_row(bwd ? mi - 1 : mi + 1, 0, 1, zoff, zoff, kn);
                    relax();
                }
            };
            // (a warp without rows goes on at once)
            if (32 * warp < (int)op.y) relax();
            if (blk) rest_of_block();
#pragma unroll 1
            for (int c = kClThreads; c < (int)op.y; c += kClThreads) {  // strips of large levels
                load_item(op.x, c + tid, op.y, bwd, blk, zoff, kn);
                if (c + 32 * warp < (int)op.y) relax();
                if (blk) rest_of_block();
            }
            arrive_n(op.z);
            if (k + 1 < n) {
                op = cl_ld<uint4>(dyn + ops + 16 * (k + 1));
                load_item(op.x, tid, op.y, bwd, blk, zoff, kn + 1);
            } else {
                load_row(0, tid, next_cnt, zoff, next_off, kn + 1);
            }
            wait_n();
            mark(lv, OP_GS);
        }
    };
    // Sums of s0 and s1 over the cluster, then the coefficient f(sums) in every thread. Lanes 0-15
    // end with the first sum, 16-31 with the second (one add per step for both); every warp
    // sends its sums to every CTA. FP32: every warp adds them up; FP64 (scarce): warp 0, and
    // warp 1 beside it for what only later steps read (g).
    auto half_sum = [&](T x, T y) {
        const bool hi = lane >= 16;
        T k = hi ? y : x;
        const T other = hi ? x : y;
        k += __shfl_xor_sync(0xffffffffu, other, 16);
#pragma unroll
        for (int o = 8; o > 0; o >>= 1) k += __shfl_xor_sync(0xffffffffu, k, o);
        return k;
    };
    auto cluster_sum = [&](T s0, T s1, int nact, auto before_wait, auto f, auto g) {
        const uint32_t mb = mb_a(), part = cl_smem(&red[ka & 1][0][0]);
        if (warp < nact) {
            const T k = half_sum(s0, s1);
            if (alive)
                cl_store(cl_map(part + (uint32_t)sizeof(T) * (2 * (rank * nact + warp) + (lane >> 4)), lane & (NR - 1)),
                         k, cl_map(mb, lane & (NR - 1)));
        }
        perhaps_late();
#ifdef AMG_BOUNDS_CHECK
        if (npeer == 0) __nanosleep(100000);  // held back by nothing but the sums and gathers
#endif
        arrive(mb, NR * nact * 2 * (int)sizeof(T));
        before_wait();
        wait_a();
        T c = 0;
        if (!F64 || warp < 2) {
            const uint32_t mine = part + (uint32_t)sizeof(T) * (2 * (lane & (NR - 1)) * nact + (lane >> 4));
            T k = cl_ld<T>(mine);
#pragma unroll 1
            for (int w2 = 1; w2 < nact; w2++) k += cl_ld<T>(mine + 2 * (uint32_t)sizeof(T) * w2);
#pragma unroll
            for (int o = 8; o > 0; o >>= 1) k += __shfl_xor_sync(0xffffffffu, k, o);
            const T other = __shfl_xor_sync(0xffffffffu, k, 16);
            s0 = lane < 16 ? k : other;
            s1 = lane < 16 ? other : k;
            if constexpr (!F64) {
                c = f(s0, s1);
                g(s0);
            } else if (warp == 0) {
                c = f(s0, s1);
                if (lane == 0) coef_s[0] = c;
            } else {
                g(s0);
            }
        }
        if constexpr (F64) {
            __syncthreads();
            c = coef_s[0];
        }
        return c;
    };
    // positive and finite (FP64 without FP64 comparisons)
    auto positive = [](T x) {
        if constexpr (F64) return (unsigned long long)__double_as_longlong(x) - 1 < 0x7FEFFFFFFFFFFFFFull;
        else return x > T(0) && isfinite(x);
    };
    // Alg. 1 on level slot lv: alpha_i from (p_i, q_i) and (r_i, p_i), 0 once it has stopped (a
    // zero residual stops it here too: its p_i and q_i are zero); what step i leaves to later
    // ones; beta_ij from (z, q_j)
    auto alpha = [&](int lv, int i, T pq, T rp) {
        const bool stopped = (i > 0 && stops[lv][i - 1]) || !positive(pq);
        if (tid == 0) stops[lv][i] = stopped;
        return stopped ? T(0) : (T)ratio<T>((double)rp, (double)pq);
    };
    // FP64: a division takes about 560 cycles, so 1 / pq is kept, off the path to the next step, as
    // a sum of two doubles (error of about 2^-106): zq / pq is then a product and an FMA, rounded
    // once but for 2^-53 of a rounding. Only where neither part leaves the normal range (pq of 2^-960
    // to 2^960); elsewhere (0 here) a division. Every beta by a division, 257^2 nodes: 6.13 -> 6.22 ms
    // per solve; in this form 6.19 (by 1 / pq alone, rounded twice and infinite for a subnormal
    // pq, 6.13).
    auto keep_pq = [&](int lv, int i, T pq) {
        if (tid != (F64 ? 32 : 0)) return;
        pqs[lv][i] = pq;
        if constexpr (F64) {
            const unsigned long long e = (unsigned long long)__double_as_longlong(pq) >> 52;
            const bool ok = e - (1023 - 960) <= 2 * 960;  // sign bit clear: positive
            const T k = ok ? T(1) / pq : T(0);
            inv_s[lv][i][0] = k;
            inv_s[lv][i][1] = ok ? k * fma(-k, pq, T(1)) : T(0);
        }
    };
    auto beta = [&](int lv, int j, T zq) {
        if constexpr (F64) {
            const T k = inv_s[lv][j][0], k2 = inv_s[lv][j][1];
            if (__double_as_longlong(k) != 0) return -fma(zq, k, zq * k2);
        }
        const T pq = pqs[lv][j];
        if constexpr (F64) return positive(pq) ? -cl_quotient(zq, pq) : T(0);
        else return positive(pq) ? -(T)ratio<T>((double)zq, (double)pq) : T(0);
    };
    auto nothing = [] {};
    auto no_pq = [](T) {};

    // ---- entry ---------------------------------------------------------------------------
    {  // dense level's right-hand side: zero beyond its rows
        T *F = vec(y.F);
#pragma unroll 1
        for (int k = tid; k < NR * y.ch; k += kClThreads)
            F[k] = (y.nsp == 0 && k < y.nd) ? __ldcg(&a.rhs[k]) : T(0);
    }
    // the first colour of a sweep from zero: own row m, right-hand side x (z zeroed before)
    auto first_colour = [&](int m, int zoff, T x) {
        if ((unsigned)(m - (int)h1.x) < h1.y) {
            const T u = x * cl_ld<T>(dyn + lt1.x + (uint32_t)sizeof(T) * m);
            lb = cl_ld<unsigned short>(dyn + lt0.x + 2 * m);
            load_dst(true, m, zoff, kn);
            push(zoff, u);
            cl_st(dyn + zoff + lb, u);
        }
    };
    // its exchange; the sweep's next colour (or all rows) is loaded before the wait
    auto first_exchange = [&](int zoff, int qoff) {
        arrive_n((int)h0.w);
        const int npre = CL_F(npre);
        const uint4 op = cl_ld<uint4>(dyn + CL_F(pre));
        if (lt2.w == 2) load_item(op.x, tid, op.y, false, CL_F(blk), zoff, kn + 1);
        else load_row(npre ? op.x : 0, tid, npre ? op.y : h0.x << lt2.x, zoff, npre ? zoff : qoff, kn + 1);
        wait_n();
    };
    if (y.nsp > 0) {  // this strip's rows of the right-hand side, and their first colour
        bind(0);
        const int zoff = p_off(0), roff = CL_F(rhs);
        zero_window(dyn + zoff);
#pragma unroll 1
        for (int m = tid; m < (int)h0.x; m += kClThreads) {
            const T x = __ldcg(&a.rhs[((const int *)at(y.top))[m]]);
            vec(roff)[m] = x;
            first_colour(m, zoff, x);
        }
        __syncthreads();  // every warp's zeros, before the neighbours may send what they leave out
        first_exchange(zoff, q_off(0));
        mark(0, OP_GS_FIRST);
    }
    __syncthreads();

    // ---- Alg. 2 / Alg. 1 over the levels ------------------------------------------------
    for (;;) {
        if (y.nsp > 0) {  // B^ of level lv for step i: pre-smoothing, then the restriction
            const int i = (int)(steps >> (4 * lv)) & 15;
            const int foff = i == 0 ? CL_F(rhs) : CL_F(r), zoff = p_off(i), toff = q_off(i);
            const int rows = (int)(h0.x << lt2.x), npre = CL_F(npre);
            if (npre > 0) sweep(CL_F(pre), npre, false, foff, zoff, rows, toff);
            const bool to_swept = lv + 1 < y.nsp;
            const int child = CL_F(child), nch = CL_F(nch), Rn = CL_F(Rn);
            const bool xchild = lt2.w == 1;
            const uint32_t blk = lt2.w == 2 ? dyn + CL_F(blk) : 0, own0 = dyn + lt0.x;
            // t = f - A z into q_i (free until step i's product)
#pragma unroll 1
            for (int c = 0;;) {
                if (c + 32 * warp < rows) {
                    const T fi = cl_ld<T>(dyn + foff + (uint32_t)sizeof(T) * mi), zi = cl_ld<T>(dyn + zoff + lb);
                    const T u = fi - (row_dot() + dg * zi);
                    if (xchild) push(toff, u);
                    cl_st_if(own, dyn + toff + lb, u);
                }
                c += kClThreads;
                if (c >= rows) break;
                load_row(0, c + tid, rows, zoff, toff, kn);
            }
            const int nwin = (int)h0.y;
            if (xchild) arrive_n((int)h0.z);
            int zn = 0;
            if (to_swept) {
                bind(lv + 1);
                zn = p_off(0);
                zero_window(dyn + zn);
            }
            // (the zeros too are complete before the next level's rows come in: the stores
            // of its first colour leave them out, those of later colours wait for this CTA's)
            if (xchild) wait_n();
            __syncthreads();
            mark(lv, OP_RESID);
            const uint32_t t = dyn + toff;
            auto child_sum = [&](int m) {
                if (blk) {  // the finest level: its block m's rows
                    T acc = 0;
                    const int e = cl_ld<unsigned short>(blk + 2 * m + 2);
                    for (int k = cl_ld<unsigned short>(blk + 2 * m); k < e; k++)
                        acc += cl_ld<T>(t + cl_ld<unsigned short>(own0 + 2 * k));
                    return acc;
                }
                T w[2] = {T(0), T(0)};
#pragma unroll
                for (int h = 0; h < 2; h++) {
                    if (h == 1 && nch == 4) break;
                    const uint2 c = cl_ld<uint2>(dyn + child + 8 * (h * Rn + m));
                    const unsigned ci[4] = {c.x & 0xFFFFu, c.x >> 16, c.y & 0xFFFFu, c.y >> 16};
                    T x[4];
#pragma unroll
                    for (int q = 0; q < 4; q++)
                        x[q] = (ci[q] != 0xFFFFu && idx_ok((int)ci[q], nwin))
                                   ? cl_ld<T>(t + (uint32_t)sizeof(T) * ci[q]) : T(0);
                    w[h] = (x[0] + x[1]) + (x[2] + x[3]);
                }
                return w[0] + w[1];
            };
            if (to_swept) {  // its right-hand side and first colour
                const uint32_t rn = dyn + CL_F(rhs);
#pragma unroll 1
                for (int m = tid; m < (int)h0.x; m += kClThreads) {
                    const T x = child_sum(m);
                    cl_st(rn + (uint32_t)sizeof(T) * m, x);
                    first_colour(m, zn, x);
                }
                first_exchange(zn, q_off(0));
                mark(lv, OP_RESTRICT);
                lv++;
                steps &= ~(15ull << (4 * lv));
                continue;
            }
            // into the dense level: every CTA gets every row
            const int nown = *(const int *)at(y.dhead);
            T *stage = vec(y.stage);
#pragma unroll 1
            for (int m = tid; m < nown; m += kClThreads) stage[m] = child_sum(m);
            __syncthreads();
            const unsigned short *pi = (const unsigned short *)at(y.down);
            const uint32_t to = dyn + y.F, mb = mb_a();
            if (alive)
#pragma unroll 1
                for (int k = tid; k < NR * nown; k += kClThreads)
                    if (idx_ok((int)pi[k >> 4], y.nd))
                        cl_store(cl_map(to + (uint32_t)sizeof(T) * pi[k >> 4], k & (NR - 1)), stage[k >> 4],
                                 cl_map(mb, k & (NR - 1)));
            if (warp == kClWarps - 1)
                cl_store_if(alive && lane < NR, cl_map(cl_smem(&token), lane & (NR - 1)), 0.f,
                            cl_map(mb, lane & (NR - 1)));
            arrive(mb, (int)sizeof(T) * y.nd + 4 * NR);
            wait_a();
            mark(lv, OP_RESTRICT);
        }
        // ---- the dense level: E = B~ [F] ------------------------------------------------
        {
            const int ch = y.ch, len = NR * ch;
            T *E = vec(y.E), *out = vec(y.out), *Rv = vec(y.Rv);
            const int nsteps = y.dense ? y.kc : 1, parts = !F64 && y.dense && y.aw == 0 ? 2 : 1;
            constexpr int LPR = 8;  // lanes per row
            constexpr int V = 16 / (int)sizeof(T);
            // FP32: [z; w] = [M; A M] r, 16 lanes per row, 16-byte reads; M r as a compensated sum
            // (Dot2 of Ogita, Rump and Oishi), four of them per lane. Bound by its 11 instructions
            // per entry: 256 rows 3.5 us per visit with M in one float and a plain sum, 3.9 so;
            // 512 rows 5.8, 8.7. The error of one application against FP64, over that of the
            // coarsest inverse in two parts with this level swept (540 right-hand sides, squares,
            // disks, cubes, graded): 1.01 in the mean with one float, 0.985 so
            auto dense_product = [&](const T *r, T *out) {
                if constexpr (!F64) {
                    const float *hi = vec(y.mat), *lo = vec(y.mat_lo), *am = hi + (size_t)ch * y.stride;
                    const int q = tid & 15;
#pragma unroll 1
                    for (int row = tid >> 4; row < ch; row += kClThreads / 16) {
                        const size_t o = (size_t)row * y.stride;
                        float s[4] = {0.f, 0.f, 0.f, 0.f}, e[4] = {0.f, 0.f, 0.f, 0.f}, w0 = 0.f, w1 = 0.f;
                        auto add = [&](int k, float m, float l, float x) {
                            const float ph = __fmul_rn(m, x);
                            const float pe = fmaf(l, x, fmaf(m, x, -ph));
                            float t2, e2;
                            two_sum(s[k], ph, t2, e2);
                            s[k] = t2;
                            e[k] = __fadd_rn(e[k], __fadd_rn(e2, pe));
                        };
                        auto join = [&](float s1, float e1) {
                            float t2, e2;
                            two_sum(s[0], s1, t2, e2);
                            s[0] = t2;
                            e[0] = __fadd_rn(e[0], __fadd_rn(e1, e2));
                        };
#pragma unroll 2
                        for (int j = 4 * q; j < len; j += 64) {
                            const float4 xv = *(const float4 *)(r + j), hv = *(const float4 *)(hi + o + j),
                                         lv4 = *(const float4 *)(lo + o + j);
                            add(0, hv.x, lv4.x, xv.x);
                            add(1, hv.y, lv4.y, xv.y);
                            add(2, hv.z, lv4.z, xv.z);
                            add(3, hv.w, lv4.w, xv.w);
                            if (parts == 2) {
                                const float4 av = *(const float4 *)(am + o + j);
                                w0 += av.x * xv.x;
                                w1 += av.y * xv.y;
                                w0 += av.z * xv.z;
                                w1 += av.w * xv.w;
                            }
                        }
                        for (int k = 1; k < 4; k++) join(s[k], e[k]);
                        w0 += w1;
#pragma unroll
                        for (int d = 8; d > 0; d >>= 1) {
                            join(__shfl_xor_sync(0xffffffffu, s[0], d), __shfl_xor_sync(0xffffffffu, e[0], d));
                            w0 += __shfl_xor_sync(0xffffffffu, w0, d);
                        }
                        if (q == 0) {
                            out[row] = __fadd_rn(s[0], e[0]);
                            if (parts == 2) out[ch + row] = w0;
                        }
                    }
                }
            };
            // this CTA's rows of a product (in `out`: `parts` times ch values) to every CTA
            auto gather_out = [&](int o0, int o1) {
                __syncthreads();
                const uint32_t mb = mb_a();
                const int per = ch / V;
                if (alive)
#pragma unroll 1
                    for (int k = tid; k < NR * parts * per; k += kClThreads) {
                        const int piece = k >> 4, part = piece >= per, o = (piece - part * per) * V;
                        const uint32_t to = dyn + (part ? o1 : o0) + (uint32_t)sizeof(T) * (rank * ch + o);
                        cl_store16(cl_map(to, k & (NR - 1)), out + part * ch + o, cl_map(mb, k & (NR - 1)));
                    }
                arrive(mb, (int)sizeof(T) * parts * len);
                wait_a();
            };
#pragma unroll 1
            for (int st = 0; st < nsteps; st++) {
                perhaps_late();
                const T *r = st == 0 ? vec(y.F) : Rv;
                const int q = tid & (LPR - 1);
                if constexpr (!F64)
                    if (y.dense) dense_product(r, out);
#pragma unroll 1
                for (int row = tid / LPR; row < (!F64 && y.dense ? 0 : ch); row += kClThreads / LPR) {
                    const T *m = vec(y.mat) + (size_t)row * y.stride;
                    T sum = 0, err = 0;
                    if constexpr (F64) {  // z = M r (or A^{-1} r): 16-byte reads
#pragma unroll 8
                        for (int j = q * V; j < len; j += LPR * V) {
                            const double2 mv = *(const double2 *)(m + j), xv = *(const double2 *)(r + j);
                            sum += mv.x * xv.x;
                            err += mv.y * xv.y;
                        }
                        sum += err;
#pragma unroll
                        for (int o = LPR / 2; o > 0; o >>= 1) sum += __shfl_xor_sync(0xffffffffu, sum, o);
                    } else {  // A^{-1} r in FP32: op_coarse's compensated sum
                        const T *ml = vec(y.mat_lo) + (size_t)row * y.stride;
#pragma unroll 1
                        for (int j = q; j < y.nd; j += LPR) {
                            const float x = r[j];
                            const float ph = __fmul_rn(m[j], x);
                            const float pe = fmaf(ml[j], x, fmaf(m[j], x, -ph));
                            float t2, e2;
                            two_sum(sum, ph, t2, e2);
                            sum = t2;
                            err = __fadd_rn(err, __fadd_rn(e2, pe));
                        }
#pragma unroll
                        for (int o = LPR / 2; o > 0; o >>= 1) {
                            const float so = __shfl_xor_sync(0xffffffffu, sum, o);
                            const float co = __shfl_xor_sync(0xffffffffu, err, o);
                            float t2, e2;
                            two_sum(sum, so, t2, e2);
                            sum = t2;
                            err = __fadd_rn(err, __fadd_rn(co, e2));
                        }
                        sum = __fadd_rn(sum, err);
                    }
                    if (q == 0) out[row] = sum;
                }
                gather_out(y.dense ? y.P[st] : y.E, y.Q[st]);
                if (y.aw > 0) {  // w = A z: four lanes per row
                    const unsigned char *A = F64 ? at(0) : a.image + (size_t)rank * y.image_stride;
                    const T *z = vec(y.P[st]), *av = (const T *)(A + y.aval);
                    const unsigned short *ac = (const unsigned short *)(A + y.acol);
                    const int row = tid >> 2;
                    if (32 * warp < 4 * ch) {
                        T sum = 0;
                        if (row < ch)
#pragma unroll (F64 ? 1 : 4)
                            for (int k = tid & 3; k < y.aw; k += 4) {
                                const int j = ac[k * ch + row];
                                if (idx_ok(j, y.nd)) sum += av[k * ch + row] * z[j];
                            }
                        sum += __shfl_xor_sync(0xffffffffu, sum, 1);
                        sum += __shfl_xor_sync(0xffffffffu, sum, 2);
                        if (row < ch && (tid & 3) == 0) out[row] = sum;
                    }
                    gather_out(y.Q[st], 0);
                }
                if (!y.dense) break;
                // Alg. 1 step st, the same in every CTA: beta_j for j < st, then alpha
                T *p = vec(y.P[st]), *w = vec(y.Q[st]);
                const bool last = st == y.kc - 1;
#pragma unroll 1
                for (int j = 0; j <= st; j++) {
                    const T *qj = vec(y.Q[j]), *pj = vec(y.P[j]);
                    T c = 0;
                    if constexpr (!F64) {  // every warp sums all rows: no barrier
                        T s0 = 0, s1 = 0;
#pragma unroll 2
                        for (int k = 4 * lane; k < len; k += 128) {
                            const float4 pv = *(const float4 *)(p + k), qv = *(const float4 *)(qj + k),
                                         rv = *(const float4 *)(r + k);
                            s0 += pv.x * qv.x; s1 += pv.x * rv.x;
                            s0 += pv.y * qv.y; s1 += pv.y * rv.y;
                            s0 += pv.z * qv.z; s1 += pv.z * rv.z;
                            s0 += pv.w * qv.w; s1 += pv.w * rv.w;
                        }
                        const T k = half_sum(s0, s1), other = __shfl_xor_sync(0xffffffffu, k, 16);
                        s0 = lane < 16 ? k : other;
                        s1 = lane < 16 ? other : k;
                        if (j < st) {
                            c = beta(kClLevels, j, s0);
                        } else {
                            c = alpha(kClLevels, st, s0, s1);
                            keep_pq(kClLevels, st, s0);
                        }
                        __syncthreads();  // every warp has read what changes now
                    } else {  // two warps per value; one thread each for the coefficients
                        if (warp < 4) {
                            const T *u1 = warp < 2 ? qj : r;
                            T x = 0;
#pragma unroll 4
                            for (int k = lane + 32 * (warp & 1); k < len; k += 64) x += p[k] * u1[k];
#pragma unroll
                            for (int o = 16; o > 0; o >>= 1) x += __shfl_xor_sync(0xffffffffu, x, o);
                            if (lane == 0) coef_s[1 + warp] = x;
                        }
                        __syncthreads();
                        if (tid == 0)
                            coef_s[0] = j < st ? beta(kClLevels, j, coef_s[1] + coef_s[2])
                                               : alpha(kClLevels, st, coef_s[1] + coef_s[2], coef_s[3] + coef_s[4]);
                        else if (tid == 32 && j == st)
                            keep_pq(kClLevels, st, coef_s[1] + coef_s[2]);
                        __syncthreads();
                        c = coef_s[0];
                    }
#pragma unroll 1
                    for (int k = tid; k < len; k += kClThreads) {
                        if (j < st) {
                            p[k] += c * pj[k];
                            w[k] += c * qj[k];
                        } else {
                            E[k] = st > 0 ? E[k] + c * p[k] : c * p[k];
                            if (!last) Rv[k] = r[k] - c * w[k];
                        }
                    }
                    __syncthreads();
                }
            }
            mark(y.nsp, OP_COARSE);
        }
        if (y.nsp == 0) break;
        // ---- back up: B^ of level lv after the correction, Alg. 1 step i ------------------
        bool done = false;
        for (;;) {
            const int i = (int)(steps >> (4 * lv)) & 15;
            const int foff = i == 0 ? CL_F(rhs) : CL_F(r), zoff = p_off(i), qoff = q_off(i);
            const int post = CL_F(post), npost = CL_F(npost), nact = CL_F(nact), eoff = CL_F(e);
            const int rows = (int)(h0.x << lt2.x), nwin = (int)h0.y;
            const bool last = i == y.kc - 1;
            const uint32_t z = dyn + zoff;
            {  // z += P e on the window; the colour swept next is overwritten unread
                const uint4 op = cl_ld<uint4>(dyn + post);
                load_item(op.x, tid, op.y, true, lt2.w == 2 ? CL_F(blk) : 0, zoff, kn + (lt2.w == 2));
                const uint32_t en = dyn + (lv + 1 < y.nsp ? cl_ld<int>(lvb + (uint32_t)(sizeof(ClLev) + offsetof(ClLev, e)))
                                                          : y.E);
                const uint32_t par = dyn + CL_F(parent);
                const uint2 ls = cl_ld<uint2>(dyn + lt1.w + 32);
                const int nen = lv + 1 < y.nsp ? ((const ClHead *)at(lvs[lv + 1].head))->nwin : y.nd;  // (index checks)
                perhaps_late();
#pragma unroll 1
                for (unsigned k = tid; k < (unsigned)nwin; k += kClThreads)
                    if (k < ls.x || k >= ls.y) {
                        const uint32_t zk = z + (uint32_t)sizeof(T) * k;
                        const unsigned pk = cl_ld<unsigned short>(par + 2 * k);
                        if (idx_ok((int)pk, nen)) cl_st(zk, cl_ld<T>(zk) + cl_ld<T>(en + (uint32_t)sizeof(T) * pk));
                    }
                __syncthreads();
                if (lt2.w == 2) {  // (blocks: the colour swept next is read too, so the neighbours
                    arrive_n(0);   // must have added it everywhere before its rows come in)
                    wait_n();
                }
                mark(lv, OP_PROLONG);
            }
            sweep(post, npost, true, foff, zoff, rows, zoff);
            if (lt2.w == 2) {  // B^_0 is all: z is the result
                done = true;
                break;
            }
#pragma unroll 1
            for (int j = 0; j < i; j++) {  // p_i = z + sum_j beta_j p_j, on the window
                T zq = 0;
                const uint32_t qj = dyn + q_off(j), pj = dyn + p_off(j);
#pragma unroll 1
                for (int m = tid; m < (int)h0.x; m += kClThreads) {
                    const uint32_t l2 = cl_ld<unsigned short>(dyn + lt0.x + 2 * m);
                    zq += cl_ld<T>(z + l2) * cl_ld<T>(qj + l2);
                }
                const T c = cluster_sum(zq, T(0), nact, nothing, [&](T x, T) { return beta(lv, j, x); }, no_pq);
                mark(lv, OP_MULTIDOT);
                perhaps_late();
#pragma unroll 1
                for (int k = tid; k < nwin; k += kClThreads) {
                    const uint32_t o = (uint32_t)sizeof(T) * k;
                    cl_st(z + o, cl_ld<T>(z + o) + c * cl_ld<T>(pj + o));
                }
                __syncthreads();
                mark(lv, OP_ORTH);
            }
            // q = A p; (p, q), (r, p); the next step's z = 0
            T pq = 0, rp = 0;
#pragma unroll 1
            for (int c = 0;;) {
                if (c + 32 * warp < rows) {
                    const T fi = cl_ld<T>(dyn + foff + (uint32_t)sizeof(T) * mi), zi = cl_ld<T>(z + lb);
                    const T qi = row_dot() + dg * zi;
                    cl_st_if(own, dyn + qoff + lb, qi);
                    const T zo = own ? zi : T(0);
                    pq += zo * qi;
                    rp += fi * zo;
                }
                c += kClThreads;
                if (c >= rows) break;
                load_row(0, c + tid, rows, zoff, zoff, kn);
            }
            const int poff = last ? eoff : p_off(i + 1), roff = CL_F(r);
            if (!last) zero_window(dyn + poff);
            auto load_own = [&](int m) {  // offset, 1 / a_ii and destinations of own row m
                if (m >= (int)h0.x) return;
                lb = cl_ld<unsigned short>(dyn + lt0.x + 2 * m);
                dinv = cl_ld<T>(dyn + lt1.x + (uint32_t)sizeof(T) * m);
                load_dst(true, m, poff, kn);
            };
            const T al = cluster_sum(pq, rp, nact, [&] { load_own(tid); },
                                     [&](T x, T y2) { return alpha(lv, i, x, y2); },
                                     [&](T x) { keep_pq(lv, i, x); });
            mark(lv, OP_SPMV_DOT);
            perhaps_late();
            // e (+)= alpha p, r = r - alpha q; the next step's first colour
#pragma unroll 1
            for (int m = tid; m < (int)h0.x;) {
                const T zi = cl_ld<T>(z + lb);
                T u = i > 0 ? cl_ld<T>(dyn + eoff + lb) + al * zi : al * zi;
                cl_st(dyn + eoff + lb, u);
                bool to = last && lv > 0;
                if (!last) {
                    const uint32_t mo = (uint32_t)sizeof(T) * m;
                    const T rn = cl_ld<T>(dyn + foff + mo) - al * cl_ld<T>(dyn + qoff + lb);
                    cl_st(dyn + roff + mo, rn);
                    to = (unsigned)(m - (int)h1.x) < h1.y;
                    if (to) {
                        u = rn * dinv;
                        cl_st(dyn + poff + lb, u);
                    }
                }
                if (to) push(poff, u);
                m += kClThreads;
                load_own(m);
            }
            if (!last) {
                first_exchange(poff, q_off(i + 1));
                mark(lv, OP_UPDATE);
                steps += 1ull << (4 * lv);
                break;  // B^ for the next step
            }
            if (lv == 0) {
                mark(lv, OP_UPDATE);
                done = true;
                break;
            }
            arrive_n((int)h0.z);  // e, to the windows the prolongation reads
            bind(lv - 1);
            wait_n();
            mark(lv, OP_UPDATE);
            lv--;
        }
        if (done) break;
    }
    __syncthreads();
    if (alive) {
        if (y.nsp > 0) {
            const int nown = (int)h0.x;  // (level 0 is bound)
            const unsigned short *own = (const unsigned short *)at(lvs[0].own);
            const T *e = vec(lt2.w == 2 ? p_off(0) : CL_F(e));
#pragma unroll 1
            for (int m = tid; m < nown; m += kClThreads) a.e[((const int *)at(y.top))[m]] = *(const T *)((const unsigned char *)e + own[m]);
        } else {
            const T *E = vec(y.E);
#pragma unroll 1
            for (int k = rank * y.ch + tid; k < min(y.nd, (rank + 1) * y.ch); k += kClThreads) a.e[k] = E[k];
        }
    }
    cl_sync_all();  // no CTA leaves while a neighbour may still write into it
    if (*gave_up) cl_drain(mb0 + 32);
    if (a.ts && rank == 0 && tid == 0) *a.ts = global_ns();
}

// ---------------------------------------------------------------------------------------
// setup of the cluster's image (device)

// a level as setup left it; cr: its colour ranges
struct ClSrc {
    int n, ncol, uw;
    const int *sl, *col;
    const int *parent;           // pi-row of the next level
    const int4 *ch, *ch2;        // children of the next level's rows
    const double *val64;
    const float *val32;
    const int *bptr;             // finest level: row ranges of its blocks (the next level's rows)
    int cr[kClColors + 1];
};
struct ClSrcs {
    int nsp;                     // lv[nsp]: the dense level (n, ncol, cr)
    ClSrc lv[kClLevels + 1];
};

__device__ __forceinline__ int cl_colour(const ClSrc &S, int i) {
    int c = 0;
    while (c + 1 < S.ncol && i >= S.cr[c + 1]) c++;
    return c;
}
// the CTA that owns row i of colour c: the last part that starts at or before it
__host__ __device__ inline int cl_part(int len, int r) { return (int)((long long)len * r / kClRanks); }
__device__ __forceinline__ int cl_owner(const ClSrc &S, int c, int i) {
    const int len = S.cr[c + 1] - S.cr[c];
    return (kClRanks * (i - S.cr[c] + 1) - 1) / len;
}
// the CTA that owns row i (colour c) of level a: the finest level's rows go with their block
__device__ __forceinline__ int cl_row_owner(const ClSrcs &G, int a, int c, int i) {
    const ClSrc &S = G.lv[a];
    return S.bptr ? cl_owner(G.lv[a + 1], c, S.parent[i]) : cl_owner(S, c, i);
}
// Window tables: [level][rank][colour] (first, last + 1). The children of the next level's rows
// that lie in another strip than the row's owner have tables of their own: cwin[0] with the
// next level's strips as owners (a swept level), cwin[1] with the owner of a row's first child
// (the dense level, whose rows have no strips: fo[R]).
__device__ __forceinline__ void cl_extend(int2 *w, int i) {
    volatile int *v = (volatile int *)w;
    if (i < v[0]) atomicMin(&w->x, i);
    if (i + 1 > v[1]) atomicMax(&w->y, i + 1);
}
__host__ __device__ inline size_t cl_win(int a, int r, int c) {
    return ((size_t)a * kClRanks + r) * kClColors + c;
}
__device__ __forceinline__ int cl_child(const ClSrc &S, int R, int q) {
    const int4 ch = (q < 4 ? S.ch : S.ch2)[R];
    return (q & 3) == 0 ? ch.x : (q & 3) == 1 ? ch.y : (q & 3) == 2 ? ch.z : ch.w;
}

// columns of own rows, both ways, and children of own next-level rows in other strips. Rows
// of a strip's inside touch nothing; the few at its edges hit a table entry that mostly holds
// them already (read before the atomic).
__global__ void k_cl_windows(const __grid_constant__ ClSrcs G, int2 *win, int2 *cwin, size_t words,
                             int *fo) {
    const int a = blockIdx.y;
    const ClSrc &S = G.lv[a], &N = G.lv[a + 1];
    const int i = blockIdx.x * blockDim.x + threadIdx.x;
    if (i < S.n) {
        const int c = cl_colour(S, i), r = cl_row_owner(G, a, c, i);
        const int s0 = S.sl[i >> 5], width = (S.sl[(i >> 5) + 1] - s0) >> 5;
        for (int k = 1; k < width; k++) {
            const int j = S.col[s0 + 32 * k + (i & 31)];
            if (j < 0) continue;
            const int cj = cl_colour(S, j), rj = cl_row_owner(G, a, cj, j);
            if (rj == r) continue;
            cl_extend(win + cl_win(a, r, cj), j);
            cl_extend(win + cl_win(a, rj, c), i);
        }
    }
    if (i < N.n) {
        const int ra = cl_owner(N, cl_colour(N, i), i);
        int rb = S.bptr ? ra : -1;  // (a block's rows go with it)
        for (int q = 0; q < (S.bptr ? 0 : S.ch2 ? 8 : 4); q++) {
            const int j = cl_child(S, i, q);
            if (j < 0) continue;
            const int cj = cl_colour(S, j), rj = cl_owner(S, cj, j);
            if (rb < 0) rb = rj;
            if (rj != ra) cl_extend(cwin + cl_win(a, ra, cj), j);
            if (rj != rb) cl_extend(cwin + words + cl_win(a, rb, cj), j);
        }
        if (a == G.nsp - 1) fo[i] = max(rb, 0);
        if (a == G.nsp - 2) fo[G.lv[G.nsp].n + i] = max(rb, 0);
    }
}

// one CTA, level by level: the children's part joins the window (the last level's next one
// is dense, the one before may have either kind); then the parents of the window's rows join
// the next level's window
__global__ void __launch_bounds__(1024) k_cl_parents(const __grid_constant__ ClSrcs G, int2 *win,
                                                     const int2 *cwin, size_t words) {
    const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
    for (int a = 0; a < G.nsp; a++) {
        const ClSrc &S = G.lv[a];
        for (int k = threadIdx.x; k < kClRanks * S.ncol; k += blockDim.x) {
            const size_t o = cl_win(a, k / S.ncol, k % S.ncol);
            for (int kind = 0; kind < 2; kind++) {
                if (kind == 0 ? a == G.nsp - 1 : a < G.nsp - 2) continue;
                const int2 w = cwin[kind * words + o];
                if (w.x < w.y) {
                    win[o].x = min(win[o].x, w.x);
                    win[o].y = max(win[o].y, w.y);
                }
            }
        }
        __syncthreads();
        if (a + 1 < G.nsp) {
            const ClSrc &N = G.lv[a + 1];
            for (int k = warp; k < kClRanks * S.ncol; k += (int)(blockDim.x >> 5)) {
                const int r = k / S.ncol;
                const int2 w = win[cl_win(a, r, k % S.ncol)];
                for (int i = w.x + lane; i < w.y; i += 32) {
                    const int p = S.parent[i];
                    cl_extend(win + cl_win(a + 1, r, cl_colour(N, p)), p);
                }
            }
            __syncthreads();
        }
    }
}

// the constant image of strip blockIdx.y, level blockIdx.z (nsp: the coarsest inverse); the
// tables at its start (op lists, heads) are there already. geo: [level][rank][colour]; over_n:
// entries used in each strip's list of further destinations
template <class T>
__global__ void k_cl_image(const __grid_constant__ ClSrcs G, const __grid_constant__ ClLayout y,
                           unsigned char *image, const ClColor *geo, int *over_n,
                           const double *Ainv, const float *Ainv2) {
    const int a = blockIdx.z, r = blockIdx.y;
    unsigned char *im = image + (size_t)r * y.image_stride;
    const int t0 = blockIdx.x * blockDim.x + threadIdx.x, nt = gridDim.x * blockDim.x;
    if (a == y.nsp) {
        if (y.dense) {  // A's rows (columns are pi-rows)
            const ClSrc &S = G.lv[a];
            for (int k = t0; k < y.ch * y.aw; k += nt) {
                const int row = k % y.ch, slot = k / y.ch, i = r * y.ch + row;
                if (i >= y.nd) continue;
                const int s0 = S.sl[i >> 5], width = (S.sl[(i >> 5) + 1] - s0) >> 5;
                const int o = s0 + 32 * slot + (i & 31), j = slot < width ? S.col[o] : -1;
                ((unsigned short *)(im + y.acol))[k] = (unsigned short)(j >= 0 ? j : i);
                T v = T(0);
                if (j >= 0) {
                    if constexpr (sizeof(T) == 8) v = S.val64[o];
                    else v = S.val32[o];
                }
                ((T *)(im + y.aval))[k] = v;
            }
            return;
        }
        for (int k = t0; k < y.ch * y.nd; k += nt) {
            const int row = k / y.nd, j = k - row * y.nd, i = r * y.ch + row;
            if (i >= y.nd) continue;
            const size_t s = (size_t)i * y.nd + j, d = (size_t)row * y.stride + j;
            if constexpr (sizeof(T) == 8) {
                ((double *)(im + y.mat))[d] = Ainv[s];
            } else {
                ((float *)(im + y.mat))[d] = Ainv2[s];
                ((float *)(im + y.mat_lo))[d] = Ainv2[(size_t)y.nd * y.nd + s];
            }
        }
        return;
    }
    const ClLev &L = y.lv[a];
    const ClSrc &S = G.lv[a];
    const ClHead H = *(const ClHead *)(im + L.head);
    const ClColor *tab = geo + cl_win(a, r, 0);
    T *val = (T *)(im + L.val), *diag = (T *)(im + L.diag), *dinv = (T *)(im + L.dinv);
    unsigned short *col = (unsigned short *)(im + L.col), *own = (unsigned short *)(im + L.own);
    unsigned short *par = (unsigned short *)(im + L.parent), *child = (unsigned short *)(im + L.child);
    uint4 *dst = (uint4 *)(im + L.dst);  // (d0, 0, d1 or bit 31 and a list, 0)
    unsigned *over = (unsigned *)(im + L.over);
    auto local = [&](const ClColor *tb, const ClSrc &s, int i) {  // window index of pi-row i
        const ClColor &C = tb[cl_colour(s, i)];
        return (unsigned short)(C.li0 + i - C.g0);
    };
    constexpr int B = (int)sizeof(T);  // own rows, columns and destinations are byte offsets
    const int G1 = 1 << L.lg;
    constexpr int V = 16 / (int)sizeof(T);  // values per 16-byte piece
    for (int m = t0; m < H.nown; m += nt) {
        int c = 0;
        while (c + 1 < L.ncol && m >= tab[c + 1].m0) c++;
        const int i = tab[c].g0 + m - tab[c].m0;
        const int li = tab[c].li0 + m - tab[c].m0;
        own[m] = (unsigned short)(B * li);
        const int s0 = S.sl[i >> 5], width = (S.sl[(i >> 5) + 1] - s0) >> 5;
        // lane q of the row takes slots 1 + ns q ..; padding: value 0, the row's own column
        for (int k = 1; k < 1 + L.ns * G1; k++) {
            const int o = s0 + 32 * k + (i & 31);
            const int j = k < width ? S.col[o] : -1;
            T v = T(0);
            if (j >= 0) {
                if constexpr (sizeof(T) == 8) v = S.val64[o];
                else v = S.val32[o];
            }
            const int vr = m * G1 + (k - 1) / L.ns, e = (k - 1) % L.ns;
            col[(size_t)vr * kClSlots + e] = (unsigned short)(B * (j >= 0 ? local(tab, S, j) : li));
            val[((size_t)(e / V) * L.R + vr) * V + e % V] = v;
        }
        const double d = S.val64[s0 + (i & 31)];
        if constexpr (sizeof(T) == 8) diag[m] = d;
        else diag[m] = S.val32[s0 + (i & 31)];
        dinv[m] = (T)(1.0 / d);
        // the strips whose window holds the row
        unsigned to[kClRanks];
        int nd = 0;
        for (int q = 0; q < kClRanks; q++) {
            const ClColor &C = geo[cl_win(a, q, c)];
            const int k = C.li0 + i - C.g0 - C.seg0;  // position in its window
            if (q != r && k >= 0 && k < C.seglen) to[nd++] = (unsigned)q << 16 | (unsigned)(B * (C.seg0 + k));
        }
        uint4 d2 = make_uint4(nd > 0 ? to[0] : kClNone, 0, nd > 1 ? to[1] : kClNone, 0);
        if (nd > 2) {
            const int o = atomicAdd(&over_n[a * kClRanks + r], nd);
            for (int k = 1; k < nd; k++) over[o + k - 1] = to[k];
            over[o + nd - 1] = kClNone;
            d2.z = 0x80000000u | (unsigned)o;
        }
        dst[m] = d2;
        if (a == 0) ((int *)(im + y.top))[m] = i;
    }
    const bool swept = a + 1 < y.nsp;
    const ClColor *ntab = swept ? geo + cl_win(a + 1, r, 0) : nullptr;
    for (int k = t0; k < H.nwin; k += nt) {
        int c = 0;
        while (c + 1 < L.ncol && k >= tab[c + 1].seg0) c++;
        const int p = S.parent[tab[c].g0 + k - tab[c].li0];
        par[k] = swept ? local(ntab, G.lv[a + 1], p) : (unsigned short)p;
    }
    const int nn = swept ? ((const ClHead *)(im + y.lv[a + 1].head))->nown : *(const int *)(im + y.dhead);
    for (int m = t0; m < nn; m += nt) {
        int R;
        if (swept) {
            int c = 0;
            while (c + 1 < y.lv[a + 1].ncol && m >= ntab[c + 1].m0) c++;
            R = ntab[c].g0 + m - ntab[c].m0;
        } else {
            R = ((const unsigned short *)(im + y.down))[m];
        }
        if (S.bptr) {
            const int i = S.bptr[R], c = cl_colour(S, i);
            ((unsigned short *)(im + L.blk))[m] = (unsigned short)(tab[c].m0 + i - tab[c].g0);
            if (m == nn - 1) ((unsigned short *)(im + L.blk))[nn] = (unsigned short)H.nown;
            continue;
        }
        for (int q = 0; q < L.nch; q++) {
            const int j = cl_child(S, R, q);
            // four per 8-byte entry
            child[((size_t)(q >> 2) * L.Rn + m) * 4 + (q & 3)] = j >= 0 ? local(tab, S, j) : (unsigned short)0xFFFF;
        }
    }
}

// column blockIdx.x of M = B^_D (Alg. 2 on level D, one above the coarsest, whose solve is
// exact: a linear map) and of A M, in FP64: the steps of the cycle on one unit vector
template <class T>
__global__ void __launch_bounds__(128)
k_dense_cycle(const __grid_constant__ ClSrc S, const __grid_constant__ ClLayout y,
              unsigned char *image, const double *Ainv, int nc) {
    extern __shared__ double sd[];
    const int n = S.n, tid = threadIdx.x, nt = blockDim.x, unit = blockIdx.x;
    double *z = sd, *t = z + n, *dinv = t + n, *fc = dinv + n, *ec = fc + nc;
    auto dot = [&](int i, int k0) {
        const int s0 = S.sl[i >> 5], width = (S.sl[(i >> 5) + 1] - s0) >> 5;
        double acc = 0.0;
        for (int k = k0; k < width; k++) {
            const int o = s0 + 32 * k + (i & 31), j = S.col[o];
            if (j >= 0) acc += S.val64[o] * z[j];
        }
        return acc;
    };
    for (int i = tid; i < n; i += nt) {
        z[i] = 0.0;
        dinv[i] = 1.0 / S.val64[S.sl[i >> 5] + (i & 31)];
    }
    __syncthreads();
    auto sweep = [&](int c) {
        for (int i = S.cr[c] + tid; i < S.cr[c + 1]; i += nt)
            z[i] = ((i == unit ? 1.0 : 0.0) - dot(i, 1)) * dinv[i];
        __syncthreads();
    };
    for (int sw = 0; sw < y.nu_pre; sw++)
        for (int c = 0; c < S.ncol; c++) sweep(c);
    for (int i = tid; i < n; i += nt) t[i] = (i == unit ? 1.0 : 0.0) - dot(i, 0);
    __syncthreads();
    for (int R = tid; R < nc; R += nt) {
        double v = 0.0;
        for (int q = 0; q < (S.ch2 ? 8 : 4); q++) {
            const int j = cl_child(S, R, q);
            if (j >= 0) v += t[j];
        }
        fc[R] = v;
    }
    __syncthreads();
    for (int R = tid; R < nc; R += nt) {
        double v = 0.0;
        for (int j = 0; j < nc; j++) v += Ainv[(size_t)j * nc + R] * fc[j];  // symmetric
        ec[R] = v;
    }
    __syncthreads();
    for (int i = tid; i < n; i += nt) z[i] += ec[S.parent[i]];
    __syncthreads();
    for (int sw = 0; sw < y.nu_post; sw++)
        for (int c = S.ncol - 1; c >= 0; c--) sweep(c);
    for (int i = tid; i < n; i += nt) {
        unsigned char *im = image + (size_t)(i / y.ch) * y.image_stride;
        const size_t o = (size_t)(i % y.ch) * y.stride + unit;
        const T hi = (T)z[i];
        ((T *)(im + y.mat))[o] = hi;
        if constexpr (sizeof(T) == 4) {
            ((T *)(im + y.mat_lo))[o] = (T)(z[i] - (double)hi);
            if (y.aw == 0) ((T *)(im + y.mat))[(size_t)y.ch * y.stride + o] = (T)dot(i, 0);
        }
    }
}

#undef CL_F

}  // namespace amg
