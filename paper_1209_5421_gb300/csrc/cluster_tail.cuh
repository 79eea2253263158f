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
// of its window on the level above. Every vector of a level is stored in window order, one
// index for all of them.
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
// Sums over the cluster and gathers to all CTAs count on two mbarriers of their own.
//
// The level above the coarsest: B^ there is linear (the coarsest solve is exact), so setup
// forms M = B^ and A M as dense matrices once (k_dense_cycle, FP64), each CTA keeps 1/16 of
// their rows, and one product with a residual gives p and A p of an Alg. 1 step; that replaces
// about 13 dependent steps. Where the matrices do not fit, the level is swept like the others
// and the coarsest solve is the dense product.
#pragma once

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
constexpr int kClBatch = 9;        // slots read together (one batch for a 9-point row)

// one colour of one CTA's strip
struct ClColor {
    int li0, cnt;      // own rows: window index of the first, number
    int m0;            // its index among the own rows of all colours (matrix rows)
    int seg0, seglen;  // the colour's window
    int push0, npush;  // its rows' destinations
    int expect;        // bytes its window receives from the neighbours in an exchange
    int g0;            // pi-row of the first own row
    int pad[3];
};
// rows [j0, j0 + cnt) of the colour's own rows go to CTA dst, window index dli there
struct ClPush {
    int dst_color;     // dst + 256 colour
    int j0, cnt, dli;
};
struct ClHead {        // of one level's strip
    int nown, nwin, npush, expect_all;
};

// a swept level: sizes, and byte offsets into the shared memory (the same in every CTA)
struct ClLev {
    int level, n, ncol, w;
    int R;             // matrix rows (own rows of the largest strip, 8 mod 32)
    int c_first, c_last;
    unsigned cmask;    // non-empty colours
    int nch;           // children per row of the next level's rows: 4 or 8
    int Rn;            // stride of the children's table (own rows of the next level)
    int xchild;        // 1: a child of an own next-level row may lie in another strip
    int head, tab, push, val, col, dinv, own, parent, child;  // constant image
    int rhs, e, r, p[kMaxKcycle], q[kMaxKcycle];              // vectors
};

struct ClLayout {
    int nsp;           // swept levels: tl .. tl + nsp - 1; the dense level follows
    int tl;
    int dense;         // 1: M and A M of the level above the coarsest, 0: coarsest inverse
    int kc, nu_pre, nu_post;
    int nd, ch, stride;  // dense level: rows, rows per CTA (multiple of 4), row stride
    int mat, mat_lo;     // M then A M (or the inverse; FP32: high parts, low parts)
    int dhead, down;     // gather into the dense level: own rows (count; their pi-rows)
    int peers;           // neighbour CTAs: count, ranks
    int F, Rv, E, out, P[kMaxKcycle], Q[kMaxKcycle];  // dense level's vectors (every CTA: all)
    int stage;           // one value per own row of the dense level
    int image_bytes, bytes;
    ClLev lv[kClLevels];
};

template <class T>
struct ClArgs {
    ClLayout y;
    const unsigned char *image;  // [kClRanks][image_bytes]
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
__device__ __forceinline__ void cl_mb_arrive(uint32_t mb) {
    asm volatile("mbarrier.arrive.shared::cta.b64 _, [%0];" ::"r"(mb) : "memory");
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

// sum over slots k0 <= k < w of row m (matrix rows stored slot by slot, stride R); padding
// has value 0 and the row's own column
template <class T>
__device__ __forceinline__ T cl_row_dot(const T *val, const unsigned short *col, int m, int R,
                                        int k0, int w, const T *x, int nwin) {
    T acc = 0;
    for (int kb = k0; kb < w; kb += kClBatch) {
        unsigned short c[kClBatch];
        T v[kClBatch], xv[kClBatch];
#pragma unroll
        for (int j = 0; j < kClBatch; j++) {
            const bool in = kb + j < w;
            c[j] = in ? col[(kb + j) * R + m] : (unsigned short)0;
            v[j] = in ? val[(kb + j) * R + m] : T(0);
        }
#pragma unroll
        for (int j = 0; j < kClBatch; j++)
            xv[j] = (kb + j < w && idx_ok((int)c[j], nwin)) ? x[c[j]] : T(0);
#pragma unroll
        for (int j = 0; j < kClBatch; j++) acc += v[j] * xv[j];
    }
    return acc;
}

// ---------------------------------------------------------------------------------------
extern __shared__ __align__(16) unsigned char cl_dyn[];

template <class T>
__global__ void __launch_bounds__(kClThreads, 1)
k_cluster_tail(const __grid_constant__ ClArgs<T> a) {
    constexpr bool F64 = sizeof(T) == 8;
    constexpr int NR = kClRanks;
    __shared__ __align__(8) unsigned long long mbs[5];  // neighbours x 2, all CTAs x 2, image
    __shared__ __align__(16) T red[2][NR][4];           // sums over the cluster: partials
    __shared__ T sred[F64 ? 3 * kClThreads : 4 * kClWarps];
    __shared__ T coef[4], lsum[4];
    __shared__ T pqs[kClLevels + 1][kMaxKcycle];        // (p_i, A p_i) of every level
    __shared__ int stops[kClLevels + 1][kMaxKcycle];    // Alg. 1 stopped at or before step i
    __shared__ int gave_up_s, token, img_ok;
    volatile int *gave_up = &gave_up_s;
    const ClLayout &y = a.y;
    const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
    int rank;
    asm("mov.u32 %0, %%cluster_ctarank;" : "=r"(rank));
    const uint32_t mb0 = cl_smem(mbs);
    if (tid == 0) {
        cl_mb_init(mb0, kClWarps);
        cl_mb_init(mb0 + 8, kClWarps);
        cl_mb_init(mb0 + 16, 1);
        cl_mb_init(mb0 + 24, 1);
        cl_mb_init(mb0 + 32, 1);
        asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
        gave_up_s = 0;
        img_ok = 1;
        token = 0;
    }
    __syncthreads();
    if (tid == 0) {  // this CTA's constant image, one bulk copy
        cl_mb_expect(mb0 + 32, y.image_bytes);
        asm volatile(
            "cp.async.bulk.shared::cluster.global.mbarrier::complete_tx::bytes [%0], [%1], %2, [%3];" ::"r"(
                cl_smem(cl_dyn)),
            "l"(a.image + (size_t)rank * y.image_bytes), "r"(y.image_bytes), "r"(mb0 + 32)
            : "memory");
    }
    cl_sync_all();  // every CTA's mbarriers are ready
    if (tid == 0 && !cl_mb_try(mb0 + 32, 0) &&
        !cl_wait_slow(mb0 + 32, 0, gave_up, a.err, kBarrierLimitNs))
        img_ok = 0;
    __syncthreads();
    if (img_ok) (void)cl_mb_try(mb0 + 32, 0);  // complete: every thread acquires the copy
    // an error of an earlier launch of this application, or no image: nothing to run (the
    // copy in flight is waited for above; the CTAs leave together)
    bool alive = img_ok && !(ld_volatile_int(a.err) & kErrTimeout);
    if (!img_ok) {
        cl_sync_all();
        return;
    }
    unsigned kn = 0, ka = 0;  // exchanges so far: neighbours, all CTAs
    int extra = a.extra;
    auto at = [&](int off) { return cl_dyn + off; };
    const int npeer = ((const int *)at(y.peers))[0];
    long long tp0 = 0;
    const bool mark_on = a.tprof && rank == 0 && tid == 0;
    // profiling: cycles and count per (level, kind), summed here and added up at the end
    __shared__ unsigned prof_s[2][16 * (kClLevels + 2)];
    if (mark_on)
        for (int k = 0; k < 2 * 16 * (kClLevels + 2); k++) (&prof_s[0][0])[k] = 0;
    auto mark = [&](int level, int kind) {
        if (!mark_on) return;
        const long long t1 = clock64();
        const int slot = 16 * (level - y.tl) + kind;
        prof_s[0][slot] += (unsigned)(t1 - tp0);
        prof_s[1][slot] += 1;
        tp0 = t1;
    };
    if (mark_on) tp0 = clock64();

    // this CTA's arrivals of neighbour exchange kn (which receives `bytes` of rows) and the
    // wait for everybody's
    auto exchange = [&](int bytes) {
        const uint32_t mb = mb0 + 8 * (kn & 1);
        __syncwarp();
        if (alive) {
            if (lane == 0) {
                if (warp == 0) {
                    cl_mb_expect(mb, bytes + 4 * npeer + extra);
                    extra = 0;
                } else {
                    cl_mb_arrive(mb);
                }
            }
            if (warp == kClWarps - 1)
                for (int p = lane; p < npeer; p += 32) {
                    const int dst = ((const int *)at(y.peers))[1 + p];
                    cl_store(cl_map(cl_smem(&token), dst), 0.f, cl_map(mb, dst));
                }
            if (!cl_mb_try(mb, (kn >> 1) & 1))
                alive = cl_wait_slow(mb, (kn >> 1) & 1, gave_up, a.err, a.limit_ns);
        }
        kn++;
    };
    // the wait of an exchange between all CTAs; thread 0 announces the bytes it receives
    auto mb_all = [&]() { return mb0 + 16 + 8 * (ka & 1); };
    auto wait_all = [&](int bytes) {
        const uint32_t mb = mb_all();
        if (alive) {
            if (tid == 0) {
                cl_mb_expect(mb, bytes + extra);
                extra = 0;
            }
            if (!cl_mb_try(mb, (ka >> 1) & 1))
                alive = cl_wait_slow(mb, (ka >> 1) & 1, gave_up, a.err, a.limit_ns);
        }
        ka++;
    };
    // row j of a colour's own rows to the neighbours that hold it
    auto push_row = [&](const ClLev &L, const ClColor &C, int j, uint32_t vec, T v) {
        const ClPush *P = (const ClPush *)at(L.push) + C.push0;
        const uint32_t mb = mb0 + 8 * (kn & 1);
        for (int e = 0; e < C.npush; e++) {
            const ClPush q = P[e];
            if ((unsigned)(j - q.j0) < (unsigned)q.cnt && alive) {
                const int dst = q.dst_color & 255;
                cl_store(cl_map(vec + (uint32_t)sizeof(T) * (q.dli + j - q.j0), dst), v,
                         cl_map(mb, dst));
            }
        }
    };
    // every own row of vector `off` (complete in this CTA) to the neighbours
    auto push_all = [&](const ClLev &L, int off) {
        const ClHead &H = *(const ClHead *)at(L.head);
        const ClPush *P = (const ClPush *)at(L.push);
        const T *v = (const T *)at(off);
        const uint32_t vec = cl_smem(v), mb = mb0 + 8 * (kn & 1);
        if (alive)
            for (int e = warp; e < H.npush; e += kClWarps) {
                const ClPush q = P[e];
                const int dst = q.dst_color & 255;
                const ClColor &C = ((const ClColor *)at(L.tab))[q.dst_color >> 8];
                const T *src = v + C.li0 + q.j0;
                const uint32_t to = cl_map(vec + (uint32_t)sizeof(T) * q.dli, dst),
                               mbd = cl_map(mb, dst);
                for (int j = lane; j < q.cnt; j += 32)
                    cl_store(to + (uint32_t)sizeof(T) * j, src[j], mbd);
            }
    };
    // Sums of v[0..nv) over the own rows' threads (warps [0, nact)) of this CTA (ALL = false)
    // or of the cluster; coefs(s, c) turns the sums into coefficients, the same in every CTA.
    // FP32: sums and coefficients in every thread; FP64 (scarce): one warp per sum, the
    // coefficients by one thread.
    auto reduce = [&](auto all_tag, T (&v)[3], int nv, int nact, auto coefs, T (&c)[2]) {
        constexpr bool ALL = decltype(all_tag)::value;
        nact = min(nact, kClWarps);
        T s[3] = {T(0), T(0), T(0)};
        if constexpr (!F64) {
            if (warp < nact) {
#pragma unroll
                for (int k = 0; k < 3; k++)
                    if (k < nv) {
                        T x = v[k];
#pragma unroll
                        for (int o = 16; o > 0; o >>= 1) x += __shfl_down_sync(0xffffffffu, x, o);
                        if (lane == 0) sred[4 * warp + k] = x;
                    }
            }
            __syncthreads();
            if constexpr (ALL) {
                if (warp == 0 && lane < NR && alive) {
                    float p[4] = {0.f, 0.f, 0.f, 0.f};
                    for (int w2 = 0; w2 < nact; w2++)
#pragma unroll
                        for (int k = 0; k < 3; k++)
                            if (k < nv) p[k] += sred[4 * w2 + k];
                    const uint32_t mb = mb_all();
                    asm volatile(
                        "st.async.shared::cluster.mbarrier::complete_tx::bytes.v4.f32 [%0], {%1, %2, %3, %4}, [%5];" ::"r"(
                            cl_map(cl_smem(&red[ka & 1][rank][0]), lane)),
                        "f"(p[0]), "f"(p[1]), "f"(p[2]), "f"(p[3]), "r"(cl_map(mb, lane))
                        : "memory");
                }
                const T(*part)[4] = red[ka & 1];
                wait_all(NR * 16);
#pragma unroll
                for (int k = 0; k < 3; k++)
                    if (k < nv) {
                        T x = part[lane & (NR - 1)][k];
#pragma unroll
                        for (int o = NR / 2; o > 0; o >>= 1) x += __shfl_xor_sync(0xffffffffu, x, o);
                        s[k] = x;
                    }
            } else {
                for (int w2 = 0; w2 < nact; w2++)
#pragma unroll
                    for (int k = 0; k < 3; k++)
                        if (k < nv) s[k] += sred[4 * w2 + k];
                __syncthreads();  // sred is reused by the next reduction
            }
            coefs(s, c);
        } else {
            if (warp < nact)
#pragma unroll
                for (int k = 0; k < 3; k++)
                    if (k < nv) sred[k * kClThreads + tid] = v[k];
            __syncthreads();
            if (warp < nv) {
                T x = 0;
                for (int j = lane; j < 32 * nact; j += 32) x += sred[warp * kClThreads + j];
#pragma unroll
                for (int o = 16; o > 0; o >>= 1) x += __shfl_xor_sync(0xffffffffu, x, o);
                if constexpr (ALL) {
                    if (lane < NR && alive)
                        cl_store(cl_map(cl_smem(&red[ka & 1][rank][warp]), lane), x,
                                 cl_map(mb_all(), lane));
                } else if (lane == 0) {
                    lsum[warp] = x;
                }
            }
            if constexpr (ALL) {
                const T(*part)[4] = red[ka & 1];
                wait_all(NR * 8 * nv);
                if (warp == 0) {
#pragma unroll
                    for (int k = 0; k < 3; k++)
                        if (k < nv) {
                            T x = part[lane & (NR - 1)][k];
#pragma unroll
                            for (int o = NR / 2; o > 0; o >>= 1)
                                x += __shfl_xor_sync(0xffffffffu, x, o);
                            s[k] = x;
                        }
                }
            } else {
                __syncthreads();
                if (warp == 0)
                    for (int k = 0; k < nv; k++) s[k] = lsum[k];
            }
            if (tid == 0) {
                T cc[2] = {T(0), T(0)};
                coefs(s, cc);
                coef[0] = cc[0];
                coef[1] = cc[1];
            }
            __syncthreads();
            c[0] = coef[0];
            c[1] = coef[1];
        }
    };
    
    // alpha_i of Alg. 1 from the sums (p, q), (r, p), (r, r); c[1] = 1 if Alg. 1 has stopped
    auto alpha_of = [&](int lv, int i) {
        return [=](const T *s, T *c) {
            const bool prev = i > 0 && (stops[lv][i - 1] || s[2] == T(0));
            const bool stopped = prev || !(s[0] > T(0)) || !isfinite(s[0]);
            c[0] = stopped ? T(0) : (T)ratio<T>((double)s[1], (double)s[0]);
            c[1] = stopped ? T(1) : T(0);
        };
    };

    // one colour of a Gauss-Seidel sweep
    auto gs_colour = [&](const ClLev &L, int c, const T *f, T *z) {
        const ClColor C = ((const ClColor *)at(L.tab))[c];
        const int nwin = ((const ClHead *)at(L.head))->nwin;
        const T *val = (const T *)at(L.val), *dinv = (const T *)at(L.dinv);
        const unsigned short *col = (const unsigned short *)at(L.col);
        const uint32_t vec = cl_smem(z);
        for (int j = tid; j < C.cnt; j += kClThreads) {
            const int li = C.li0 + j;
            const T u = (f[li] - cl_row_dot(val, col, C.m0 + j, L.R, 1, L.w, z, nwin)) * dinv[li];
            z[li] = u;
            push_row(L, C, j, vec, u);
        }
        exchange(C.expect);
        mark(L.level, OP_GS);
    };
    // z = 0 on the window, except the colour whose values come next
    auto zero_window = [&](const ClLev &L, T *z) {
        const ClColor &C = ((const ClColor *)at(L.tab))[L.c_first];
        const int nwin = ((const ClHead *)at(L.head))->nwin;
        const int s0 = C.seg0, s1 = C.seg0 + C.seglen;
        for (int i = tid; i < nwin; i += kClThreads)
            if (i < s0 || i >= s1) z[i] = T(0);
    };

    // ---- entry: this strip's rows of the right-hand side -------------------------------
    if (y.nsp > 0) {
        const ClLev &L = y.lv[0];
        const ClColor *tab = (const ClColor *)at(L.tab);
        T *rhs = (T *)at(L.rhs), *z = (T *)at(L.p[0]);
        for (int c = 0; c < L.ncol; c++)
            for (int j = tid; j < tab[c].cnt; j += kClThreads)
                rhs[tab[c].li0 + j] = __ldcg(&a.rhs[tab[c].g0 + j]);
        zero_window(L, z);
        __syncthreads();
        const ClColor C = tab[L.c_first];
        const T *dinv = (const T *)at(L.dinv);
        const uint32_t vec = cl_smem(z);
        for (int j = tid; j < C.cnt; j += kClThreads) {
            const T u = rhs[C.li0 + j] * dinv[C.li0 + j];
            z[C.li0 + j] = u;
            push_row(L, C, j, vec, u);
        }
        exchange(C.expect);
        mark(L.level, OP_GS_FIRST);
    }
    {  // dense level's vectors: zero beyond its rows
        T *F = (T *)at(y.F);
        for (int i = tid; i < NR * y.ch; i += kClThreads)
            F[i] = (y.nsp == 0 && i < y.nd) ? __ldcg(&a.rhs[i]) : T(0);
    }
    __syncthreads();

    // ---- Alg. 2 / Alg. 1 over the levels ------------------------------------------------
    int lv = 0;            // current swept level
    unsigned long long steps = 0;  // Alg. 1 step of every swept level, 4 bits each
    for (;;) {
        if (y.nsp > 0) {  // B^ of level lv for step i: pre-smoothing, then the restriction
            const ClLev &L = y.lv[lv];
            const int i = (int)(steps >> (4 * lv)) & 15;
            const T *f = (const T *)at(i == 0 ? L.rhs : L.r);
            T *z = (T *)at(L.p[i]);
            for (int sw = 0; sw < y.nu_pre; sw++)
                for (int c = sw == 0 ? L.c_first + 1 : 0; c < L.ncol; c++)
                    if (L.cmask >> c & 1) gs_colour(L, c, f, z);
            const ClHead H = *(const ClHead *)at(L.head);
            const bool to_swept = lv + 1 < y.nsp;
            T *t = (T *)at(L.q[i]);  // free until step i's product writes it
            {
                const unsigned short *own = (const unsigned short *)at(L.own);
                const T *val = (const T *)at(L.val);
                const unsigned short *col = (const unsigned short *)at(L.col);
                for (int m = tid; m < H.nown; m += kClThreads) {
                    const int li = own[m];
                    t[li] = f[li] - cl_row_dot(val, col, m, L.R, 0, L.w, z, H.nwin);
                }
                if (to_swept) zero_window(y.lv[lv + 1], (T *)at(y.lv[lv + 1].p[0]));
            }
            __syncthreads();
            if (L.xchild) {
                push_all(L, L.q[i]);
                exchange(H.expect_all);
            }
            mark(L.level, OP_RESID);
            const unsigned short *child = (const unsigned short *)at(L.child);
            auto child_sum = [&](int m) {
                T v[8];
#pragma unroll
                for (int q = 0; q < 8; q++) {
                    const int ci = q < L.nch ? child[q * L.Rn + m] : 0xFFFF;
                    v[q] = (ci != 0xFFFF && idx_ok(ci, H.nwin)) ? t[ci] : T(0);
                }
                const T lo = (v[0] + v[1]) + (v[2] + v[3]);
                return L.nch == 8 ? lo + ((v[4] + v[5]) + (v[6] + v[7])) : lo;
            };
            if (to_swept) {
                const ClLev &N = y.lv[lv + 1];
                const int nown = ((const ClHead *)at(N.head))->nown;
                const unsigned short *own = (const unsigned short *)at(N.own);
                const ClColor C = ((const ClColor *)at(N.tab))[N.c_first];
                const T *dinv = (const T *)at(N.dinv);
                T *rhs = (T *)at(N.rhs), *zn = (T *)at(N.p[0]);
                const uint32_t vec = cl_smem(zn);
                for (int m = tid; m < nown; m += kClThreads) {
                    const int li = own[m];
                    const T v = child_sum(m);
                    rhs[li] = v;
                    const int j = m - C.m0;
                    if ((unsigned)j < (unsigned)C.cnt) {
                        const T u = v * dinv[li];
                        zn[li] = u;
                        push_row(N, C, j, vec, u);
                    }
                }
                exchange(C.expect);
                mark(L.level, OP_RESTRICT);
                lv++;
                steps &= ~(15ull << (4 * lv));
                continue;
            }
            // into the dense level: every CTA gets every row
            const int nown = *(const int *)at(y.dhead);
            T *stage = (T *)at(y.stage);
            for (int m = tid; m < nown; m += kClThreads) stage[m] = child_sum(m);
            __syncthreads();
            if (alive) {
                const unsigned short *pi = (const unsigned short *)at(y.down);
                const uint32_t vec = cl_smem(at(y.F)), mb = mb_all();
                for (int k = tid; k < NR * nown; k += kClThreads)
                    cl_store(cl_map(vec + (uint32_t)sizeof(T) * pi[k >> 4], k & (NR - 1)), stage[k >> 4],
                             cl_map(mb, k & (NR - 1)));
            }
            wait_all((int)sizeof(T) * y.nd);
            mark(L.level, OP_RESTRICT);
        }
        // ---- the dense level: e = B~ [F] ------------------------------------------------
        {
            const int ch = y.ch, len = NR * ch;
            const int dl = y.tl + y.nsp;  // its level number
            T *E = (T *)at(y.E), *out = (T *)at(y.out);
            auto gather_out = [&](int dst0, int dst1, int parts) {  // `out` to every CTA
                constexpr int V = 16 / (int)sizeof(T);
                const int per = ch / V;  // 16-byte pieces per part
                if (alive)
                    for (int k = tid; k < NR * parts * per; k += kClThreads) {
                        const int dst = k & (NR - 1), piece = k >> 4;
                        const int part = piece >= per, o = (piece - part * per) * V;
                        const uint32_t to = cl_smem(at(part ? dst1 : dst0)) +
                                            (uint32_t)sizeof(T) * (rank * ch + o);
                        cl_store16(cl_map(to, dst), out + part * ch + o, cl_map(mb_all(), dst));
                    }
                wait_all((int)sizeof(T) * parts * len);
            };
            constexpr int LPR = 8;  // lanes per row
            const int q = tid & (LPR - 1);
            if (!y.dense) {  // coarsest level: e = A^{-1} F (FP32: op_coarse's compensated sum)
                const T *F = (const T *)at(y.F);
                for (int row = tid / LPR; row < ch; row += kClThreads / LPR) {
                    const T *m = (const T *)at(y.mat) + (size_t)row * y.stride;
                    if constexpr (!F64) {
                        const T *ml = (const T *)at(y.mat_lo) + (size_t)row * y.stride;
                        float s = 0.f, cs = 0.f;
                        for (int j = q; j < y.nd; j += LPR) {
                            const float x = F[j];
                            const float ph = __fmul_rn(m[j], x);
                            const float pe = fmaf(ml[j], x, fmaf(m[j], x, -ph));
                            float t2, e2;
                            two_sum(s, ph, t2, e2);
                            s = t2;
                            cs = __fadd_rn(cs, __fadd_rn(e2, pe));
                        }
#pragma unroll
                        for (int o = LPR / 2; o > 0; o >>= 1) {
                            const float so = __shfl_down_sync(0xffffffffu, s, o, LPR);
                            const float co = __shfl_down_sync(0xffffffffu, cs, o, LPR);
                            float t2, e2;
                            two_sum(s, so, t2, e2);
                            s = t2;
                            cs = __fadd_rn(cs, __fadd_rn(co, e2));
                        }
                        if (q == 0) out[row] = __fadd_rn(s, cs);
                    } else {
                        double s = 0.0;
                        for (int j = q; j < y.nd; j += LPR) s += m[j] * F[j];
#pragma unroll
                        for (int o = LPR / 2; o > 0; o >>= 1) s += __shfl_down_sync(0xffffffffu, s, o, LPR);
                        if (q == 0) out[row] = s;
                    }
                }
                __syncthreads();
                gather_out(y.E, y.E, 1);
                mark(dl, OP_COARSE);
            } else {
                T *Rv = (T *)at(y.Rv);
                const int nact = (y.nd + 31) / 32;
                for (int i = 0; i < y.kc; i++) {
                    // [z; w] = [M; A M] r: this CTA's rows, 16-byte reads
                    const T *x = (const T *)at(i == 0 ? y.F : y.Rv);
                    constexpr int V = 16 / (int)sizeof(T);
                    for (int row = tid / LPR; row < 2 * ch; row += kClThreads / LPR) {
                        const T *m = (const T *)at(y.mat) + (size_t)row * y.stride;
                        T s = 0;
                        for (int j = q * V; j < len; j += LPR * V) {
                            if constexpr (!F64) {
                                const float4 mv = *(const float4 *)(m + j), xv = *(const float4 *)(x + j);
                                s += mv.x * xv.x;
                                s += mv.y * xv.y;
                                s += mv.z * xv.z;
                                s += mv.w * xv.w;
                            } else {
                                const double2 mv = *(const double2 *)(m + j), xv = *(const double2 *)(x + j);
                                s += mv.x * xv.x;
                                s += mv.y * xv.y;
                            }
                        }
#pragma unroll
                        for (int o = LPR / 2; o > 0; o >>= 1) s += __shfl_down_sync(0xffffffffu, s, o, LPR);
                        if (q == 0) out[row] = s;
                    }
                    __syncthreads();
                    gather_out(y.P[i], y.Q[i], 2);
                    // Alg. 1 step i, the same in every CTA
                    T *p = (T *)at(y.P[i]), *qv = (T *)at(y.Q[i]);
                    const T *r = x;
                    T c[2];
                    if (i > 0) {
                        T v[3] = {T(0), T(0), T(0)};
                        for (int k = tid; k < y.nd; k += kClThreads)
#pragma unroll
                            for (int j = 0; j < 3; j++)
                                if (j < i) v[j] += p[k] * ((const T *)at(y.Q[j]))[k];
                        for (int j = 0; j < i; j++) {  // one coefficient per sum
                            T vj[3] = {j == 0 ? v[0] : j == 1 ? v[1] : v[2], T(0), T(0)};
                            reduce(std::false_type{}, vj, 1, nact,
                                   [&](const T *s, T *cc) {
                                       const T pq = pqs[kClLevels][j];
                                       cc[0] = pq > T(0) ? -(T)ratio<T>((double)s[0], (double)pq) : T(0);
                                   },
                                   c);
                            const T *pj = (const T *)at(y.P[j]), *qj = (const T *)at(y.Q[j]);
                            for (int k = tid; k < y.nd; k += kClThreads) {
                                p[k] += c[0] * pj[k];
                                qv[k] += c[0] * qj[k];
                            }
                        }
                    }
                    T v[3] = {T(0), T(0), T(0)};
                    for (int k = tid; k < y.nd; k += kClThreads) {
                        v[0] += p[k] * qv[k];
                        v[1] += r[k] * p[k];
                        v[2] += r[k] * r[k];
                    }
                    auto f = alpha_of(kClLevels, i);
                    reduce(std::false_type{}, v, 3, nact,
                           [&](const T *s, T *cc) {
                               f(s, cc);
                               if (tid == 0) {
                                   pqs[kClLevels][i] = s[0];
                                   stops[kClLevels][i] = cc[1] != T(0);
                               }
                           },
                           c);
                    const T al = c[0];
                    const bool last = i == y.kc - 1;
                    for (int k = tid; k < y.nd; k += kClThreads) {
                        E[k] = i == 0 ? al * p[k] : E[k] + al * p[k];
                        if (!last) Rv[k] = r[k] - al * qv[k];
                    }
                    if (i == 0 && !last)
                        for (int k = y.nd + tid; k < len; k += kClThreads) Rv[k] = T(0);
                    __syncthreads();
                }
                mark(dl, OP_COARSE);
            }
        }
        if (y.nsp == 0) break;
        // ---- back up: B^ of level lv after the correction, Alg. 1 step i ------------------
        bool done = false;
        for (;;) {
            const ClLev &L = y.lv[lv];
            const int i = (int)(steps >> (4 * lv)) & 15;
            const ClHead H = *(const ClHead *)at(L.head);
            const ClColor *tab = (const ClColor *)at(L.tab);
            const T *f = (const T *)at(i == 0 ? L.rhs : L.r);
            T *z = (T *)at(L.p[i]);
            {  // z += P e on the window; the colour swept next is overwritten unread
                const bool from_swept = lv + 1 < y.nsp;
                const T *en = (const T *)at(from_swept ? y.lv[lv + 1].e : y.E);
                const unsigned short *par = (const unsigned short *)at(L.parent);
                const int s0 = tab[L.c_last].seg0, s1 = s0 + tab[L.c_last].seglen;
                for (int k = tid; k < H.nwin; k += kClThreads)
                    if (k < s0 || k >= s1) z[k] += en[par[k]];
                __syncthreads();
                mark(L.level, OP_PROLONG);
            }
            for (int sw = 0; sw < y.nu_post; sw++)
                for (int c = L.c_last; c >= 0; c--)
                    if (L.cmask >> c & 1) gs_colour(L, c, f, z);
            const unsigned short *own = (const unsigned short *)at(L.own);
            const int nact = (H.nown + 31) / 32;
            const bool last = i == y.kc - 1;
            T c[2];
            if (i > 0) {  // p_i = z + sum_j beta_j p_j, on the window
                T v[3] = {T(0), T(0), T(0)};
                for (int m = tid; m < H.nown; m += kClThreads) {
                    const int li = own[m];
                    const T zl = z[li];
#pragma unroll
                    for (int j = 0; j < 3; j++)
                        if (j < i) v[j] += zl * ((const T *)at(L.q[j]))[li];
                }
                for (int j = 0; j < i; j++) {
                    T vj[3] = {j == 0 ? v[0] : j == 1 ? v[1] : v[2], T(0), T(0)};
                    reduce(std::true_type{}, vj, 1, nact,
                           [&](const T *s, T *cc) {
                               const T pq = pqs[lv][j];
                               cc[0] = pq > T(0) ? -(T)ratio<T>((double)s[0], (double)pq) : T(0);
                           },
                           c);
                    mark(L.level, OP_MULTIDOT);
                    const T *pj = (const T *)at(L.p[j]);
                    for (int k = tid; k < H.nwin; k += kClThreads) z[k] += c[0] * pj[k];
                }
                __syncthreads();
                mark(L.level, OP_ORTH);
            }
            T *qv = (T *)at(L.q[i]);
            {  // q = A p; (p, q), (r, p), (r, r)
                const T *val = (const T *)at(L.val);
                const unsigned short *col = (const unsigned short *)at(L.col);
                T v[3] = {T(0), T(0), T(0)};
                for (int m = tid; m < H.nown; m += kClThreads) {
                    const int li = own[m];
                    const T acc = cl_row_dot(val, col, m, L.R, 0, L.w, z, H.nwin);
                    qv[li] = acc;
                    const T pl = z[li], rl = f[li];
                    v[0] += pl * acc;
                    v[1] += rl * pl;
                    v[2] += rl * rl;
                }
                if (!last) zero_window(L, (T *)at(L.p[i + 1]));
                auto fa = alpha_of(lv, i);
                reduce(std::true_type{}, v, 3, nact,
                       [&](const T *s, T *cc) {
                           fa(s, cc);
                           if (tid == 0) {
                               pqs[lv][i] = s[0];
                               stops[lv][i] = cc[1] != T(0);
                           }
                       },
                       c);
                mark(L.level, OP_SPMV_DOT);
            }
            {  // e (+)= alpha p, r = r - alpha q; the next step's first colour
                const T al = c[0];
                T *e = (T *)at(L.e), *r = (T *)at(L.r);
                const ClColor C = tab[L.c_first];
                const T *dinv = (const T *)at(L.dinv);
                T *zn = last ? nullptr : (T *)at(L.p[i + 1]);
                const uint32_t vec = last ? 0 : cl_smem(zn);
                for (int m = tid; m < H.nown; m += kClThreads) {
                    const int li = own[m];
                    e[li] = i == 0 ? al * z[li] : e[li] + al * z[li];
                    if (!last) {
                        const T rn = f[li] - al * qv[li];
                        r[li] = rn;
                        const int j = m - C.m0;
                        if ((unsigned)j < (unsigned)C.cnt) {
                            const T u = rn * dinv[li];
                            zn[li] = u;
                            push_row(L, C, j, vec, u);
                        }
                    }
                }
                if (!last) {
                    exchange(C.expect);
                } else if (lv > 0) {  // e, to the windows the prolongation reads
                    __syncthreads();
                    push_all(L, L.e);
                    exchange(H.expect_all);
                }
                mark(L.level, OP_UPDATE);
            }
            if (!last) {
                steps += 1ull << (4 * lv);
                break;  // B^ for the next step
            }
            if (lv == 0) {
                done = true;
                break;
            }
            lv--;
        }
        if (done) break;
    }
    __syncthreads();
    if (alive) {
        if (y.nsp > 0) {
            const ClLev &L = y.lv[0];
            const ClColor *tab = (const ClColor *)at(L.tab);
            const T *e = (const T *)at(L.e);
            for (int c = 0; c < L.ncol; c++)
                for (int j = tid; j < tab[c].cnt; j += kClThreads)
                    a.e[tab[c].g0 + j] = e[tab[c].li0 + j];
        } else {
            const T *E = (const T *)at(y.E);
            for (int i = rank * y.ch + tid; i < min(y.nd, (rank + 1) * y.ch); i += kClThreads)
                a.e[i] = E[i];
        }
    }
    if (mark_on)
        for (int k = 0; k < 16 * (y.nsp + 1); k++)
            if (prof_s[1][k]) {
                a.tprof[16 * y.tl + k] += prof_s[0][k];
                a.tprof[16 * kMaxLevels + 16 * y.tl + k] += prof_s[1][k];
            }
    cl_sync_all();  // no CTA leaves while a neighbour may still write into it
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
// window tables: [level][rank][colour] (first, last + 1); cwin: the children's part alone
__device__ __forceinline__ void cl_extend(int2 *w, int i) {
    volatile int *v = (volatile int *)w;
    if (i < v[0]) atomicMin(&w->x, i);
    if (i + 1 > v[1]) atomicMax(&w->y, i + 1);
}
__device__ __forceinline__ int2 *cl_win(int2 *win, int a, int r, int c) {
    return win + ((size_t)a * kClRanks + r) * kClColors + c;
}

// columns of own rows, both ways, and children of own next-level rows in other strips
__global__ void k_cl_windows(const __grid_constant__ ClSrcs G, int2 *win, int2 *cwin) {
    const int a = blockIdx.y;
    const ClSrc &S = G.lv[a], &N = G.lv[a + 1];
    const int i = blockIdx.x * blockDim.x + threadIdx.x;
    if (i < S.n) {
        const int c = cl_colour(S, i), r = cl_owner(S, c, i);
        const int s0 = S.sl[i >> 5], width = (S.sl[(i >> 5) + 1] - s0) >> 5;
        for (int k = 1; k < width; k++) {
            const int j = S.col[s0 + 32 * k + (i & 31)];
            if (j < 0) continue;
            const int cj = cl_colour(S, j), rj = cl_owner(S, cj, j);
            if (rj == r) continue;
            cl_extend(cl_win(win, a, r, cj), j);
            cl_extend(cl_win(win, a, rj, c), i);
        }
    }
    if (i < N.n) {
        const int rn = cl_owner(N, cl_colour(N, i), i);
        for (int q = 0; q < (S.ch2 ? 8 : 4); q++) {
            const int4 ch = (q < 4 ? S.ch : S.ch2)[i];
            const int j = (q & 3) == 0 ? ch.x : (q & 3) == 1 ? ch.y : (q & 3) == 2 ? ch.z : ch.w;
            if (j < 0) continue;
            const int cj = cl_colour(S, j);
            if (cl_owner(S, cj, j) != rn) cl_extend(cl_win(cwin, a, rn, cj), j);
        }
    }
}

// one CTA, level by level: the children's part joins the window; then the parents of the
// window's rows join the next level's window
__global__ void __launch_bounds__(1024) k_cl_parents(const __grid_constant__ ClSrcs G, int2 *win,
                                                     const int2 *cwin) {
    const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
    for (int a = 0; a < G.nsp; a++) {
        const ClSrc &S = G.lv[a];
        for (int k = threadIdx.x; k < kClRanks * S.ncol; k += blockDim.x) {
            const int r = k / S.ncol, c = k - r * S.ncol;
            const size_t o = ((size_t)a * kClRanks + r) * kClColors + c;
            if (cwin[o].x < cwin[o].y) {
                win[o].x = min(win[o].x, cwin[o].x);
                win[o].y = max(win[o].y, cwin[o].y);
            }
        }
        __syncthreads();
        if (a + 1 < G.nsp) {
            const ClSrc &N = G.lv[a + 1];
            for (int k = warp; k < kClRanks * S.ncol; k += (int)(blockDim.x >> 5)) {
                const int r = k / S.ncol, c = k - r * S.ncol;
                const int2 w = *cl_win(win, a, r, c);
                for (int i = w.x + lane; i < w.y; i += 32) {
                    const int p = S.parent[i];
                    cl_extend(cl_win(win, a + 1, r, cl_colour(N, p)), p);
                }
            }
            __syncthreads();
        }
    }
}

// the constant image of strip blockIdx.y, level blockIdx.z (nsp: the coarsest inverse); the
// tables at its start are there already
template <class T>
__global__ void k_cl_image(const __grid_constant__ ClSrcs G, const __grid_constant__ ClLayout y,
                           unsigned char *image, const double *Ainv, const float *Ainv2) {
    const int a = blockIdx.z, r = blockIdx.y;
    unsigned char *im = image + (size_t)r * y.image_bytes;
    const int t0 = blockIdx.x * blockDim.x + threadIdx.x, nt = gridDim.x * blockDim.x;
    if (a == y.nsp) {
        if (y.dense) return;
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
    const ClColor *tab = (const ClColor *)(im + L.tab);
    T *val = (T *)(im + L.val), *dinv = (T *)(im + L.dinv);
    unsigned short *col = (unsigned short *)(im + L.col), *own = (unsigned short *)(im + L.own);
    unsigned short *par = (unsigned short *)(im + L.parent), *child = (unsigned short *)(im + L.child);
    auto local = [&](const ClColor *tb, const ClSrc &s, int i) {  // window index of pi-row i
        const ClColor &C = tb[cl_colour(s, i)];
        return (unsigned short)(C.li0 + i - C.g0);
    };
    for (int m = t0; m < H.nown; m += nt) {
        int c = 0;
        while (c + 1 < L.ncol && m >= tab[c + 1].m0) c++;
        const int i = tab[c].g0 + m - tab[c].m0;
        const int li = tab[c].li0 + m - tab[c].m0;
        own[m] = (unsigned short)li;
        const int s0 = S.sl[i >> 5], width = (S.sl[(i >> 5) + 1] - s0) >> 5;
        for (int k = 0; k < L.w; k++) {
            const int o = s0 + 32 * k + (i & 31);
            const int j = k < width ? S.col[o] : -1;
            col[k * L.R + m] = j >= 0 ? local(tab, S, j) : (unsigned short)li;
            T v = T(0);
            if (j >= 0) {
                if constexpr (sizeof(T) == 8) v = S.val64[o];
                else v = S.val32[o];
            }
            val[k * L.R + m] = v;
        }
        dinv[li] = (T)(1.0 / S.val64[s0 + (i & 31)]);
    }
    const bool swept = a + 1 < y.nsp;
    const ClColor *ntab = swept ? (const ClColor *)(im + y.lv[a + 1].tab) : nullptr;
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
        for (int q = 0; q < L.nch; q++) {
            const int4 ch = (q < 4 ? S.ch : S.ch2)[R];
            const int j = (q & 3) == 0 ? ch.x : (q & 3) == 1 ? ch.y : (q & 3) == 2 ? ch.z : ch.w;
            child[q * L.Rn + m] = j >= 0 ? local(tab, S, j) : (unsigned short)0xFFFF;
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
            const int4 ch = (q < 4 ? S.ch : S.ch2)[R];
            const int j = (q & 3) == 0 ? ch.x : (q & 3) == 1 ? ch.y : (q & 3) == 2 ? ch.z : ch.w;
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
        T *row = (T *)(image + (size_t)(i / y.ch) * y.image_bytes + y.mat) + (size_t)(i % y.ch) * y.stride;
        row[unit] = (T)z[i];
        row[(size_t)y.ch * y.stride + unit] = (T)dot(i, 0);
    }
}

}  // namespace amg
