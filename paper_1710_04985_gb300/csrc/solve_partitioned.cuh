// Partitioned self-scheduled solve, one right-hand side, on the plan's sliced
// copy in part order (SPTRSV_ALGO_SELF_PARTITIONED; layout in solve_parts.cu): a
// thread block takes one part (consecutive rows, by level inside the part) and
// keeps the part's unknowns in shared memory.
//
// What bounds it: the chain of dependent rows.  A hop inside a part costs a
// shared-memory poll, the FMAs that follow the last arrival (an FP64
// instruction holds its SM sub-partition's FP64 unit for ~64 cycles) and the
// publication; a hop between parts costs an L2 handshake.  A warp runs this
// code at 4 to 5 cycles per instruction, so instructions count as much as
// memory: what can be decided when the copy is built is not decided here.
//  * A group is at most 32/W rows of ONE level of the part, so no row of a warp
//    waits for another row of it, and the warp waits, folds and publishes as
//    one, without divergence.
//  * An entry's slot says whether it belongs to an earlier part or to this one,
//    and its column is the address to poll; lanes without an entry read a word
//    that holds 0.  Loads need nothing but the group's descriptor.
//  * Entries of earlier parts come first in fold order: they are polled in L2,
//    or in another block's shared memory (clusters), and folded; then the
//    part's own values are polled in shared memory only, so that no polling
//    round of this second wait is an L2 round trip.
//  * Warps take the part's groups in turn, so the next group is known: its rows
//    and entries are loaded before the waits of the current one.
//  * What the part reads is prefetched into L2 by bulk requests: rows, 1/d(i)
//    and b when the part is taken, slices a fixed distance ahead of the groups
//    being solved (all at once, the parts of a large matrix evict each other's).
// A warp that does not get all its values within a quarter of the spin limit
// goes on in slow_group(), in which every row is folded and published by itself;
// a value that never comes (spin limit) thus holds up only the
// rows that depend on it.
//
// Measured against the blocked kernel on a CSR copy that served this form
// before (its rounds polled both kinds of dependency and a group could straddle
// levels): L and U of the 128^3 ILU(0), FP64, parts of 16384 rows, clusters of 4:
// 678 -> 490 us; both triangles of the 9-point 1021 x 1023 grid, FP32, 4 lanes,
// parts of 8192 rows: 3.73 -> 1.38 ms; 27-point 61 x 47 x 53, FP64: 0.44 -> 0.24 ms;
// 128 general systems, 16 lanes: 3.88 -> 3.62 ms.
//
// Deadlock freedom: parts are taken in order, and a part depends on itself and
// on earlier parts.  Inside a part every warp solves its groups in ascending
// order, so the smallest unfinished group is its warp's current one, and it
// waits only for finished groups or earlier parts.  Every wait is bounded.  Rows are folded and reduced in the order of the other
// self-scheduled forms, so results are bitwise theirs at the same width.
#pragma once

#include "internal.h"

namespace sptrsv {

namespace {

constexpr int kMaxCluster = 8;
constexpr int kMaxBlock = 512;
constexpr long long kNoEnd = 1ll << 62;  // polls: the wait ends by the spin limit

// Brings [p, p + bytes) into L2 with one instruction, rounded inwards to the
// 16-byte pieces it works on.
__device__ __forceinline__ void prefetch_range(const void* p, long long bytes) {
    const unsigned long long a = (unsigned long long)p, lo = (a + 15) & ~15ull;
    const unsigned long long hi = (a + (unsigned long long)bytes) & ~15ull;
    if (hi > lo)
        asm volatile("cp.async.bulk.prefetch.L2.global [%0], %1;" ::"l"(lo),
                     "r"((unsigned)(hi - lo)));
}

// ---- shared memory by 32-bit address
__device__ __forceinline__ unsigned smem_addr(const void* p) {
    return (unsigned)__cvta_generic_to_shared(p);
}
__device__ __forceinline__ double lds(unsigned a, double) {
    unsigned long long v;
    asm volatile("ld.volatile.shared.b64 %0, [%1];" : "=l"(v) : "r"(a) : "memory");
    return __longlong_as_double((long long)v);
}
__device__ __forceinline__ float lds(unsigned a, float) {
    unsigned v;
    asm volatile("ld.volatile.shared.b32 %0, [%1];" : "=r"(v) : "r"(a) : "memory");
    return __uint_as_float(v);
}

// ---- thread-block clusters: distributed shared memory of the cluster's blocks
__device__ __forceinline__ unsigned cluster_rank() {
    unsigned r;
    asm volatile("mov.u32 %0, %%cluster_ctarank;" : "=r"(r));
    return r;
}
// Every thread of every block of the cluster; orders shared-memory accesses
// around it across the cluster.
__device__ __forceinline__ void cluster_sync() {
    asm volatile("barrier.cluster.arrive.release.aligned;\n\tbarrier.cluster.wait.acquire.aligned;"
                 ::: "memory");
}
// Address `a` of this block's shared memory in block `rank`'s.
__device__ __forceinline__ unsigned cluster_addr(unsigned a, unsigned rank) {
    unsigned r;
    asm volatile("mapa.shared::cluster.u32 %0, %1, %2;" : "=r"(r) : "r"(a), "r"(rank));
    return r;
}
__device__ __forceinline__ double ld_cluster(unsigned a, double) {
    unsigned long long v;
    asm volatile("ld.relaxed.cluster.shared::cluster.b64 %0, [%1];" : "=l"(v) : "r"(a) : "memory");
    return __longlong_as_double((long long)v);
}
__device__ __forceinline__ float ld_cluster(unsigned a, float) {
    unsigned v;
    asm volatile("ld.relaxed.cluster.shared::cluster.b32 %0, [%1];" : "=r"(v) : "r"(a) : "memory");
    return __uint_as_float(v);
}
__device__ __forceinline__ int ld_cluster_int(unsigned a) {
    int v;
    asm volatile("ld.relaxed.cluster.shared::cluster.b32 %0, [%1];" : "=r"(v) : "r"(a) : "memory");
    return v;
}
// Publication into this block's shared memory, visible to the cluster.
__device__ __forceinline__ void st_cluster(unsigned a, double v) {
    asm volatile("st.relaxed.cluster.shared::cta.b64 [%0], %1;" ::"r"(a),
                 "l"((unsigned long long)__double_as_longlong(v))
                 : "memory");
}
__device__ __forceinline__ void st_cluster(unsigned a, float v) {
    asm volatile("st.relaxed.cluster.shared::cta.b32 [%0], %1;" ::"r"(a), "r"(__float_as_uint(v))
                 : "memory");
}

// What a warp knows about its part.
struct PartCtx {
    int p0;              // the part's first position
    int g0;              // the cluster's first position (p0 without clusters)
    unsigned xs_a;       // shared-memory address of the part's unknowns
    unsigned crank;      // rank of this block in its cluster
    const int* pst;      // first position of each part of the cluster (shared memory)
};

// Address of the unknown at position pos (g0 <= pos < p0) in the shared memory
// of the cluster's block that holds it.
template <typename T>
__device__ __forceinline__ unsigned remote_addr(const PartCtx& c, int pos) {
    unsigned r = 0;
    for (unsigned j = 1; j < c.crank; ++j)
        if (c.pst[j] <= pos) r = j;
    return cluster_addr(c.xs_a + (unsigned)(pos - c.pst[r]) * (unsigned)sizeof(T), r);
}

// Published value of an earlier part: at a position, or (remote) at an address
// in the cluster's shared memory.
template <typename T, bool CL>
__device__ __forceinline__ T poll_ext(const T* xp, int at, bool remote) {
    if (CL && remote) return ld_cluster((unsigned)at, T(0));
    return ld_relaxed(xp + at);
}

template <typename T>
__device__ __forceinline__ void publish_global(const SolveParams& p, int k, int i, T xi,
                                               double xbase) {
    st_relaxed((T*)p.xp + k, xi);
    if (p.xacc)
        accumulate_with(p, i, 0, xi, xbase);
    else
        ((T*)p.x)[(long long)i * p.ldx] = xi;
}

}  // namespace

// One group in the general way: every row is folded as its values come and
// published by itself.  Starts from the stored data, and skips rows that are
// published already, so it can be given up (false) after `budget` polls without
// an end and taken up again.
template <typename T, int W, bool CL>
__device__ __noinline__ bool slow_group(const SolveParams& p, const PartCtx& ctx, int g,
                                        long long budget) {
    constexpr int E = kChunk;
    constexpr unsigned FULL = 0xffffffffu;
    const int lane = threadIdx.x & 31, grp = lane / W, sl = lane - grp * W;
    const unsigned gmask = group_mask<W>(lane);
    const int4 d = p.grp[g];
    const int X = d.z, S = d.z + (d.w >> 12), span = (d.w >> 6) & 63;
    const int k = d.x + grp;
    const bool has_row = grp < (d.w & 63);
    const int off = k - ctx.p0;
    const unsigned own = ctx.xs_a + (unsigned)off * (unsigned)sizeof(T);
    int i = -1;
    T sum = T(0);
    double xbase = 0.0;
    bool published = true;
    if (has_row) {
        i = p.jlev[k];
        published = !Marker<T>::pending(lds(own, T(0)));
        if (sl == 0) {
            sum = ((const T*)p.b)[(long long)i * p.ldb];
            if (!p.unit) sum *= ((const T*)p.dinv)[k];
            xbase = accumulate_base(p, i, 0);
        }
    }
    const long long at = (long long)d.y * 32 + lane;
    int s0 = 0, c[E];
    T a[E], v[E];
    unsigned live = 0, pend = 0;
    auto poll = [&](int e) -> T {
        if (s0 + e >= X) return lds(ctx.xs_a + (unsigned)c[e] * (unsigned)sizeof(T), T(0));
        const bool remote = CL && c[e] >= ctx.g0;
        return poll_ext<T, CL>((const T*)p.xp, remote ? (int)remote_addr<T>(ctx, c[e]) : c[e],
                               remote);
    };
    auto load_chunk = [&]() {
        live = 0;
#pragma unroll
        for (int e = 0; e < E; ++e) {
            const int s = s0 + e;
            c[e] = -1;
            a[e] = v[e] = T(0);
            if (s < S) {
                c[e] = p.idx[at + 32ll * s];
                a[e] = ((const T*)p.vals)[at + 32ll * s];
                if (c[e] != (s < X ? -1 : p.max_part)) live |= 1u << e;
            }
        }
        pend = live;
    };
    // lanes of published rows have nothing left to do
    bool lane_done = published || S == 0;
    if (!lane_done) load_chunk();
    long long waits = 0, total = 0;
    unsigned ns = 32;
    while (true) {
        if (!lane_done && pend == 0) {
            if (live) sum = fold_chunk(sum, a, v, live);
            s0 += E;
            if (s0 >= S)
                lane_done = true;
            else
                load_chunk();
        }
        const unsigned done = __ballot_sync(FULL, lane_done);
        const bool fresh = !published && (done & gmask) == gmask;
        if (__any_sync(FULL, fresh)) {
            const T tot = group_sum_span<W>(sum, FULL, span);
            if (fresh && sl == 0 && i != p.withhold) {
                const T xi = publishable(tot);
                st_cluster(own, xi);
                publish_global(p, k, i, xi, xbase);
            }
        }
        published = published || fresh;
        if (__all_sync(FULL, published)) return true;
        if (__any_sync(FULL, !lane_done && pend == 0)) continue;  // fold first
        if (!__any_sync(FULL, pend != 0)) {
            waits = 0;
            ns = 32;
            continue;
        }
        const unsigned before = pend;
        do {
#pragma unroll
            for (int e = 0; e < E; ++e)
                if (pend & (1u << e)) v[e] = poll(e);
#pragma unroll
            for (int e = 0; e < E; ++e)
                if ((pend & (1u << e)) && !Marker<T>::pending(v[e])) pend &= ~(1u << e);
            if (++total > budget) return false;
            if (++waits >= p.spin.limit) {
                if (pend) {
                    report(p.status, i, kCodeTimeout);
#pragma unroll
                    for (int e = 0; e < E; ++e)
                        if (pend & (1u << e)) v[e] = Marker<T>::canonical_nan();
                    pend = 0;
                }
                waits = 0;
                break;
            }
            if (__any_sync(FULL, pend != before)) break;
            if (waits >= p.spin.hot) {
                __nanosleep(ns);
                ns = ns < p.spin.max_ns ? ns * 2 : p.spin.max_ns;
            }
        } while (true);
    }
}

// Waits for the values of N shared-memory slots; false if they have not all come
// within `patience` polls.  A wait of more than kHotPolls leaves the issue slots
// to the warps that are nearer to the frontier.
constexpr int kHotPolls = 64;
template <typename T, int N>
__device__ __forceinline__ bool wait_slots(const unsigned (&c)[N], T (&v)[N], long long patience) {
    long long polls = 0;
    while (true) {
        bool pend = false;
#pragma unroll
        for (int e = 0; e < N; ++e) v[e] = lds(c[e], T(0));
#pragma unroll
        for (int e = 0; e < N; ++e) pend |= Marker<T>::pending(v[e]);
        if (!__any_sync(0xffffffffu, pend)) return true;
        if (++polls > kHotPolls) {
            if (polls > patience) return false;
            __nanosleep(32);
        }
    }
}

// Folds the last r of N slots in order (1 <= r <= N, uniform).  A lane without
// an entry in a folded slot adds -0 * 0, which changes nothing.  In FP64 the
// unused slots are branched around (64 cycles each); in FP32 they are folded too.
__device__ __forceinline__ float fold_slots(float sum, const float (&a)[4], const float (&v)[4],
                                            int) {
#pragma unroll
    for (int e = 0; e < 4; ++e) sum = fmaf(-a[e], v[e], sum);
    return sum;
}
__device__ __forceinline__ double fold_slots(double sum, const double (&a)[4],
                                             const double (&v)[4], int r) {
    if (r >= 3) {
        if (r == 4) sum = fma(-a[0], v[0], sum);
        sum = fma(-a[1], v[1], sum);
    }
    if (r >= 2) sum = fma(-a[2], v[2], sum);
    return fma(-a[3], v[3], sum);
}
// Sum over a row's lanes.  FP32 adds every level (a branch costs more).
template <int W>
__device__ __forceinline__ float row_sum(float v, int) {
    return group_sum<W>(v, 0xffffffffu);
}
template <int W>
__device__ __forceinline__ double row_sum(double v, int span) {
    return group_sum_span<W>(v, 0xffffffffu, span);
}

// CL: clusters of cs blocks.  A cluster takes cs consecutive parts at once (one
// ticket), block r the r-th; a dependency on one of the earlier parts of the
// same cluster is read from that block's shared memory.  Three cluster
// barriers per ticket: after it is taken, after every block has read it and
// reset its part's unknowns, and when every block is done (no block reuses, or
// exits with, shared memory another still reads).
template <typename T, int W, bool CL>
__global__ void __launch_bounds__(kMaxBlock, 1) part_solve_k1(const __grid_constant__ SolveParams p,
                                                      int cs) {
    extern __shared__ __align__(16) unsigned char part_smem[];
    // max_part unknowns, the word that reads 0, and one that nobody reads
    T* xs = (T*)part_smem;
    __shared__ int s_part;
    __shared__ int s_pst[kMaxCluster];
    constexpr int NI = kOwnChunk;  // own-part slots, and
    constexpr int NX = kExtChunk;  // earlier-part slots of a group loaded ahead
    constexpr unsigned FULL = 0xffffffffu;
    const int lane = threadIdx.x & 31;
    const int warp = threadIdx.x >> 5;
    const int nw = blockDim.x >> 5;
    const int grp = lane / W;
    const int sl = lane - grp * W;
    const T* b = (const T*)p.b;
    const T* xp = (const T*)p.xp;
    const int n = p.n;
    // polls of one wait before the general way takes over
    const long long patience = p.spin.limit / 4 + 1;
    PartCtx ctx;
    ctx.xs_a = smem_addr(xs);
    ctx.crank = CL ? cluster_rank() : 0u;
    ctx.pst = s_pst;
    const int zero = p.max_part;  // column of a slot without an entry
    if (threadIdx.x == 0) xs[zero] = T(0);
    auto part_start = [&](long long j) -> int { return j < p.nparts ? p.part_ptr[j] : n; };
    auto prefetch_slices = [&](int q0, int q1) {
        prefetch_range(p.idx + 32ll * q0, 128ll * (q1 - q0));
        prefetch_range((const T*)p.vals + 32ll * q0, 32ll * (long long)sizeof(T) * (q1 - q0));
    };
    while (true) {
        long long part;
        if (!CL) {
            if (threadIdx.x == 0) s_part = atomicAdd(p.ticket, 1);
            __syncthreads();
            part = s_part;
            if (part >= p.nparts) break;
            ctx.g0 = ctx.p0 = part_start(part);
        } else {
            if (ctx.crank == 0 && threadIdx.x == 0) s_part = atomicAdd(p.ticket, 1);
            cluster_sync();
            const long long t =
                ctx.crank == 0 ? s_part : ld_cluster_int(cluster_addr(smem_addr(&s_part), 0));
            part = t * cs + ctx.crank;
            ctx.g0 = part_start(t * cs);
            ctx.p0 = part_start(part);
            if ((int)threadIdx.x < cs) s_pst[threadIdx.x] = part_start(t * cs + threadIdx.x);
        }
        const int in_part = part_start(part + 1) - ctx.p0;
        const int gfirst = part < p.nparts ? p.grp_ptr[part] : 0;
        const int gend = part < p.nparts ? p.grp_ptr[part + 1] : 0;
        int qend = 0, qahead = 0;  // end of the part's slices; slices to prefetch ahead
        if (gend > gfirst) {
            const int4 d0 = p.grp[gfirst], d1 = p.grp[gend - 1];
            qend = d1.y + d1.z + (d1.w >> 12);
            const long long per = ((long long)(qend - d0.y) * 4 * nw) / (gend - gfirst);
            qahead = per < qend - d0.y ? (int)per + 1 : qend - d0.y;  // four rounds of groups
            if (threadIdx.x == 0) {
                prefetch_slices(d0.y, d0.y + qahead < qend ? d0.y + qahead : qend);
                prefetch_range(p.grp + gfirst, 16ll * (gend - gfirst));
                prefetch_range(p.jlev + ctx.p0, 4ll * in_part);
                if (!p.unit)
                    prefetch_range((const T*)p.dinv + ctx.p0, (long long)sizeof(T) * in_part);
                if (p.ldb == 1)
                    prefetch_range(b + p.part_row[part], (long long)sizeof(T) * in_part);
            }
        }
        for (int k = threadIdx.x; k < in_part; k += blockDim.x)
            xs[k] = Marker<T>::pending_value();
        if (!CL) {
            __syncthreads();
        } else {
            cluster_sync();
            if (ctx.g0 >= n) break;  // the same for the whole cluster
        }

        // ---- the warp's groups are gfirst + warp, + nw, ...; the next one: row,
        // entries, right-hand side (nd), and the descriptor after that (nd2)
        int gn = gfirst + warp;
        int4 nd = make_int4(0, 0, 0, 0), nd2 = nd;
        int n_i = -1, n_c[NI], n_xc[NX];
        T n_a[NI], n_xa[NX], n_b = T(0), n_d = T(1);
        double n_xbase = 0.0;
        auto next_group = [&]() {
            const int* cp = p.idx + ((long long)nd.y * 32 + lane);
            const T* ap = (const T*)p.vals + ((long long)nd.y * 32 + lane);
            const int X = nd.z, I = nd.w >> 12;
#pragma unroll
            for (int e = 0; e < NX; ++e) {
                n_xc[e] = -1;
                n_xa[e] = T(0);
                if (e < X) {
                    n_xc[e] = cp[32 * e];
                    n_xa[e] = ap[32 * e];
                }
            }
            cp += 32ll * X;
            ap += 32ll * X;
            // the first chunk: what full chunks leave, in the last slots
            const int skip = NI - (I <= NI ? I : (I - 1) % NI + 1);
#pragma unroll
            for (int e = 0; e < NI; ++e) {
                n_c[e] = zero;
                n_a[e] = T(0);
                if (e >= skip) {
                    n_c[e] = cp[32 * (e - skip)];
                    n_a[e] = ap[32 * (e - skip)];
                }
            }
            n_i = -1;
            if (grp < (nd.w & 63)) {
                n_i = p.jlev[nd.x + grp];
                if (sl == 0 && !p.unit) n_d = ((const T*)p.dinv)[nd.x + grp];
            }
        };
        auto next_rhs = [&]() {
            if (n_i >= 0 && sl == 0) {
                n_b = b[(long long)n_i * p.ldb];
                n_xbase = accumulate_base(p, n_i, 0);
            }
        };
        if (gn < gend) {
            nd = p.grp[gn];
            next_group();
            next_rhs();
            if (gn + nw < gend) nd2 = p.grp[gn + nw];
        }
        bool stuck = false;
        int g = gn;
        for (; g < gend; g = gn) {
            // ---- the next group becomes the current one
            const int X = nd.z, I = nd.w >> 12, span = (nd.w >> 6) & 63;
            const int base = nd.y;
            const int k = nd.x + grp, i = n_i;
            const bool out = i >= 0 && sl == 0 && i != p.withhold;
            // lanes that publish nothing store to the word that nobody reads
            const unsigned own =
                ctx.xs_a + (unsigned)(out ? k - ctx.p0 : zero + 1) * (unsigned)sizeof(T);
            const double xbase = n_xbase;
            int xc[NX];
            unsigned c[NI];
            T a[NI], v[NI], xa[NX], xv[NX];
#pragma unroll
            for (int e = 0; e < NX; ++e) {
                xc[e] = n_xc[e];
                xa[e] = n_xa[e];
                xv[e] = T(0);
            }
#pragma unroll
            for (int e = 0; e < NI; ++e) {
                c[e] = ctx.xs_a + (unsigned)n_c[e] * (unsigned)sizeof(T);
                a[e] = n_a[e];
            }
            unsigned rem = 0;  // slots in the cluster's shared memory
            auto place = [&]() {
                if (!CL) return;
                rem = 0;
#pragma unroll
                for (int e = 0; e < NX; ++e)
                    if (xc[e] >= ctx.g0) {
                        xc[e] = (int)remote_addr<T>(ctx, xc[e]);
                        rem |= 1u << e;
                    }
            };
            auto poll = [&](int e) -> T {
                return poll_ext<T, CL>(xp, xc[e], (rem & (1u << e)) != 0);
            };
            if (X > 0) {  // values of earlier parts: first polls
                place();
#pragma unroll
                for (int e = 0; e < NX; ++e)
                    if (xc[e] >= 0) xv[e] = poll(e);
            }
            T sum = T(0);
            if (i >= 0 && sl == 0) sum = p.unit ? n_b : n_b * n_d;
            gn = g + nw;
            nd = nd2;
            if (gn < gend) next_group();
            if (gn + nw < gend) nd2 = p.grp[gn + nw];
            bool ok = true;
            if (X <= NX && I <= NI) {
                // ---- the usual group: one chunk of each kind.  The part's own
                // values are looked at in the same rounds as the earlier parts',
                // so a row whose last value comes from an earlier part is folded
                // without another round.
                bool pend = true;
                if (X > 0) {
                    long long polls = 0;
                    while (true) {
                        bool px = false;
#pragma unroll
                        for (int e = 0; e < NX; ++e) px |= Marker<T>::pending(xv[e]);
#pragma unroll
                        for (int e = 0; e < NI; ++e) v[e] = lds(c[e], T(0));
                        if (!__any_sync(FULL, px)) break;
                        if (++polls > kHotPolls) {
                            if (polls > patience) {
                                ok = false;
                                break;
                            }
                            __nanosleep(32);
                        }
#pragma unroll
                        for (int e = 0; e < NX; ++e)
                            if (Marker<T>::pending(xv[e])) xv[e] = poll(e);
                    }
                    sum = fma(-xa[0], xv[0], sum);  // no entry: adds -0 * 0
                    if (X > 1) sum = fma(-xa[1], xv[1], sum);
                    pend = false;
#pragma unroll
                    for (int e = 0; e < NI; ++e) pend |= Marker<T>::pending(v[e]);
                    pend = __any_sync(FULL, pend);
                }
                if (I > 0) {
                    if (ok && pend) ok = wait_slots(c, v, patience);
                    if (ok) sum = fold_slots(sum, a, v, I);
                }
            } else {
                // ---- long rows: chunks of NX, then of NI slots
                long long polls = 0;
                for (int x0 = 0; x0 < X;) {
                    while (true) {
                        bool pend = false;
#pragma unroll
                        for (int e = 0; e < NX; ++e) pend |= Marker<T>::pending(xv[e]);
                        if (!__any_sync(FULL, pend)) break;
                        if (++polls > kHotPolls) {
                            if (polls > patience) {
                                ok = false;
                                break;
                            }
                            __nanosleep(32);
                        }
#pragma unroll
                        for (int e = 0; e < NX; ++e)
                            if (Marker<T>::pending(xv[e])) xv[e] = poll(e);
                    }
                    if (!ok) break;
                    sum = fma(-xa[0], xv[0], sum);
                    if (X - x0 > 1) sum = fma(-xa[1], xv[1], sum);
                    x0 += NX;
                    if (x0 >= X) break;
                    const long long at = 32ll * (base + x0) + lane;
#pragma unroll
                    for (int e = 0; e < NX; ++e) {
                        xc[e] = -1;
                        xa[e] = xv[e] = T(0);
                        if (x0 + e < X) {
                            xc[e] = p.idx[at + 32 * e];
                            xa[e] = ((const T*)p.vals)[at + 32 * e];
                        }
                    }
                    place();
#pragma unroll
                    for (int e = 0; e < NX; ++e)
                        if (xc[e] >= 0) xv[e] = poll(e);
                }
                if (ok && I > 0) {  // the next chunk is loaded before the wait for this one
                    int r = I <= NI ? I : (I - 1) % NI + 1;
                    long long at = 32ll * (base + X + r) + lane;
                    for (int left = I - r;; left -= NI) {
                        int c2[NI];
                        T a2[NI];
                        if (left > 0) {
#pragma unroll
                            for (int e = 0; e < NI; ++e) {
                                c2[e] = p.idx[at + 32 * e];
                                a2[e] = ((const T*)p.vals)[at + 32 * e];
                            }
                            at += 32 * NI;
                        }
                        ok = wait_slots(c, v, patience);
                        if (!ok) break;
                        sum = fold_slots(sum, a, v, r);
                        if (left == 0) break;
                        r = NI;
#pragma unroll
                        for (int e = 0; e < NI; ++e) {
                            c[e] = ctx.xs_a + (unsigned)c2[e] * (unsigned)sizeof(T);
                            a[e] = a2[e];
                        }
                    }
                }
            }
            if (ok) {
                const T xi = publishable(row_sum<W>(sum, span));
                st_cluster(own, xi);
                if (out) publish_global(p, k, i, xi, xbase);
            } else if (!slow_group<T, W, CL>(p, ctx, g, patience)) {
                stuck = true;
                break;
            }
            if (gn < gend) next_rhs();
            const int qp = base + qahead;
            if (lane == 0 && qp < qend) prefetch_slices(qp, qp + X + I < qend ? qp + X + I : qend);
        }
        if (stuck) {
            // A value has not come for long.  The rows of this warp's later groups
            // that do not need it must not wait for it: turns of a few polls for
            // every unfinished group, until all are done or the polls reach the
            // spin limit; then one after another, each to its end.
            constexpr int kTurn = 256;
            bool done = false;
            for (long long polls = 0; !done && polls < p.spin.limit;) {
                done = true;
                for (int q = g; q < gend; q += nw)
                    if (!slow_group<T, W, CL>(p, ctx, q, kTurn)) {
                        done = false;
                        polls += kTurn;
                    }
            }
            for (int q = g; !done && q < gend; q += nw) slow_group<T, W, CL>(p, ctx, q, kNoEnd);
        }
        if (!CL)
            __syncthreads();  // every group of the part is done before xs is reused
        else
            cluster_sync();  // ... and no other block of the cluster still reads it
    }
}

namespace {

// Lets the kernel take the device's opt-in shared memory (parts beyond 48 KB;
// once per device).
template <typename T, int W, bool CL>
cudaError_t part_attrs() {
    static unsigned long long done = 0;  // one bit per device
    int dev = 0, optin = 0;
    cudaError_t e = cudaGetDevice(&dev);
    if (e != cudaSuccess) return e;
    const unsigned long long bit = 1ull << (dev & 63);
    if (done & bit) return cudaSuccess;
    e = cudaDeviceGetAttribute(&optin, cudaDevAttrMaxSharedMemoryPerBlockOptin, dev);
    if (e == cudaSuccess)
        e = cudaFuncSetAttribute(part_solve_k1<T, W, CL>,
                                 cudaFuncAttributeMaxDynamicSharedMemorySize, optin - 64);
    if (e == cudaSuccess) done |= bit;
    return e;
}

cudaLaunchConfig_t part_config(int grid, int block, size_t smem, int cluster, cudaStream_t s,
                               cudaLaunchAttribute* attr) {
    cudaLaunchConfig_t cfg = {};
    cfg.gridDim = dim3((unsigned)grid, 1, 1);
    cfg.blockDim = dim3((unsigned)block, 1, 1);
    cfg.dynamicSmemBytes = smem;
    cfg.stream = s;
    attr[0].id = cudaLaunchAttributeClusterDimension;
    attr[0].val.clusterDim.x = (unsigned)cluster;
    attr[0].val.clusterDim.y = 1;
    attr[0].val.clusterDim.z = 1;
    cfg.attrs = attr;
    cfg.numAttrs = 1;
    return cfg;
}

// Launches, or (resident) counts the blocks of one launch that can be resident
// at once.
template <typename T, int W, bool CL>
cudaError_t part_c(const SolveParams& p, int grid, int block, int cluster, cudaStream_t s,
                   int num_sms, int* resident) {
    const size_t smem = sizeof(T) * ((size_t)p.max_part + 2);  // checked by the caller
    cudaError_t e = part_attrs<T, W, CL>();
    if (e != cudaSuccess) return e;
    cudaLaunchAttribute attr[1];
    if (resident) {
        int nb = 0;
        if (!CL) {
            e = cudaOccupancyMaxActiveBlocksPerMultiprocessor(&nb, part_solve_k1<T, W, CL>,
                                                              block, smem);
            nb *= num_sms;
        } else {
            cudaLaunchConfig_t cfg = part_config(cluster, block, smem, cluster, nullptr, attr);
            e = cudaOccupancyMaxActiveClusters(&nb, part_solve_k1<T, W, CL>, &cfg);
            nb *= cluster;
        }
        *resident = e == cudaSuccess ? nb : 0;
        return e;
    }
    if (!CL) {
        part_solve_k1<T, W, CL><<<grid, block, smem, s>>>(p, 1);
        return cudaGetLastError();
    }
    cudaLaunchConfig_t cfg = part_config(grid, block, smem, cluster, s, attr);
    return cudaLaunchKernelEx(&cfg, part_solve_k1<T, W, CL>, p, cluster);
}

template <typename T, int W>
cudaError_t part_w(const SolveParams& p, int grid, int block, int cluster, cudaStream_t s,
                   int num_sms, int* resident) {
    // Larger blocks run as kMaxBlock threads: the groups in flight want more than
    // the 64 registers that 1024 threads leave, and warps that wait take issue
    // slots from those that do not.
    if (block > kMaxBlock) block = kMaxBlock;
    return cluster > 1 ? part_c<T, W, true>(p, grid, block, cluster, s, num_sms, resident)
                       : part_c<T, W, false>(p, grid, block, 1, s, num_sms, resident);
}

}  // namespace

// One translation unit per type (solve_partitioned_f64.cu, _f32.cu): the
// instances take most of the build.
template <typename T>
cudaError_t part_any(int lanes, const SolveParams& p, int grid, int block, int cluster,
                     cudaStream_t s, int num_sms, int* resident) {
    if (cluster < 1 || cluster > kMaxCluster) return cudaErrorInvalidValue;
    switch (lanes) {
        case 1: return part_w<T, 1>(p, grid, block, cluster, s, num_sms, resident);
        case 2: return part_w<T, 2>(p, grid, block, cluster, s, num_sms, resident);
        case 4: return part_w<T, 4>(p, grid, block, cluster, s, num_sms, resident);
        case 8: return part_w<T, 8>(p, grid, block, cluster, s, num_sms, resident);
        case 16: return part_w<T, 16>(p, grid, block, cluster, s, num_sms, resident);
        case 32: return part_w<T, 32>(p, grid, block, cluster, s, num_sms, resident);
        default: return cudaErrorInvalidValue;
    }
}

}  // namespace sptrsv
