// Self-scheduled solve (Alg. 3, SLFR) for one right-hand side with every row at its own
// pace: a row is folded as its values come and published by itself, whatever the other
// rows of its warp wait for.  Tickets, waits and order of the sums are those of
// solve_self.cu, whose kernel takes the rows of a ticket as one where they are alike;
// results are bitwise the same.
//
// Where this one runs (the rule is in api.cu), with what both take, us, FP64 unless said
// otherwise, grids of 2 x 256 threads per SM:
//  * Rows that differ, few lanes per row.  Asking every ticket whether its rows are
//    alike, taking them and handing them to a function costs four warp reductions and a
//    second chain of loads, for an answer that is mostly no.  General matrix of 100001
//    rows: adjoint with 1 / 2 / 4 lanes 13160 / 10030 / 6160 asked and 10780 / 8460 /
//    5480 here; a chain of 20000 rows, level-ordered, FP32, 1 lane 14280 and 11690.
//  * One lane per row and rows of one chunk, in place: a lane publishes from inside its
//    wait, where the other kernel waits for 32 rows (5-point 1024 x 1024: 2480 and 2054).
//  * Very wide levels, where rows in flight are all that counts: 64 registers a thread
//    hold twice the warps (diagonal system of 10^6 rows, 8 lanes, uncapped grid: 280 and
//    184; at the default shape 87 and 80).
//
// What bounds it: the dependency hop, as there; on very wide levels the chain of loads
// a row starts with and the FP64 unit.
#include "rows_apart.cuh"

namespace sptrsv {

// A value has not come for long: ticket t and the one the warp also holds take turns,
// and the warp's remaining tickets follow here (a call from which the kernel returned
// would cost it registers all the time).
template <typename T, int W, bool MAP, bool PERM>
__device__ __noinline__ void rest_apart(const SolveParams& p, int t, int tn) {
    const long long patience = p.spin.limit / 4 + 1;
    bool stuck = true;
    while (true) {
        if (stuck) tn = stuck_rows<T, W, MAP, PERM, false>(p, t, tn, p.ticket, nullptr);
        t = __shfl_sync(0xffffffffu, tn, 0);
        if ((long long)t * (32 / W) >= p.n) return;
        if ((threadIdx.x & 31) == 0) tn = atomicAdd(p.ticket, 1);
        stuck = !rows_apart<T, W, MAP, PERM, false>(p, t, nullptr, false, patience);
    }
}

template <typename T, int W, bool MAP, bool PERM>
__global__ void __launch_bounds__(1024)
    apart_solve_k1(const __grid_constant__ SolveParams p) {
    constexpr int R = 32 / W;
    constexpr int E = kChunk;
    constexpr unsigned FULL = 0xffffffffu;
    const int lane = threadIdx.x & 31;
    const int grp = lane / W;
    const int sl = lane - grp * W;
    const unsigned gmask = group_mask<W>(lane);
    const T* __restrict__ vals = (const T*)p.vals;
    const T* b = (const T*)p.b;
    T* x = (T*)p.x;
    T* xpub = PERM ? (T*)p.xp : x;  // the array rows publish to and wait on
    const long long ldp = PERM ? 1 : p.ldx;
    const long long patience = p.spin.limit / 4 + 1;
    // fold order: an upper row from its last entry back (the copies store it so)
    const bool rvs = !PERM && p.diag_first;
    int t = 0;
    if (lane == 0) t = atomicAdd(p.ticket, 1);
    t = __shfl_sync(FULL, t, 0);
    while ((long long)t * R < p.n) {
        int tn = 0;
        if (lane == 0) tn = atomicAdd(p.ticket, 1);  // consumed after this one
        const long long k = (long long)t * R + grp;
        const bool has_row = k < p.n;
        int i = 0, beg = 0, end = 0;
        T dinv = T(1), sum = T(0);
        double xbase = 0.0;  // refinement: the solution the row's value is added to
        const int self_col = PERM ? (int)k : 0;
        if (has_row) {
            i = p.jlev[k];
            beg = p.ptr[PERM ? k : i];
            end = p.ptr[(PERM ? k : i) + 1];
            if (sl == 0) {  // whatever does not depend on x, while the values are on their way
                if (!p.unit) {
                    const int q = p.diag_first ? beg : end - 1;
                    const T d = vals[MAP ? p.vmap[q] : q];
                    dinv = p.prescaled ? d : T(1) / d;  // a pre-scaled copy holds 1/d(i)
                }
                sum = b[(long long)i * p.ldb];
                if (!p.unit) sum *= dinv;
                xbase = accumulate_base(p, i, 0);
            }
        }
        if (W > 1 && !p.unit && !p.prescaled) dinv = __shfl_sync(FULL, dinv, grp * W);
        const int span = warp_span<W>(has_row, end - beg);
        int q0 = beg + sl, c[E];
        T a[E], v[E];
        unsigned live = 0, pend = 0;  // entries that count / still unpublished
        auto load_chunk = [&]() {
            live = pend = 0;
#pragma unroll
            for (int e = 0; e < E; ++e) {
                const int q = q0 + e * W;
                c[e] = -1;
                a[e] = T(0);
                v[e] = T(0);
                if (q < end) {
                    const int pq = rvs ? beg + end - 1 - q : q;  // fold order -> storage
                    const int cc = p.idx[pq];
                    if (cc != (PERM ? self_col : i)) {
                        c[e] = cc;
                        a[e] = vals[MAP ? p.vmap[pq] : pq];
                        live |= 1u << e;
                    }
                }
            }
#pragma unroll
            for (int e = 0; e < E; ++e)
                if (live & (1u << e)) v[e] = ld_relaxed(xpub + (long long)c[e] * ldp);
            if (!p.unit && !p.prescaled) {
#pragma unroll
                for (int e = 0; e < E; ++e)
                    if (live & (1u << e)) a[e] *= dinv;
            }
#pragma unroll
            for (int e = 0; e < E; ++e)
                if ((live & (1u << e)) && Marker<T>::pending(v[e])) pend |= 1u << e;
        };
        auto publish_row = [&](T tot) {
            const T val = publishable(tot);
            st_relaxed(xpub + (PERM ? k : (long long)i * p.ldx), val);
            if (p.xacc)
                accumulate_with(p, i, 0, val, xbase);
            else if (PERM)
                x[(long long)i * p.ldx] = val;
        };
        bool lane_done = q0 >= end;
        if (!lane_done) load_chunk();
        bool published = !has_row;
        long long waits = 0;
        unsigned ns = 32;
        while (true) {
            if (!lane_done && pend == 0) {  // fold a complete chunk in fold order
                sum = fold_chunk(sum, a, v, live);
                q0 += W * E;
                if (q0 >= end) {
                    lane_done = true;
                    // one lane per row: no lane reduction to wait for
                    if (W == 1 && has_row && i != p.withhold) {
                        publish_row(sum);
                        published = true;
                    }
                } else {
                    load_chunk();
                }
            }
            const unsigned done = __ballot_sync(FULL, lane_done);
            const bool fresh = !published && (done & gmask) == gmask;
            if (__any_sync(FULL, fresh)) {  // FP64 is scarce on GB300: reduce only then
                const T tot = group_sum_span<W>(sum, FULL, span);
                if (fresh && sl == 0 && i != p.withhold) publish_row(tot);
            }
            published = published || fresh;
            if (__all_sync(FULL, published)) break;
            // A lane with a complete chunk folds it first; the warp enters the tight
            // wait when every lane is done or waiting, so a row that another row of
            // this ticket waits on is never held back.
            if (__any_sync(FULL, !lane_done && pend == 0)) continue;
            if (!__any_sync(FULL, pend != 0)) {
                waits = 0;
                ns = 32;
                continue;
            }
            // re-poll until something arrives anywhere in the warp
            const unsigned before = pend;
            do {
#pragma unroll
                for (int e = 0; e < E; ++e)
                    if (pend & (1u << e)) v[e] = ld_relaxed(xpub + (long long)c[e] * ldp);
#pragma unroll
                for (int e = 0; e < E; ++e)
                    if ((pend & (1u << e)) && !Marker<T>::pending(v[e])) pend &= ~(1u << e);
                // one lane per row and this was the row's last chunk: fold and publish
                // before the warp leaves the wait
                if (W == 1 && !lane_done && pend == 0 && q0 + E >= end) {
                    sum = fold_chunk(sum, a, v, live);
                    q0 += E;
                    lane_done = true;
                    if (has_row && i != p.withhold) publish_row(sum);
                    published = true;
                }
                if (++waits > patience) {
                    rest_apart<T, W, MAP, PERM>(p, t, tn);
                    return;
                }
                if (W == 1) {
                    // leave it when every lane is done or one needs its next chunk
                    const unsigned w =
                        __reduce_or_sync(FULL, lane_done ? 0u : (pend != 0 ? 1u : 2u));
                    if ((w & 2u) || !(w & 1u)) break;
                } else if (__any_sync(FULL, pend != before)) {
                    break;  // something arrived
                }
                if (waits >= p.spin.hot) {
                    __nanosleep(ns);
                    ns = ns < p.spin.max_ns ? ns * 2 : p.spin.max_ns;
                }
            } while (true);
        }
        t = __shfl_sync(FULL, tn, 0);
    }
}

namespace {

template <int W>
struct Lanes {
    static constexpr int value = W;
};

// Calls f(kernel) with the instance a launch with these choices uses.
template <typename F>
cudaError_t apart_any(bool f64, int lanes, bool map, bool perm, F f) {
    auto w = [&](auto t, auto l) {
        using T = decltype(t);
        constexpr int W = decltype(l)::value;
        return perm ? f(apart_solve_k1<T, W, false, true>)
                    : map ? f(apart_solve_k1<T, W, true, false>)
                          : f(apart_solve_k1<T, W, false, false>);
    };
    auto any = [&](auto t) {
        switch (lanes) {
            case 1: return w(t, Lanes<1>());
            case 2: return w(t, Lanes<2>());
            case 4: return w(t, Lanes<4>());
            case 8: return w(t, Lanes<8>());
            case 16: return w(t, Lanes<16>());
            case 32: return w(t, Lanes<32>());
            default: return cudaErrorInvalidValue;
        }
    };
    return f64 ? any(double()) : any(float());
}

}  // namespace

cudaError_t launch_apart_k1(bool f64, int lanes, const SolveParams& p, int grid, int block,
                            cudaStream_t s) {
    return apart_any(f64, lanes, !p.xp && p.vmap, p.xp != nullptr, [&](auto k) {
        k<<<grid, block, 0, s>>>(p);
        return cudaGetLastError();
    });
}

int apart_blocks_per_sm(bool f64, int lanes, bool map, bool perm, int block) {
    int nb = 0;
    const cudaError_t e = apart_any(f64, lanes, map, perm, [&](auto k) {
        return cudaOccupancyMaxActiveBlocksPerMultiprocessor(&nb, k, block, 0);
    });
    return e == cudaSuccess && nb > 0 ? nb : 1;
}

}  // namespace sptrsv
