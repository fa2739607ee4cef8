// The rows of a ticket one by one, for the single-RHS kernels of the in-place and
// level-ordered forms (solve_self.cu, solve_apart.cu): where rows differ, and where a
// value does not come.
#pragma once
#include "self_rows.cuh"

namespace sptrsv {

// The rows of ticket t one by one: every row is folded as its values come and
// published by itself.  Gives up (false) after `budget` polls without an end;
// again: rows that are published already are skipped.
template <typename T, int W, bool MAP, bool PERM, bool SMALL>
__device__ __noinline__ bool rows_apart(const SolveParams& p, long long t, T* xs, bool again,
                                        long long budget) {
    constexpr int R = 32 / W;
    constexpr int E = kChunk;
    constexpr unsigned FULL = 0xffffffffu;
    const int lane = threadIdx.x & 31;
    const int grp = lane / W;
    const int sl = lane - grp * W;
    const unsigned gmask = group_mask<W>(lane);
    T* xpub = SMALL ? xs : PERM ? (T*)p.xp : (T*)p.x;
    const long long ldp = (SMALL || PERM) ? 1 : p.ldx;
    Row<T> r = take_row<T, W, PERM>(p, t * R + grp);
    start_row<T, W, MAP>(p, r, sl);
    const int span = warp_span<W>(r.has, r.end - r.beg);
    const long long own = (PERM ? r.k : (long long)r.i) * ldp;
    auto look = [&](long long at) -> T {
        return SMALL ? lds_relaxed(xpub + at) : ld_relaxed(xpub + at);
    };
    bool published = !r.has || (again && !Marker<T>::pending(look(own)));
    int q0 = r.beg + sl, c[E];
    T a[E], v[E];
    unsigned live = 0, pend = 0;
    auto load_chunk = [&]() {
        load_entries<T, W, MAP, PERM, E>(p, r, q0, c, a);
        live = pend = 0;
#pragma unroll
        for (int e = 0; e < E; ++e) {
            v[e] = T(0);
            if (c[e] >= 0) {
                live |= 1u << e;
                v[e] = look((long long)c[e] * ldp);
            }
        }
        if (!p.unit && !p.prescaled) {
#pragma unroll
            for (int e = 0; e < E; ++e)
                if (live & (1u << e)) a[e] *= r.dinv;
        }
#pragma unroll
        for (int e = 0; e < E; ++e)
            if ((live & (1u << e)) && Marker<T>::pending(v[e])) pend |= 1u << e;
    };
    bool lane_done = published || q0 >= r.end;
    if (!lane_done) load_chunk();
    long long waits = 0, total = 0;
    unsigned ns = 32;
    while (true) {
        if (!lane_done && pend == 0) {  // fold a complete chunk in fold order
            if (live) r.sum = fold_chunk(r.sum, a, v, live);
            q0 += W * E;
            if (q0 >= r.end)
                lane_done = true;
            else
                load_chunk();
        }
        const unsigned done = __ballot_sync(FULL, lane_done);
        const bool fresh = !published && (done & gmask) == gmask;
        if (__any_sync(FULL, fresh)) {
            const T tot = group_sum_span<W>(r.sum, FULL, span);
            if (fresh && sl == 0 && r.i != p.withhold) {
                const T val = publishable(tot);
                if (SMALL)
                    *(volatile T*)(xpub + own) = val;
                else
                    st_relaxed(xpub + own, val);
                if (p.xacc)
                    accumulate_with(p, r.i, 0, val, r.xbase);
                else if (PERM || SMALL)
                    ((T*)p.x)[(long long)r.i * p.ldx] = val;
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
                if (pend & (1u << e)) v[e] = look((long long)c[e] * ldp);
#pragma unroll
            for (int e = 0; e < E; ++e)
                if ((pend & (1u << e)) && !Marker<T>::pending(v[e])) pend &= ~(1u << e);
            if (++total > budget) return false;
            if (++waits >= p.spin.limit) {
                if (pend) {
                    report(p.status, r.i, kCodeTimeout);
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

// A value that ticket t's rows wait for has not come for long.  The rows of the
// ticket this warp also holds must not wait for it where they do not need it:
// turns of a few polls for both, until both are done or the polls reach the spin
// limit, then one after the other to its end.  Returns (in lane 0) the warp's
// next ticket.
template <typename T, int W, bool MAP, bool PERM, bool SMALL>
__device__ __noinline__ int stuck_rows(const SolveParams& p, long long t, int tn, int* ticket,
                                       T* xs) {
    constexpr int kTurn = 256;
    constexpr long long kNoEnd = 1ll << 62;  // the wait ends by the spin limit
    const long long t2 = __shfl_sync(0xffffffffu, tn, 0);
    const bool held = !SMALL && t2 * (32 / W) < p.n;
    bool done = false, done2 = !held;
    for (long long polls = 0; !(done && done2) && polls < p.spin.limit; polls += kTurn) {
        if (!done) done = rows_apart<T, W, MAP, PERM, SMALL>(p, t, xs, true, kTurn);
        if (!done2) done2 = rows_apart<T, W, MAP, PERM, SMALL>(p, t2, xs, true, kTurn);
    }
    if (!done) rows_apart<T, W, MAP, PERM, SMALL>(p, t, xs, true, kNoEnd);
    if (!done2) rows_apart<T, W, MAP, PERM, SMALL>(p, t2, xs, true, kNoEnd);
    if (held && (threadIdx.x & 31) == 0) tn = atomicAdd(ticket, 1);
    return tn;
}

}  // namespace sptrsv
