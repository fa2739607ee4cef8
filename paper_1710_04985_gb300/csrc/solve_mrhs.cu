// Multi-right-hand-side solves, self-scheduled (Alg. 3) or level-scheduled
// (Alg. 1).  A sub-warp of W lanes owns one row; lane l handles the
// right-hand-side columns l, l + W, ...  Each stored entry is read once per
// column tile and applied to all of them, so the matrix traffic is shared by
// the k solves (the multiple-right-hand-side case of Sec. 1).  No reduction
// is needed: each lane accumulates its own column in fold order (farthest
// dependency first: an upper row from its last entry back) and
// publishes it by itself, so in the self-scheduled form every (row, column)
// value is its own ready flag.
//
// What bounds the self-scheduled form: on narrow levels the dependency hop, as
// for one right-hand side; on wide ones the rows in flight (a warp holds 32/W
// rows for one or two passes over their columns, and a row starts with a chain of
// dependent loads: ticket, row, row pointers, entries, values), then the FP64
// unit.  So a warp runs through its tickets as a pipeline: while it waits for
// the values of one, the row and the row pointers of the next are on their way,
// and a row's next chunk of entries is loaded before the wait for the current
// one (rows of one chunk keep it in registers for all their columns).  As with
// one right-hand side (solve_self.cu), rows that are alike are waited for and
// folded as one, and the rows of other matrices go their own pace.
#include "internal.h"

namespace sptrsv {

// Level-scheduled row: all dependencies are final (earlier launches).
template <typename T, int W, bool MAP>
__device__ __forceinline__ void mrhs_row_level(const SolveParams& p, int i, int sl) {
    const T* __restrict__ vals = (const T*)p.vals;
    const T* b = (const T*)p.b;
    T* x = (T*)p.x;
    const int beg = p.ptr[i], end = p.ptr[i + 1];
    T di = T(1);
    if (!p.unit) {
        const int q = p.diag_first ? beg : end - 1;
        di = vals[MAP ? p.vmap[q] : q];
    }
    for (int c0 = 0; c0 < p.nrhs; c0 += W) {
        const int c = c0 + sl;
        if (c >= p.nrhs) break;
        T acc = T(0);
        for (int q = beg; q < end; ++q) {
            const int j = p.idx[q];
            if (j == i) continue;
            acc += vals[MAP ? p.vmap[q] : q] * x[(long long)j * p.ldx + c];
        }
        T xi = b[(long long)i * p.ldb + c] - acc;
        if (!p.unit) xi = xi / di;
        x[(long long)i * p.ldx + c] = xi;
    }
}

namespace {

constexpr int kMaxMrhsBlock = 256;  // larger blocks run as several of this size
constexpr int kMrhsHot = 64;        // polls of one wait before the warp backs off

// A row's entries in fold order (farthest dependency first: an upper row from
// its last entry back; the level-ordered copy already stores it that way round),
// the diagonal, which comes last, left out.
struct Entries {
    int beg, end;  // stored entries
    int m;         // entries that count
    int back;      // fold order runs from the last stored entry back
    __device__ __forceinline__ int at(int t) const { return back ? end - 1 - t : beg + t; }
};
template <bool PERM>
__device__ __forceinline__ Entries entries_of(const SolveParams& p, int self, int beg, int end) {
    Entries r = {beg, end, end - beg, !PERM && p.diag_first};
    if (r.m > 0 && (!p.unit || p.idx[r.at(r.m - 1)] == self)) --r.m;
    return r;
}

// Entries t0 .. t0 + E - 1: the unknown to wait for (-1: none) and the stored
// value (0).
template <typename T, bool MAP, int E>
__device__ __forceinline__ void load_entries(const SolveParams& p, const Entries& r, int t0,
                                             int (&c)[E], T (&a)[E]) {
    const T* __restrict__ vals = (const T*)p.vals;
#pragma unroll
    for (int e = 0; e < E; ++e) {
        c[e] = -1;
        a[e] = T(0);
        if (t0 + e < r.m) {
            const int q = r.at(t0 + e);
            c[e] = p.idx[q];
            a[e] = vals[MAP ? p.vmap[q] : q];
        }
    }
}

template <typename T, int E>
__device__ __forceinline__ void scale_entries(const SolveParams& p, T dinv, const int (&c)[E],
                                              T (&a)[E]) {
    if (p.unit || p.prescaled) return;
#pragma unroll
    for (int e = 0; e < E; ++e)
        if (__any_sync(0xffffffffu, c[e] >= 0)) {
            if (c[e] >= 0) a[e] *= dinv;
        }
}

// 1/d(i) of a row (a pre-scaled copy holds it); 1 for a unit diagonal.
template <typename T, bool MAP>
__device__ __forceinline__ T row_dinv(const SolveParams& p, int beg, int end) {
    if (p.unit || end <= beg) return T(1);
    const int q = p.diag_first ? beg : end - 1;
    const T d = ((const T*)p.vals)[MAP ? p.vmap[q] : q];
    return p.prescaled ? d : T(1) / d;
}

template <typename T, bool PERM>
__device__ __forceinline__ void publish_column(const SolveParams& p, T* at, int i, int col,
                                               T acc) {
    const T val = publishable(acc);
    st_relaxed(at, val);
    if (p.xacc)
        accumulate_published(p, i, col, val);
    else if (PERM)
        ((T*)p.x)[(long long)i * p.ldx + col] = val;
}

}  // namespace

// The rows of ticket t, every lane at its own pace: a column is folded as its
// values come and published by itself.  Gives up (false) after `budget` polls
// without an end; again: columns that are published already are skipped.
// ONE: one count of polls for both ends, the budget and the spin limit.
template <typename T, int W, bool MAP, bool PERM, bool ONE>
__device__ __forceinline__ bool mrhs_apart(const SolveParams& p, long long t, bool again,
                                        long long budget) {
    constexpr unsigned FULL = 0xffffffffu;
    constexpr int E = kChunk;
    constexpr int R = 32 / W;
    const int lane = threadIdx.x & 31;
    const int sl = lane % W;
    const T* b = (const T*)p.b;
    T* xpub = PERM ? (T*)p.xp : (T*)p.x;
    const long long ldp = PERM ? p.nrhs : p.ldx;
    const long long k = t * R + lane / W;
    int i = 0, beg = 0, end = 0;
    if (k < p.n) {
        i = p.jlev[k];
        beg = p.ptr[PERM ? k : i];
        end = p.ptr[(PERM ? k : i) + 1];
    }
    const T dinv = k < p.n ? row_dinv<T, MAP>(p, beg, end) : T(1);
    const Entries row = entries_of<PERM>(p, PERM ? (int)k : i, beg, end);
    const long long prow = (PERM ? k : (long long)i) * ldp;
    int col = sl, t0 = 0, c[E], c2[E];
    T a[E], a2[E], v[E], acc = T(0);
    unsigned live = 0, pend = 0;
    bool lane_done = k >= p.n;
    // next column that is not published yet; its first chunk is issued
    auto start_column = [&]() {
        while (again && col < p.nrhs && !Marker<T>::pending(ld_relaxed(xpub + prow + col)))
            col += W;
        if (col >= p.nrhs) {
            lane_done = true;
            return;
        }
        acc = b[(long long)i * p.ldb + col];
        if (!p.unit) acc *= dinv;
        t0 = 0;
        load_entries<T, MAP, E>(p, row, 0, c2, a2);
    };
    // the issued chunk becomes the current one; the one after it is issued
    auto adopt_chunk = [&]() {
        live = pend = 0;
#pragma unroll
        for (int e = 0; e < E; ++e) {
            c[e] = c2[e];
            a[e] = a2[e];
            v[e] = T(0);
            if (c[e] >= 0) {
                live |= 1u << e;
                v[e] = ld_relaxed(xpub + (long long)c[e] * ldp + col);
            }
        }
        if (t0 + E < row.m) load_entries<T, MAP, E>(p, row, t0 + E, c2, a2);
        if (!p.unit && !p.prescaled) {
#pragma unroll
            for (int e = 0; e < E; ++e)
                if (live & (1u << e)) a[e] *= dinv;
        }
#pragma unroll
        for (int e = 0; e < E; ++e)
            if ((live & (1u << e)) && Marker<T>::pending(v[e])) pend |= 1u << e;
    };
    if (!lane_done) start_column();
    if (!lane_done) adopt_chunk();
    const long long stop = budget < p.spin.limit ? budget + 1 : p.spin.limit;
    long long waits = 0, total = 0;
    unsigned ns = 32;
    while (true) {
        if (!lane_done && pend == 0) {
            if (live) acc = fold_chunk(acc, a, v, live);
            t0 += E;
            if (t0 >= row.m) {  // column done: publish it, move to the next one
                if (i != p.withhold) publish_column<T, PERM>(p, xpub + prow + col, i, col, acc);
                col += W;
                start_column();
            }
            if (!lane_done) adopt_chunk();
        }
        if (__all_sync(FULL, lane_done)) return true;
        if (__any_sync(FULL, !lane_done && pend == 0)) continue;  // fold first
        const unsigned before = pend;
        do {
#pragma unroll
            for (int e = 0; e < E; ++e)
                if (pend & (1u << e)) v[e] = ld_relaxed(xpub + (long long)c[e] * ldp + col);
#pragma unroll
            for (int e = 0; e < E; ++e)
                if ((pend & (1u << e)) && !Marker<T>::pending(v[e])) pend &= ~(1u << e);
            if (!ONE && ++total > budget) return false;
            if (++waits >= (ONE ? stop : p.spin.limit)) {
                if (ONE && waits > budget) return false;
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

// The warp's tickets in hand (bits of `left`: h0, h1, h2), then all that remain, by
// mrhs_apart.  If a value does not come for long (again: it has not come for the
// tickets in hand already), the rows of the other tickets the warp holds must not
// wait for it where they do not need it: turns of a few polls for all of them,
// until they are done or the polls reach the spin limit, then one after the other
// to its end.  No ticket is taken ahead meanwhile: its rows would wait for that end,
// and with them the rows of other warps that need them and not the missing value.
template <typename T, int W, bool MAP, bool PERM, bool ONE>
__device__ __forceinline__ void apart_rest(const SolveParams& p, int h0, int h1, int h2,
                                           unsigned left, bool again) {
    constexpr unsigned FULL = 0xffffffffu;
    constexpr int R = 32 / W;
    constexpr int kTurn = 256;
    constexpr long long kNoEnd = 1ll << 62;  // the wait ends by the spin limit
    auto ticket = [&]() {
        int t = 0;
        if ((threadIdx.x & 31) == 0) t = atomicAdd(p.ticket, 1);
        return t;  // in lane 0
    };
    long long polls = 0;
    int slot = 0, tn = -1;  // no ticket taken ahead
    while (true) {
        if (left == 0) {
            h0 = __shfl_sync(FULL, tn, 0);
            tn = ticket();  // consumed after this one
            if (h0 < 0) continue;
            if ((long long)h0 * R >= p.n) return;
            left = 1;
            slot = 0;
            again = false;
        }
        while (!(left >> slot & 1u)) slot = slot == 2 ? 0 : slot + 1;
        const int t = slot == 0 ? h0 : slot == 1 ? h1 : h2;
        const long long budget = !again                  ? p.spin.limit / 4 + 1
                                 : polls < p.spin.limit ? kTurn : kNoEnd;
        if (mrhs_apart<T, W, MAP, PERM, ONE>(p, t, again, budget)) {
            left &= ~(1u << slot);
        } else if (!again) {  // stuck: the ticket ahead takes turns with this one
            again = true;
            polls = 0;
            h1 = __shfl_sync(FULL, tn, 0);
            tn = -1;
            if ((long long)h1 * R < p.n) left |= 2u;
        } else {
            polls += kTurn;
        }
        slot = slot == 2 ? 0 : slot + 1;
    }
}

// Level-scheduled form: one launch per level.
template <typename T, int W, bool MAP>
__global__ void __launch_bounds__(1024) level_mrhs_k(const __grid_constant__ SolveParams p) {
    const long long g = ((long long)blockIdx.x * blockDim.x + threadIdx.x) / W;
    if (g < p.cnt) mrhs_row_level<T, W, MAP>(p, p.jlev[p.kbeg + g], (threadIdx.x & 31) % W);
}

// PERM: the pattern is the plan's level-ordered copy (position k = row
// jlev[k], columns renumbered to positions, values pre-scaled for a non-unit
// matrix); columns publish to the position-ordered buffer p.xp ([n][nrhs])
// that waiting lanes poll, so a level's unknowns are one contiguous run, and
// are stored to x (or added to p.xacc) for the caller.
//
// Rows that are not alike: every ticket by mrhs_apart.
template <typename T, int W, bool MAP, bool PERM>
__global__ void __launch_bounds__(kMaxMrhsBlock)
    apart_mrhs_k(const __grid_constant__ SolveParams p) {
    apart_rest<T, W, MAP, PERM, true>(p, 0, 0, 0, 0, false);
}

// Rows that are alike.  MULTI: rows of more than one chunk of entries.
template <typename T, int W, bool MAP, bool PERM, bool MULTI>
__global__ void __launch_bounds__(kMaxMrhsBlock, 3)
    solve_mrhs_k(const __grid_constant__ SolveParams p) {
    constexpr unsigned FULL = 0xffffffffu;
    constexpr int E = kChunk;
    constexpr int R = 32 / W;
    const int lane = threadIdx.x & 31;
    const int grp = lane / W;
    const int sl = lane - grp * W;
    const T* b = (const T*)p.b;
    T* xpub = PERM ? (T*)p.xp : (T*)p.x;  // the array columns publish to and wait on
    const long long ldp = PERM ? p.nrhs : p.ldx;
    auto ticket = [&]() {
        int t = 0;
        if (lane == 0) t = atomicAdd(p.ticket, 1);
        return t;  // in lane 0
    };
    // ---- the pipeline: t is solved, the rows of t1 are being loaded, the ticket
    // after it is on its way
    int n_i = 0, n_beg = 0, n_end = 0, n_lev = 0;  // row of ticket t1
    bool n_has = false;
    auto load_row = [&](int t1) {
        const long long k = (long long)t1 * R + grp;
        n_has = k < p.n;
        if (n_has) n_i = p.jlev[k];
    };
    auto load_ptrs = [&](int t1) {
        n_beg = n_end = 0;
        if (n_has) {
            const long long r = PERM ? (long long)t1 * R + grp : (long long)n_i;
            n_beg = p.ptr[r];
            n_end = p.ptr[r + 1];
            if (R > 1) n_lev = p.lev[n_i];
        }
    };
    int t = __shfl_sync(FULL, ticket(), 0);
    load_row(t);
    load_ptrs(t);
    int t1 = __shfl_sync(FULL, ticket(), 0);
    while ((long long)t * R < p.n) {
        const int i = n_i, lev = n_lev;
        const long long k = (long long)t * R + grp;
        const Entries row = entries_of<PERM>(p, PERM ? (int)k : i, n_beg, n_end);
        const long long prow = (PERM ? k : (long long)i) * ldp;
        const int nch = MULTI ? max(1, __reduce_max_sync(FULL, (row.m + E - 1) / E)) : 1;
        bool todo = n_has, ok = true, staged = false;
        int c[E], c2[E];
        T a[E], a2[E], v[E];
        load_entries<T, MAP, E>(p, row, 0, c, a);
        const T dinv = todo ? row_dinv<T, MAP>(p, row.beg, row.end) : T(1);
        const int tn = ticket();
        scale_entries(p, dinv, c, a);
        while (true) {  // level by level, if the ticket straddles levels
            bool mine = todo;
            if (R > 1) {
                const int low = __reduce_min_sync(FULL, todo ? lev : 0x7fffffff);
                mine = todo && lev == low;
            }
            int col = sl;
            for (int c0 = 0; c0 < p.nrhs; c0 += W, col += W) {
                const bool act = mine && col < p.nrhs;
                T acc = T(0);
                if (act) acc = b[(long long)i * p.ldb + col];
                for (int ch = 0; ch < nch; ++ch) {
#pragma unroll
                    for (int e = 0; e < E; ++e) {
                        v[e] = T(0);
                        if (act && c[e] >= 0) v[e] = ld_relaxed(xpub + (long long)c[e] * ldp + col);
                    }
                    // the chunk after this one (after the last: the first)
                    if (MULTI && nch > 1)
                        load_entries<T, MAP, E>(p, row, ch + 1 < nch ? (ch + 1) * E : 0, c2, a2);
                    if (!staged) load_row(t1);
                    if (ch == 0 && !p.unit && act) acc *= dinv;
                    unsigned slots = 0;
#pragma unroll
                    for (int e = 0; e < E; ++e)
                        if (__any_sync(FULL, c[e] >= 0)) slots |= 1u << e;
                    long long polls = 0;
                    while (true) {
                        bool pend = false;
#pragma unroll
                        for (int e = 0; e < E; ++e) pend |= Marker<T>::pending(v[e]);
                        if (!__any_sync(FULL, pend)) break;
                        if (++polls > kMrhsHot) {
                            if (polls > p.spin.limit / 4) {
                                ok = false;
                                break;
                            }
                            __nanosleep(32);
                        }
#pragma unroll
                        for (int e = 0; e < E; ++e)
                            if (Marker<T>::pending(v[e]))
                                v[e] = ld_relaxed(xpub + (long long)c[e] * ldp + col);
                    }
                    if (!ok) break;
#pragma unroll
                    for (int e = 0; e < E; ++e)
                        if (slots & (1u << e)) acc = fma(-a[e], v[e], acc);  // no entry: -0 * 0
                    if (!staged) {
                        load_ptrs(t1);
                        staged = true;
                    }
                    if (MULTI && nch > 1) {
#pragma unroll
                        for (int e = 0; e < E; ++e) {
                            c[e] = c2[e];
                            a[e] = a2[e];
                        }
                        scale_entries(p, dinv, c, a);
                    }
                }
                if (!ok) break;
                if (act && i != p.withhold)
                    publish_column<T, PERM>(p, xpub + prow + col, i, col, acc);
            }
            todo = todo && !mine;
            if (!ok || !__any_sync(FULL, todo)) break;
        }
        const int t2 = __shfl_sync(FULL, tn, 0);
        if (!ok) {
            apart_rest<T, W, MAP, PERM, false>(p, t, t1, t2,
                                        1u | ((long long)t1 * R < p.n ? 2u : 0u) |
                                            ((long long)t2 * R < p.n ? 4u : 0u), true);
            return;
        }
        t = t1;
        t1 = t2;
    }
}

namespace {

template <typename T, int W, bool MAP, bool PERM, typename F>
cudaError_t mrhs_r(MrhsRows rows, F f) {
    return rows == kMrhsApart ? f(apart_mrhs_k<T, W, MAP, PERM>)
           : rows == kMrhsAlike ? f(solve_mrhs_k<T, W, MAP, PERM, true>)
                                : f(solve_mrhs_k<T, W, MAP, PERM, false>);
}

template <typename T, int W, typename F>
cudaError_t mrhs_w(bool map, bool perm, MrhsRows rows, F f) {
    return perm ? mrhs_r<T, W, false, true>(rows, f)
                : map ? mrhs_r<T, W, true, false>(rows, f) : mrhs_r<T, W, false, false>(rows, f);
}

// Calls f(kernel) with the instance a launch with these choices uses.
template <typename T, typename F>
cudaError_t mrhs_t(int lanes, bool map, bool perm, MrhsRows rows, F f) {
    switch (lanes) {
        case 4: return mrhs_w<T, 4>(map, perm, rows, f);
        case 8: return mrhs_w<T, 8>(map, perm, rows, f);
        case 16: return mrhs_w<T, 16>(map, perm, rows, f);
        case 32: return mrhs_w<T, 32>(map, perm, rows, f);
        default: return cudaErrorInvalidValue;
    }
}

template <typename F>
cudaError_t mrhs_any(bool f64, int lanes, bool map, bool perm, MrhsRows rows, F f) {
    return f64 ? mrhs_t<double>(lanes, map, perm, rows, f)
               : mrhs_t<float>(lanes, map, perm, rows, f);
}

template <typename T, int W>
cudaError_t level_w(const SolveParams& p, int block, cudaStream_t s) {
    const int grid = (int)(((long long)p.cnt * W + block - 1) / block);
    if (p.vmap)
        level_mrhs_k<T, W, true><<<grid, block, 0, s>>>(p);
    else
        level_mrhs_k<T, W, false><<<grid, block, 0, s>>>(p);
    return cudaGetLastError();
}

template <typename T>
cudaError_t level_t(int lanes, const SolveParams& p, int block, cudaStream_t s) {
    switch (lanes) {
        case 4: return level_w<T, 4>(p, block, s);
        case 8: return level_w<T, 8>(p, block, s);
        case 16: return level_w<T, 16>(p, block, s);
        case 32: return level_w<T, 32>(p, block, s);
        default: return cudaErrorInvalidValue;
    }
}

}  // namespace

cudaError_t launch_mrhs(bool f64, int lanes, bool self, MrhsRows rows, const SolveParams& p,
                        int grid, int block, cudaStream_t s) {
    if (!self) return f64 ? level_t<double>(lanes, p, block, s) : level_t<float>(lanes, p, block, s);
    if (block > kMaxMrhsBlock) {  // the same warps in blocks of kMaxMrhsBlock threads
        grid = (int)(((long long)grid * block + kMaxMrhsBlock - 1) / kMaxMrhsBlock);
        block = kMaxMrhsBlock;
    }
    // a level-ordered copy holds its values gathered: no map
    return mrhs_any(f64, lanes, !p.xp && p.vmap, p.xp != nullptr, rows, [&](auto k) {
        k<<<grid, block, 0, s>>>(p);
        return cudaGetLastError();
    });
}

int mrhs_blocks_per_sm(bool f64, int lanes, bool map, bool perm, MrhsRows rows, int block) {
    int nb = 0;
    const int run = block > kMaxMrhsBlock ? kMaxMrhsBlock : block;
    const cudaError_t e = mrhs_any(f64, lanes, map, perm, rows, [&](auto k) {
        return cudaOccupancyMaxActiveBlocksPerMultiprocessor(&nb, k, run, 0);
    });
    if (e != cudaSuccess || nb < 1) return 1;
    nb = (int)((long long)nb * run / block);  // in blocks of the size asked for
    return nb > 0 ? nb : 1;
}

}  // namespace sptrsv
