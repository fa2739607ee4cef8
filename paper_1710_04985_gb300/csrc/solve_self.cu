// Self-scheduled solve (Alg. 3, SLFR) for one right-hand side.
//
// Differences from the paper's SLFR kernel (Sec. 4.3), for sm_103a:
//  * Rows are handed out in level order (jlev), as in the paper, but by a
//    ticket counter rather than by warp index: a warp takes ticket t only
//    while running, and every row it waits on belongs to a smaller ticket,
//    already held by a running warp.  No residency assumption is needed.
//  * No dependency counters and no CSC fan-out: the output x is pre-filled
//    with a marker, and each lane waits directly on the x(j) it needs with a
//    GPU-scope relaxed load.  The published value is its own ready flag, so
//    a dependency costs one L2 round trip and no fence.
//  * A row is reduced by a sub-warp of W lanes (W chosen per matrix).  The
//    paper lets lane 0 spin and relies on warp lockstep, which sm_70 and
//    later no longer guarantee.  Here the whole warp stays converged, in one of
//    two ways.  Rows of one level never depend on one another, so the warp waits
//    until all their values are there, folds, reduces and publishes them as one
//    (a ticket that straddles a few levels does so level by level).  Where the
//    rows of a ticket differ (a long row among short ones), every row is
//    folded and published as soon as its own values are there (rows_apart).
//
// What bounds it: a hop of the dependency chain, which is an L2 handshake
// (~350 ns), the fold and lane reduction that follow the last arrival (~64 cycles
// per FP64 instruction) and the instructions around them (4 to 5 cycles each, a
// taken branch ~30).  The loop that polls therefore does nothing else, a row's
// next chunk of entries is loaded before the wait for the current one, and
// whatever does not depend on x is computed before the first wait.  A warp that
// waits for more than a quarter of the spin limit goes on in rows_apart(), so that
// a value that never comes holds up only the rows that depend on it.
//
// Measured against the kernel before (every row folded and published by itself,
// tickets of any levels in one round loop), plan defaults, FP64, us: 7-point
// 61 x 47 x 53 in place 205 -> 182 and its adjoint 210 -> 182, 27-point of that
// size 467 -> 354, 128^3 ILU(0) L 570 -> 536; general matrix of 150001 rows 5656 ->
// 5300 and its adjoint 5688 -> 4927 (16 lanes; 32 lanes 4858 -> 4670), of 600001 rows
// with 32 lanes 18924 -> 18425.  Of these, two entries a lane instead of four at
// 16 and 32 lanes and a lane sum with at most three branches give the last 3 to 8 %
// on the 27-point and the general ones.
#include "rows_apart.cuh"

namespace sptrsv {

template <typename T>
__global__ void prep_self_k(int n, int nrhs, T* x, long long ldx, const T* b, long long ldb,
                            T* bcopy, int* ticket) {
    const long long total = (long long)n * nrhs;
    const long long stride = (long long)gridDim.x * blockDim.x;
    if (nrhs == 1) {
        for (long long e = (long long)blockIdx.x * blockDim.x + threadIdx.x; e < total; e += stride) {
            if (bcopy) bcopy[e] = b[e * ldb];
            x[e * ldx] = Marker<T>::pending_value();
        }
    } else {
        for (long long e = (long long)blockIdx.x * blockDim.x + threadIdx.x; e < total; e += stride) {
            const long long r = e / nrhs;
            const long long c = e - r * nrhs;
            if (bcopy) bcopy[e] = b[r * ldb + c];
            x[r * ldx + c] = Marker<T>::pending_value();
        }
    }
    if (blockIdx.x == 0 && threadIdx.x == 0) *ticket = 0;
}

cudaError_t launch_prep_self(bool f64, int n, int nrhs, void* x, long long ldx, const void* b,
                             long long ldb, void* bcopy, int* ticket, int grid, cudaStream_t s) {
    long long want = ((long long)n * nrhs + 255) / 256;
    int g = (int)(want < grid ? want : grid);
    if (g < 1) g = 1;
    if (f64)
        prep_self_k<double><<<g, 256, 0, s>>>(n, nrhs, (double*)x, ldx, (const double*)b, ldb,
                                              (double*)bcopy, ticket);
    else
        prep_self_k<float><<<g, 256, 0, s>>>(n, nrhs, (float*)x, ldx, (const float*)b, ldb,
                                             (float*)bcopy, ticket);
    return cudaGetLastError();
}


namespace {

constexpr int kMaxSelfBlock = 512;  // larger blocks run as several of this size
constexpr int kSelfHot = 64;        // polls of one wait before the warp backs off

// Whether the warp takes the rows of a ticket as one, where the matrix as a
// whole does not say so (SolveParams::rows_alike): equally many chunks of
// entries, lengths within a factor of about two (unless there are only two
// rows), and one level, or at most kLevels levels of rows of one chunk (longer rows of
// its second level would begin when the first is done: dense triangle of 2000 rows, 8
// lanes, 38.9 ms as one and 1.7 apart).  A general matrix of 20001 rows with 4 lanes
// per row (mean row 14 entries, longest 900) took 2.36 ms with every ticket as
// one and 1.09 ms with its rows apart.
template <int W>
__device__ __forceinline__ bool alike(bool has, int len, int lev) {
    constexpr unsigned FULL = 0xffffffffu;
    constexpr int kLevels = 4;
    const int most = __reduce_max_sync(FULL, has ? len : 0);
    const int least = __reduce_min_sync(FULL, has ? len : 0x7fffffff);
    const int top = __reduce_max_sync(FULL, has ? lev : -1);
    const int low = __reduce_min_sync(FULL, has ? lev : 0x7fffffff);
    constexpr int C = W * ChunkOf<W>::E;
    if (top - low >= (most > C ? 1 : kLevels)) return false;
    if ((most + C - 1) / C != (least + C - 1) / C) return false;
    return W >= 16 || most <= 2 * least + 2;
}

}  // namespace

// PERM: the pattern is the plan's level-ordered copy (SPTRSV_ALGO_SELF_PERMUTED):
// row position k of jlev holds the entries of row jlev[k] in fold order (an
// upper row's last entry first), with column indices renumbered to positions
// and the values copied alongside (p.ptr, p.idx, p.vals), so a warp's rows and
// the unknowns they wait on are contiguous.  Results are published in p.xp (position order,
// the array that is polled) and stored to x(jlev[k]) for the caller.  The
// arithmetic and its order are those of the unpermuted kernel, so both give
// bitwise identical results for the same sub-warp width.
//
// SMALL: one block solves the whole system with its unknowns in shared memory
// (a hop is a shared-memory poll instead of an L2 handshake), for systems that
// fit there and whose levels are too narrow to occupy more than one SM.
template <typename T, int W, bool MAP, bool PERM, bool SMALL>
__global__ void __launch_bounds__(kMaxSelfBlock, 1)
    self_solve_k1(const __grid_constant__ SolveParams p) {
    extern __shared__ __align__(16) unsigned char self_smem[];
    __shared__ int s_next;
    constexpr int R = 32 / W;
    constexpr int E = ChunkOf<W>::E;
    constexpr unsigned FULL = 0xffffffffu;
    const int lane = threadIdx.x & 31;
    const int grp = lane / W;
    const int sl = lane - grp * W;
    T* xs = (T*)self_smem;
    T* x = (T*)p.x;
    T* xpub = SMALL ? xs : PERM ? (T*)p.xp : x;  // the array rows publish to and wait on
    const long long ldp = (SMALL || PERM) ? 1 : p.ldx;
    const long long patience = p.spin.limit / 4 + 1;
    auto look = [&](int c) -> T {
        return SMALL ? lds_relaxed(xpub + c) : ld_relaxed(xpub + (long long)c * ldp);
    };
    if (SMALL) {
        for (int k = threadIdx.x; k < p.n; k += blockDim.x) xs[k] = Marker<T>::pending_value();
        if (threadIdx.x == 0) s_next = 0;
        __syncthreads();
    }
    int* const ticket = SMALL ? &s_next : p.ticket;
    int t = 0;
    if (lane == 0) t = atomicAdd(ticket, 1);
    t = __shfl_sync(FULL, t, 0);
    while ((long long)t * R < p.n) {
        int tn = 0;
        if (!SMALL && lane == 0) tn = atomicAdd(ticket, 1);  // consumed after this one
        Row<T> r = take_row<T, W, PERM>(p, (long long)t * R + grp);
        if (R > 1 && !p.rows_alike && !alike<W>(r.has, r.end - r.beg, r.lev)) {
            if (!rows_apart<T, W, MAP, PERM, SMALL>(p, t, xs, false, patience))
                tn = stuck_rows<T, W, MAP, PERM, SMALL>(p, t, tn, ticket, xs);
            if (SMALL && lane == 0) tn = atomicAdd(ticket, 1);
            t = __shfl_sync(FULL, tn, 0);
            continue;
        }
        start_row<T, W, MAP>(p, r, sl);
        int q0 = r.beg + sl, c[E];
        T a[E], v[E];
        load_entries<T, W, MAP, PERM, E>(p, r, q0, c, a);
#pragma unroll
        for (int e = 0; e < E; ++e) {
            v[e] = T(0);
            if (c[e] >= 0) v[e] = look(c[e]);
        }
        scale_entries(p, r.dinv, c, a);
        const int span = warp_span<W>(r.has, r.end - r.beg);
        const long long own = PERM ? r.k : (long long)r.i * ldp;
        bool todo = r.has, ok = true;
        const bool out = r.has && sl == 0 && r.i != p.withhold;
        while (true) {
            // the rows of the lowest level that is left
            bool act = todo;
            if (W < 32) {
                const int low = __reduce_min_sync(FULL, todo ? r.lev : 0x7fffffff);
                act = todo && r.lev == low;
            }
            while (true) {  // chunks of entries
                const bool more = __any_sync(FULL, act && q0 + W * E < r.end);
                // slots in use: the chunk's dead slots come after its live ones,
                // but for the diagonal of a row whose fold order it does not end
                unsigned slots = 0;
#pragma unroll
                for (int e = 0; e < E; ++e)
                    if (__any_sync(FULL, act && c[e] >= 0)) slots |= 1u << e;
                int c2[E];
                T a2[E];
                if (more) {
                    load_entries<T, W, MAP, PERM, E>(p, r, q0 + W * E, c2, a2);
                    scale_entries(p, r.dinv, c2, a2);
                }
                long long polls = 0;
                while (true) {
                    bool pend = false;
#pragma unroll
                    for (int e = 0; e < E; ++e) pend |= Marker<T>::pending(v[e]);
                    if (!__any_sync(FULL, act && pend)) break;
                    if (++polls > kSelfHot) {
                        if (polls > patience) {
                            ok = false;
                            break;
                        }
                        __nanosleep(32);
                    }
#pragma unroll
                    for (int e = 0; e < E; ++e)
                        if (Marker<T>::pending(v[e])) v[e] = look(c[e]);
                }
                if (!ok) break;
#pragma unroll
                for (int e = 0; e < E; ++e) {
                    if (!(slots & (1u << e))) continue;
                    if (act) r.sum = fma(-a[e], v[e], r.sum);  // no entry: adds -0 * 0
                }
                if (!more) break;
                q0 = advance(q0, W * E, r.end);
#pragma unroll
                for (int e = 0; e < E; ++e)
                    if (act) {
                        c[e] = c2[e];
                        a[e] = a2[e];
                        v[e] = T(0);
                        if (c[e] >= 0) v[e] = look(c[e]);
                    }
            }
            if (!ok) break;
            const T tot = row_sum<W>(r.sum, span);
            if (act && out) {
                const T val = publishable(tot);
                if (SMALL)
                    *(volatile T*)(xpub + own) = val;
                else
                    st_relaxed(xpub + own, val);
                if (p.xacc)
                    accumulate_with(p, r.i, 0, val, r.xbase);
                else if (PERM || SMALL)
                    x[(long long)r.i * p.ldx] = val;
            }
            if (W == 32) break;
            todo = todo && !act;
            if (!__any_sync(FULL, todo)) break;
            // lanes of the next level: q0 is still their first chunk's
            if (todo) q0 = r.beg + sl;
        }
        if (!ok) tn = stuck_rows<T, W, MAP, PERM, SMALL>(p, t, tn, ticket, xs);
        if (SMALL && lane == 0) tn = atomicAdd(ticket, 1);
        t = __shfl_sync(FULL, tn, 0);
    }
}

namespace {

// Calls f(kernel) with the instance a launch with these choices uses.
template <typename T, int W, typename F>
cudaError_t self_w(bool map, bool perm, bool small, F f) {
    if (small)
        return perm ? f(self_solve_k1<T, W, false, true, true>)
                    : map ? f(self_solve_k1<T, W, true, false, true>)
                          : f(self_solve_k1<T, W, false, false, true>);
    return perm ? f(self_solve_k1<T, W, false, true, false>)
                : map ? f(self_solve_k1<T, W, true, false, false>)
                      : f(self_solve_k1<T, W, false, false, false>);
}

template <typename T, typename F>
cudaError_t self_t(int lanes, bool map, bool perm, bool small, F f) {
    switch (lanes) {
        case 1: return self_w<T, 1>(map, perm, small, f);
        case 2: return self_w<T, 2>(map, perm, small, f);
        case 4: return self_w<T, 4>(map, perm, small, f);
        case 8: return self_w<T, 8>(map, perm, small, f);
        case 16: return self_w<T, 16>(map, perm, small, f);
        case 32: return self_w<T, 32>(map, perm, small, f);
        default: return cudaErrorInvalidValue;
    }
}

template <typename F>
cudaError_t self_any(bool f64, int lanes, bool map, bool perm, bool small, F f) {
    return f64 ? self_t<double>(lanes, map, perm, small, f)
               : self_t<float>(lanes, map, perm, small, f);
}

}  // namespace

cudaError_t launch_self_k1(bool f64, int lanes, const SolveParams& p, int grid, int block,
                           cudaStream_t s) {
    if (block > kMaxSelfBlock) {  // the same warps in blocks of kMaxSelfBlock threads
        grid = (int)(((long long)grid * block + kMaxSelfBlock - 1) / kMaxSelfBlock);
        block = kMaxSelfBlock;
    }
    // a level-ordered copy holds its values gathered: no map
    return self_any(f64, lanes, !p.xp && p.vmap, p.xp != nullptr, false, [&](auto k) {
        k<<<grid, block, 0, s>>>(p);
        return cudaGetLastError();
    });
}

// The shared memory that a one-block instance may ask for: the device's opt-in limit
// less the room of its static variables, the same on every call.  The limit belongs to
// the kernel on the device, not to a plan: a call that set its own smaller size could
// come between the two steps of another thread's larger one, whose launch then fails.
static cudaError_t small_limit(const void* k) {
    int dev = 0, optin = 0;
    cudaError_t e = cudaGetDevice(&dev);
    if (e == cudaSuccess)
        e = cudaDeviceGetAttribute(&optin, cudaDevAttrMaxSharedMemoryPerBlockOptin, dev);
    return e == cudaSuccess
               ? cudaFuncSetAttribute(k, cudaFuncAttributeMaxDynamicSharedMemorySize, optin - 128)
               : e;
}

cudaError_t launch_self_small(bool f64, int lanes, const SolveParams& p, int block,
                              cudaStream_t s) {
    const size_t smem = (f64 ? 8 : 4) * (size_t)p.n;  // checked by the caller
    if (block > kMaxSelfBlock) block = kMaxSelfBlock;
    return self_any(f64, lanes, !p.xp && p.vmap, p.xp != nullptr, true, [&](auto k) {
        if (smem > 48 * 1024 - 256) {
            const cudaError_t e = small_limit((const void*)k);
            if (e != cudaSuccess) return e;
        }
        k<<<1, block, smem, s>>>(p);
        return cudaGetLastError();
    });
}

int self_k1_blocks_per_sm(bool f64, int lanes, bool map, bool perm, int block) {
    int nb = 0;
    const int run = block > kMaxSelfBlock ? kMaxSelfBlock : block;
    const cudaError_t e = self_any(f64, lanes, map, perm, false, [&](auto k) {
        return cudaOccupancyMaxActiveBlocksPerMultiprocessor(&nb, k, run, 0);
    });
    if (e != cudaSuccess || nb < 1) return 1;
    nb = (int)((long long)nb * run / block);  // in blocks of the size asked for
    return nb > 0 ? nb : 1;
}

}  // namespace sptrsv
