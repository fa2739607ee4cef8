// Self-scheduled solve (Alg. 3, SLFR) for one right-hand side on ONE thread-block
// cluster, for systems whose levels are too narrow to occupy the GPU.
//
// The level order is cut into windows of as many rows as fit twice into a block's
// shared memory.  Every block of the cluster keeps a copy of the window's
// unknowns there: a row is published by one store into each block's shared memory
// (a lane per block) and waited for by polling the block's own copy.  Values of
// earlier windows are complete (a cluster barrier lies between two windows): they
// are loaded from global memory without a wait.  Row groups are dealt out in level
// order, a fixed one to every warp in turn; all warps of a cluster run at the same
// time and every row waits on smaller positions only, so the lowest unfinished
// group can always go on.  b(i) is read by row i before x(i) is written and
// nothing is marked beforehand: one launch, and in place needs no copy of b.
//
// What bounds it: a hop of the dependency chain as in the kernel for the whole GPU
// (solve_self.cu), with a store to a neighbour's shared memory and a poll of the own
// one (~200 ns) where that one has an L2 handshake (~700 ns there and back).  The
// rows of a warp go on and are published one by one, as their own values come.
// 16 blocks of 16 warps hold about the next ten levels of a general matrix, which
// hides the chain of loads a row starts with (order, row bounds, columns, places,
// values) without prefetching.  What limits it to narrow levels: a row costs a store
// into each of the 16 blocks, and FP64 runs on 64 units instead of 608.
//
// Measured against the kernel for the whole GPU, us, general matrices, in place, FP64
// unless said otherwise: 150001 rows with 32 lanes 4670 -> 3236 and with 16 lanes 5300
// -> 4350, its adjoint with 16 lanes 4927 -> 4254; 600001 rows 18425 -> 13188 (32
// lanes); 20001 rows 687 -> 478 (32 lanes), FP32 741 -> 367 (16 lanes); 3001 rows 177 ->
// 150.  On the level-ordered copy: 150001 rows with 32 lanes 5869 -> 3180.  Rows of a
// warp taken as one: 16 lanes 6242 (a long row holds its neighbour).
//
// A value that does not come within a quarter of the spin limit: the warp raises a
// flag in every block, all warps leave their waits and meet at the barrier, and the
// rows that are left are computed level by level, a barrier between two levels, in this
// window and the later ones.  Nothing is waited for there: what is missing then never
// comes (it is reported and taken as NaN), and every row that does not depend on it is
// exact.  A warp's groups are in level order, so it goes through them once: the rest of a
// solve takes a few times as long as usual, a barrier per level instead of a hop (40
// windows of three interleaved chains 0.42 s instead of 0.1; 3.4 s when every level went
// through its whole window).  Going back to the usual way in the next window needs a look
// for values that were never published in every wait: any such code in the wait loop cost
// FP32 solves 2 to 30 %.
#include "self_rows.cuh"

namespace sptrsv {

namespace {

constexpr int kClusterBlock = 512;         // threads per block
constexpr int kWindowBytes = 96 * 1024;    // of a window's unknowns
constexpr int kClusterHot = 64;            // polls of one wait before the warp backs off
constexpr int kMaxCluster = 16;

__device__ __forceinline__ unsigned smem_addr(const void* p) {
    return (unsigned)__cvta_generic_to_shared(p);
}
__device__ __forceinline__ void cluster_sync() {
    asm volatile("barrier.cluster.arrive.release.aligned;\n\tbarrier.cluster.wait.acquire.aligned;"
                 ::: "memory");
}
__device__ __forceinline__ unsigned cluster_addr(unsigned a, unsigned rank) {
    unsigned r;
    asm volatile("mapa.shared::cluster.u32 %0, %1, %2;" : "=r"(r) : "r"(a), "r"(rank));
    return r;
}
__device__ __forceinline__ void st_block(unsigned a, double v) {
    asm volatile("st.relaxed.cluster.shared::cluster.b64 [%0], %1;" ::"r"(a),
                 "l"(__double_as_longlong(v))
                 : "memory");
}
__device__ __forceinline__ void st_block(unsigned a, float v) {
    asm volatile("st.relaxed.cluster.shared::cluster.b32 [%0], %1;" ::"r"(a),
                 "r"(__float_as_uint(v))
                 : "memory");
}
__device__ __forceinline__ void st_block(unsigned a, int v) {
    asm volatile("st.relaxed.cluster.shared::cluster.b32 [%0], %1;" ::"r"(a), "r"(v) : "memory");
}

}  // namespace

template <typename T, int W, bool MAP, bool PERM>
__global__ void __launch_bounds__(kClusterBlock, 1)
    cluster_solve_k1(const __grid_constant__ SolveParams p, int nblocks) {
    extern __shared__ __align__(16) unsigned char ring_smem[];
    __shared__ int s_bail[2];  // by parity of the window: read after its barrier
    constexpr int R = 32 / W;
    constexpr int E = ChunkOf<W>::E;
    constexpr int H = kWindowBytes / (int)sizeof(T);  // rows of a window, a multiple of 32
    constexpr unsigned FULL = 0xffffffffu;
    const int lane = threadIdx.x & 31;
    const int grp = lane / W;
    const int sl = lane - grp * W;
    const unsigned mine = group_mask<W>(lane);
    const int rank = blockIdx.x;  // the grid is one cluster
    const int warp = threadIdx.x >> 5;
    const int nwarps = blockDim.x >> 5;
    const long long ldp = PERM ? 1 : p.ldx;
    T* const x = (T*)p.x;
    T* const xpub = PERM ? (T*)p.xp : x;
    const long long patience = p.spin.limit / 4 + 1;
    const int to = lane & (kMaxCluster - 1);  // the block this lane publishes to
    const unsigned to_ring = cluster_addr(smem_addr(ring_smem), to < nblocks ? to : rank);

    for (int k = threadIdx.x; k < H && k < p.n; k += blockDim.x)
        ((T*)ring_smem)[k] = Marker<T>::pending_value();
    if (threadIdx.x < 2) s_bail[threadIdx.x] = 0;
    cluster_sync();

    bool slow = false;
    int buf = 0;
    for (int base = 0; base < p.n; base = next_window(base, H, p.n), buf ^= 1) {
        const T* const ring = (const T*)ring_smem + buf * H;
        volatile int* const bail = &s_bail[buf];
        const unsigned to_win = to_ring + (unsigned)buf * (unsigned)kWindowBytes;
        const int rows = p.n - base < H ? p.n - base : H;
        // the unknown in column c: its place in the window, or a negative number
        auto place = [&](int c) -> int { return (PERM ? c : p.ipos[c]) - base; };
        auto look = [&](int c, int at) -> T {
            return at >= 0 ? lds_relaxed(ring + at) : ld_relaxed(xpub + (long long)c * ldp);
        };
        // publishes the sums of the rows `act` (in the first lanes of their groups)
        auto publish = [&](const Row<T>& r, bool act, T tot) {
            T val = r.i == p.withhold ? Marker<T>::pending_value() : publishable(tot);
            const unsigned rows_out = __ballot_sync(FULL, act);
#pragma unroll
            for (int q = 0; q < R; q += 2) {
                const int src = (q + (lane >> 4)) * W;
                const T v = __shfl_sync(FULL, val, src & 31);
                const int at = (int)(r.k - grp - base) + q + (lane >> 4);
                if (src < 32 && ((rows_out >> src) & 1) && to < nblocks)
                    st_block(to_win + (unsigned)at * (unsigned)sizeof(T), v);
            }
            if (act && sl == 0) {
                st_relaxed(xpub + (PERM ? r.k : (long long)r.i * ldp), val);
                if (p.xacc) {
                    if (r.i != p.withhold) accumulate_with(p, r.i, 0, val, r.xbase);
                } else if (PERM) {
                    x[(long long)r.i * p.ldx] = val;
                }
            }
        };
        if (next_window(base, H, p.n) < p.n) {
            T* const next = (T*)ring_smem + (buf ^ 1) * H;
            for (int k = threadIdx.x; k < H; k += blockDim.x) next[k] = Marker<T>::pending_value();
        }
        for (int g = rank + nblocks * warp; !slow && g * R < rows; g += nblocks * nwarps) {
            if (__any_sync(FULL, *bail != 0)) break;
            Row<T> r = take_row<T, W, PERM>(p, (long long)base + g * R + grp);
            start_row<T, W, MAP>(p, r, sl);
            int q0 = r.beg + sl, c[E], at[E];
            T a[E], v[E];
            load_entries<T, W, MAP, PERM, E>(p, r, q0, c, a);
#pragma unroll
            for (int e = 0; e < E; ++e) at[e] = c[e] >= 0 ? place(c[e]) : 0;
#pragma unroll
            for (int e = 0; e < E; ++e) {
                v[e] = T(0);
                if (c[e] >= 0) v[e] = look(c[e], at[e]);
            }
            scale_entries(p, r.dinv, c, a);
            const int span = warp_span<W>(r.has, r.end - r.beg);
            bool todo = r.has, ok = true;
            int c2[E], at2[E];
            T a2[E];
            // the row's next chunk, for the lanes `on`
            auto load_next = [&](bool on) {
                load_entries<T, W, MAP, PERM, E>(p, r, on ? q0 + W * E : r.end, c2, a2);
#pragma unroll
                for (int e = 0; e < E; ++e) at2[e] = c2[e] >= 0 ? place(c2[e]) : 0;
                scale_entries(p, r.dinv, c2, a2);
            };
            if (__any_sync(FULL, todo && q0 + W * E < r.end)) load_next(todo);
            while (true) {
                // rows go on as soon as the values of their chunk are there, each by
                // itself: a long row does not hold up its neighbour
                unsigned slots = 0;
#pragma unroll
                for (int e = 0; e < E; ++e)
                    if (__any_sync(FULL, todo && c[e] >= 0)) slots |= 1u << e;
                bool act = todo;
                long long polls = 0;
                while (true) {
                    bool pend = false;
#pragma unroll
                    for (int e = 0; e < E; ++e) pend |= Marker<T>::pending(v[e]);
                    const unsigned wait = __ballot_sync(FULL, todo && pend);
                    if (wait == 0) break;
                    if (W < 32) {
                        act = todo && (wait & mine) == 0;
                        if (__any_sync(FULL, act)) break;
                    }
                    if (++polls > kClusterHot) {
                        if (polls > patience && lane < nblocks)
                            st_block(cluster_addr(smem_addr(&s_bail[buf]), lane), 1);
                        if (__any_sync(FULL, *bail != 0) || polls > 2 * patience + 1024) {
                            ok = false;
                            break;
                        }
                        __nanosleep(32);
                    }
#pragma unroll
                    for (int e = 0; e < E; ++e)
                        if (Marker<T>::pending(v[e])) v[e] = look(c[e], at[e]);
                }
                if (!ok) break;
#pragma unroll
                for (int e = 0; e < E; ++e) {
                    if (!(slots & (1u << e))) continue;
                    if (act) r.sum = fma(-a[e], v[e], r.sum);  // no entry: adds -0 * 0
                }
                const bool more = act && q0 - sl + W * E < r.end;  // the same in the whole row
                const bool fin = act && !more;
                if (__any_sync(FULL, fin)) {
                    publish(r, fin, row_sum<W>(r.sum, span));
                    todo = todo && !fin;
                    if (W == 32 || !__any_sync(FULL, todo)) break;
                }
                if (__any_sync(FULL, more)) {
                    if (more) {
                        q0 += W * E;
#pragma unroll
                        for (int e = 0; e < E; ++e) {
                            c[e] = c2[e];
                            a[e] = a2[e];
                            at[e] = at2[e];
                            v[e] = T(0);
                            if (c[e] >= 0) v[e] = look(c[e], at[e]);
                        }
                    }
                    // the chunk after it; the other rows' next one once more
                    if (__any_sync(FULL, todo && q0 - sl + W * E < r.end)) load_next(todo);
                }
            }
            if (!ok) break;
        }
        __syncwarp();
        cluster_sync();
        slow = slow || *bail;  // the same in every block
        if (!slow) continue;
        // level by level: what has not been published by now and is not published
        // one barrier later never is
        const int last = p.lev[p.jlev[base + rows - 1]];
        int g = rank + nblocks * warp;  // this warp's lowest group with rows left
        for (int m = p.lev[p.jlev[base]]; m <= last; ++m) {
            for (; g * R < rows; g += nblocks * nwarps) {
                Row<T> r = take_row<T, W, PERM>(p, (long long)base + g * R + grp);
                const int lev = r.has ? p.lev[r.i] : m;
                const bool act = r.has && lev == m &&
                                 Marker<T>::pending(lds_relaxed(ring + (r.k - base)));
                if (__any_sync(FULL, act)) {
                    start_row<T, W, MAP>(p, r, sl);
                    int c[E];
                    T a[E];
                    for (int q0 = r.beg + sl; __any_sync(FULL, act && q0 < r.end);
                         q0 = advance(q0, W * E, r.end)) {
                        load_entries<T, W, MAP, PERM, E>(p, r, q0, c, a);
                        scale_entries(p, r.dinv, c, a);
#pragma unroll
                        for (int e = 0; e < E; ++e)
                            if (act && c[e] >= 0) {
                                T v = look(c[e], place(c[e]));
                                if (Marker<T>::pending(v)) {
                                    report(p.status, r.i, kCodeTimeout);
                                    v = Marker<T>::canonical_nan();
                                }
                                r.sum = fma(-a[e], v, r.sum);
                            }
                    }
                    publish(r, act, row_sum<W>(r.sum, warp_span<W>(r.has, r.end - r.beg)));
                }
                if (__any_sync(FULL, lev > m)) break;  // rows of a later level
            }
            __syncwarp();
            cluster_sync();
        }
    }
}

namespace {

template <int W>
struct Lanes {
    static constexpr int value = W;
};

// Calls f(kernel) with the instance a launch with these choices uses.
template <typename F>
cudaError_t cluster_any(bool f64, int lanes, bool map, bool perm, F f) {
    auto w = [&](auto t, auto l) {
        using T = decltype(t);
        constexpr int W = decltype(l)::value;
        return perm ? f(cluster_solve_k1<T, W, false, true>)
                    : map ? f(cluster_solve_k1<T, W, true, false>)
                          : f(cluster_solve_k1<T, W, false, false>);
    };
    auto any = [&](auto t) {
        switch (lanes) {
            case 16: return w(t, Lanes<16>());
            case 32: return w(t, Lanes<32>());
            default: return cudaErrorInvalidValue;
        }
    };
    return f64 ? any(double()) : any(float());
}

size_t ring_bytes(bool f64, int n) {
    const size_t bytes = (f64 ? 8 : 4) * (size_t)n;
    return bytes > kWindowBytes ? 2 * (size_t)kWindowBytes : (bytes + 15) / 16 * 16;
}

cudaLaunchConfig_t cluster_config(int nblocks, size_t smem, cudaStream_t s,
                                  cudaLaunchAttribute* attr) {
    cudaLaunchConfig_t cfg = {};
    cfg.gridDim = dim3((unsigned)nblocks, 1, 1);
    cfg.blockDim = dim3(kClusterBlock, 1, 1);
    cfg.dynamicSmemBytes = smem;
    cfg.stream = s;
    attr[0].id = cudaLaunchAttributeClusterDimension;
    attr[0].val.clusterDim.x = (unsigned)nblocks;
    attr[0].val.clusterDim.y = 1;
    attr[0].val.clusterDim.z = 1;
    cfg.attrs = attr;
    cfg.numAttrs = 1;
    return cfg;
}

}  // namespace

int cluster_blocks(bool f64, int lanes, bool map, bool perm) {
    int blocks = 0;
    // only an error of these calls is cleared, not one that the caller's code left
    auto asked = [](cudaError_t e) {
        if (e != cudaSuccess) cudaGetLastError();
        return e;
    };
    const cudaError_t rc = cluster_any(f64, lanes, map, perm, [&](auto k) {
        cudaError_t e = asked(cudaFuncSetAttribute(
            k, cudaFuncAttributeMaxDynamicSharedMemorySize, 2 * kWindowBytes));
        if (e == cudaSuccess)
            e = asked(cudaFuncSetAttribute(k, cudaFuncAttributeNonPortableClusterSizeAllowed, 1));
        if (e != cudaSuccess) return e;
        // a size that cannot be asked for is one that cannot run: the next smaller one may
        for (int c = kMaxCluster; c >= 8 && !blocks; c /= 2) {
            cudaLaunchAttribute attr[1];
            const cudaLaunchConfig_t cfg = cluster_config(c, 2 * kWindowBytes, nullptr, attr);
            int nb = 0;
            e = asked(cudaOccupancyMaxActiveClusters(&nb, k, &cfg));
            if (e == cudaSuccess && nb > 0) blocks = c;
        }
        return blocks ? cudaSuccess : e;
    });
    return rc == cudaSuccess ? blocks : 0;
}

cudaError_t launch_cluster_k1(bool f64, int lanes, const SolveParams& p, int nblocks,
                              cudaStream_t s) {
    return cluster_any(f64, lanes, !p.xp && p.vmap, p.xp != nullptr, [&](auto k) {
        cudaLaunchAttribute attr[1];
        const cudaLaunchConfig_t cfg = cluster_config(nblocks, ring_bytes(f64, p.n), s, attr);
        const cudaError_t e = cudaLaunchKernelEx(&cfg, k, p, nblocks);
        return e == cudaSuccess ? cudaGetLastError() : e;
    });
}

}  // namespace sptrsv
