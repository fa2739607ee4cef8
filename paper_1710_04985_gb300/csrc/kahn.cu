// Level analysis by Kahn's topological sort (Sec. 4.4.1), the setup the
// paper runs on the GPU, kept beside the sync-free sweep of analysis.cu for
// comparison (sptrsv_reanalyze).
//
// Kahn's algorithm peels the dependency DAG one level at a time: the roots
// (rows with no pending dependency) form level 0; removing a level's rows
// and their outgoing edges exposes the next level's roots.  Outgoing edges of
// row i are the entries of column i, read as row i of the CSR of the
// transpose (the DEP/TRANS steps of Table 1), and count(r) holds the
// dependencies of row r not yet removed.
//
// Two drivers:
//  * host loop, as in the paper: one launch per level and one device-to-host
//    copy of the queue end after it, so the host knows the next frontier;
//  * persistent: one cooperative launch sweeps every level, the frontiers
//    separated by a grid-wide barrier instead of a kernel boundary and a
//    copy.  The barrier is a monotone arrival counter with bounded waits:
//    past the spin limit a block records SPTRSV_ERR_TIMEOUT and stops, so the
//    launch always ends (a cooperative launch keeps every block resident, so
//    the limit is reached only if a block died).
// Both produce lev[] (0-based, the level at which each row became a root)
// and the level count; the level sets are then built from lev[] exactly as
// after the sweep, so every method gives the same ilev/jlev.
#include "internal.h"

namespace sptrsv {

// Level 0: count = count0; rows without dependencies are roots.
__global__ void kahn_roots_k(int n, const int* __restrict__ count0, int* count, int* lev,
                             int* queue, int* qend) {
    for (long long r = (long long)blockIdx.x * blockDim.x + threadIdx.x; r < n;
         r += (long long)gridDim.x * blockDim.x) {
        const int c = count0[r];
        count[r] = c;
        if (c == 0) {
            lev[r] = 0;
            queue[atomicAdd(qend, 1)] = (int)r;
        } else {
            lev[r] = -1;
        }
    }
}

cudaError_t launch_kahn_roots(int n, const int* count0, int* count, int* lev, int* queue,
                              int* qend, cudaStream_t s) {
    if (n <= 0) return cudaSuccess;
    long long g = ((long long)n + 255) / 256;
    if (g > 65535) g = 65535;
    kahn_roots_k<<<(int)g, 256, 0, s>>>(n, count0, count, lev, queue, qend);
    return cudaGetLastError();
}

// Removes the frontier queue[first, last) (rows of level `level`): a warp
// per frontier row, its lanes over the row's outgoing edges; a dependent
// whose count drops to zero becomes a root of level + 1 and is appended at
// *qend.  A queue entry past n (impossible for a valid pattern) is reported.
__device__ __forceinline__ void kahn_remove(const int* __restrict__ dptr,
                                            const int* __restrict__ didx, int* count, int* lev,
                                            int* queue, int* qend, int n, int i, int level,
                                            int lane, unsigned long long* status) {
    const int beg = dptr[i], end = dptr[i + 1];
    for (int q = beg + lane; q < end; q += 32) {
        const int r = didx[q];
        if (r == i) continue;
        if (atomicSub(count + r, 1) == 1) {
            lev[r] = level + 1;
            const int at = atomicAdd(qend, 1);
            if (at < n) queue[at] = r;
            else report(status, r, kCodeInternal);
        }
    }
}

__global__ void kahn_level_k(const int* __restrict__ dptr, const int* __restrict__ didx,
                             int* count, int* lev, int* queue, int* qend, int n, int first,
                             int last, int level, unsigned long long* status) {
    const int lane = threadIdx.x & 31;
    const long long warps = ((long long)gridDim.x * blockDim.x) >> 5;
    for (long long w = (((long long)blockIdx.x * blockDim.x) >> 5) + (threadIdx.x >> 5);
         first + w < last; w += warps)
        kahn_remove(dptr, didx, count, lev, queue, qend, n, __ldcg(queue + first + w), level,
                    lane, status);
}

cudaError_t launch_kahn_level(const int* dptr, const int* didx, int* count, int* lev, int* queue,
                              int* qend, int n, int first, int last, int level,
                              unsigned long long* status, int max_grid, cudaStream_t s) {
    const long long rows = (long long)last - first;
    if (rows <= 0) return cudaSuccess;
    long long g = (rows + 7) / 8;  // 8 warps per 256-thread block
    if (g > max_grid) g = max_grid;
    kahn_level_k<<<(int)g, 256, 0, s>>>(dptr, didx, count, lev, queue, qend, n, first, last,
                                        level, status);
    return cudaGetLastError();
}

// Grid-wide barrier number `gen` of a cooperative launch: every block adds one
// arrival, and `add` to a total, to one of three 64-bit words used in turn (zero
// at launch) and waits until all have arrived; *total is the sum of their `add`.
// A barrier's word is cleared after the next barrier (every block has left it by
// then) and used again by the one after that.  Release/acquire order the writes
// of one generation before the reads of the next.  Returns false if the wait ran
// past the limit (then SPTRSV_ERR_TIMEOUT is recorded).
__device__ __forceinline__ bool grid_barrier(unsigned long long* words, unsigned gen, int add,
                                             int* total, long long limit,
                                             unsigned long long* status, int row) {
    __shared__ int s_ok, s_total;
    __syncthreads();
    if (threadIdx.x == 0) {
        unsigned long long* w = words + gen % 3;
        const unsigned long long mine = ((unsigned long long)(unsigned)add << 32) | 1ull;
        asm volatile("red.release.gpu.global.add.u64 [%0], %1;" ::"l"(w), "l"(mine) : "memory");
        int ok = 1;
        long long spins = 0;
        unsigned long long v;
        while (true) {
            asm volatile("ld.acquire.gpu.global.u64 %0, [%1];" : "=l"(v) : "l"(w) : "memory");
            if ((unsigned)v >= gridDim.x) break;
            if (++spins >= limit) {
                report(status, row, kCodeTimeout);
                ok = 0;
                break;
            }
            if (spins > 64) __nanosleep(64);
        }
        if (blockIdx.x == 0) *(volatile unsigned long long*)(words + (gen + 2) % 3) = 0;
        s_ok = ok;
        s_total = (int)(v >> 32);
    }
    __syncthreads();
    *total = s_total;
    return s_ok != 0;
}

// Roots a block gathers in shared memory.
constexpr int kGather = 2048;
struct Gather {
    int row[kGather], beg[kGather], end[kGather];
    int cnt;
    int at;
};

// Persistent driver.  The frontier of level L is queue[base_L, base_L +
// size_L), with the rows' outgoing edges [beg, end) in span; its removal appends
// the roots of level L + 1 right after it.  The places of a level's roots are
// counted in three rotating words cnt[L % 3]: the roots of level L + 1 in
// cnt[(L + 1) % 3], while block 0 clears cnt[(L + 2) % 3], which nobody adds to
// before the next barrier.  The number of roots itself comes with the barrier.
//
// What bounds a level is the chain root -> edge -> counter of the dependent ->
// place in the queue -> barrier, an L2 latency each, so as many rows as possible
// go through it at once (`lanes` lanes to a row: a lane per edge of an average
// row; consecutive warps of the frontier on different SMs), a root's edge range
// is loaded by the block that found it while its place is on the way, and a
// block gathers its roots in shared memory and takes their places with one
// atomic (one atomic per root on the one counter of a level, 5490 roots on the
// 128^3 factor, had all of them queue up in L2).  Plan setup of the 128^3 ILU(0)
// L factor 4.26 -> 3.42 ms, of the 9-point 1012 x 974 lower triangle (narrow
// levels) 13.7 -> 10.9 ms, of the 27-point 70 x 89 x 103 one 4.77 -> 4.24 ms.
//
// Wide levels run on the whole grid, one grid barrier each.  A level of at
// most `narrow` rows runs on block 0 alone, which keeps going through
// consecutive narrow levels with the frontier in shared memory and block
// barriers only, and then publishes the frontier and (base, size, level) in
// ctl[0..2]; the other blocks meanwhile wait at the grid barrier that closes the
// run.  A run opens with one more grid barrier, after which every block has
// read the size it starts from.  cnt[0] holds the roots queued by kahn_roots_k;
// cnt[1], cnt[2] and words[0..2] start at zero.  Writes the level count and
// cnt[3] = rows leveled.
constexpr int kNarrowRun = 4096;

// Removes row i's edges [beg, end) with the lanes sl, sl + lanes, ...; new roots
// go to g, those beyond its room to over(place, root), place >= kGather.
template <typename F>
__device__ __forceinline__ void kahn_remove_row(const int* __restrict__ didx, int* count, int* lev,
                                                int level, int i, int beg, int end, int sl,
                                                int lanes, Gather& g, F over) {
    for (int q = beg + sl; q < end; q += lanes) {
        const int r = didx[q];
        if (r == i) continue;
        if (atomicSub(count + r, 1) == 1) {
            lev[r] = level + 1;
            const int at = atomicAdd(&g.cnt, 1);
            if (at < kGather) g.row[at] = r;
            else over(at, r);
        }
    }
}

__global__ void __launch_bounds__(1024)
    kahn_persistent_k(const int* __restrict__ dptr, const int* __restrict__ didx, int* count,
                      int* lev, int* queue, int2* span, int* cnt, int* ctl, int n, int narrow,
                      int lanes, int probe_level, int probe_min_avg, unsigned long long* words,
                      int* nlev_out, unsigned long long* status, long long limit) {
    extern __shared__ __align__(16) unsigned char kahn_smem[];
    Gather* const g = (Gather*)kahn_smem;  // two of them
    const int lane = threadIdx.x & 31;
    const int per = 32 / lanes, sl = lane % lanes;
    const int bwarps = blockDim.x >> 5, bwid = threadIdx.x >> 5;
    const long long warps = (long long)gridDim.x * bwarps;
    const long long wid = (long long)bwid * gridDim.x + blockIdx.x;
    unsigned gen = 0;
    long long base = 0;
    int size = *(volatile int*)cnt;  // roots, queued before this launch
    int level = 0, total = 0;
    bool spans = false;  // the frontier's edge ranges are in span (not level 0's)
    // Level at which the next probe is taken (0: none left).
    int next_probe = probe_level > 0 ? probe_level : 0;
    bool postponed = false;
    if (threadIdx.x == 0) g[0].cnt = g[1].cnt = 0;
    __syncthreads();
    while (size > 0) {
        // Early exit for deep, narrow graphs (a level costs more here than in
        // the sweep): every block sees the same (base, size, level) here, so
        // all of them decide alike.  Levels that are still widening (the
        // current one at least 1.5 times the average so far) get one second
        // look at four times the level, which then asks for a 1.5 times larger
        // average.
        if (next_probe > 0 && level >= next_probe) {
            next_probe = 0;
            const long long need = postponed ? (3ll * probe_min_avg) / 2 : probe_min_avg;
            if (base < (long long)level * need) {
                if (!postponed && 2ll * size * level >= 3ll * base) {
                    postponed = true;
                    next_probe = 4 * level;
                } else {
                    if (blockIdx.x == 0 && threadIdx.x == 0) *nlev_out = -1;
                    return;
                }
            }
        }
        if (size <= narrow && size <= kGather) {
            // Every block must have read the state of the barrier just passed
            // before block 0 runs ahead.  One extra grid barrier per run.
            if (!grid_barrier(words, gen++, 0, &total, limit, status, level)) return;
            if (blockIdx.x == 0) {
                int cur = 0;
                for (int k = threadIdx.x; k < size; k += blockDim.x) {
                    const int r = __ldcg(queue + base + k);
                    g[0].row[k] = r;
                    g[0].beg[k] = dptr[r];
                    g[0].end[k] = dptr[r + 1];
                }
                __syncthreads();
                // at most kNarrowRun levels per run, so the other blocks' wait
                // at the closing barrier stays far below its spin limit; a run
                // also stops at the probe level so that the probe is taken
                int run = 0;
                do {
                    Gather& to = g[cur ^ 1];
                    int* next = queue + base + size;
                    const long long room = (long long)n - base - size;
                    for (int f = bwid * per + lane / lanes; f < size; f += bwarps * per)
                        kahn_remove_row(didx, count, lev, level, g[cur].row[f], g[cur].beg[f],
                                        g[cur].end[f], sl, lanes, to, [&](int at, int r) {
                                            if (at < room) next[at] = r;
                                            else report(status, r, kCodeInternal);
                                        });
                    __syncthreads();
                    const int found = to.cnt;
                    const int kept = found < kGather ? found : kGather;
                    for (int k = threadIdx.x; k < kept; k += blockDim.x) {
                        const int r = to.row[k];
                        to.beg[k] = dptr[r];
                        to.end[k] = dptr[r + 1];
                    }
                    __syncthreads();
                    if (threadIdx.x == 0) to.cnt = 0;
                    base += size;
                    size = found;
                    ++level;
                    ++run;
                    cur ^= 1;
                } while (run < kNarrowRun && size > 0 && size <= narrow && size <= kGather &&
                         (next_probe == 0 || level < next_probe));
                // the frontier for the grid
                for (int k = threadIdx.x; k < size; k += blockDim.x) {
                    if (base + k >= n) {
                        report(status, (int)base, kCodeInternal);
                        break;
                    }
                    if (k < kGather) {
                        queue[base + k] = g[cur].row[k];
                        span[base + k] = make_int2(g[cur].beg[k], g[cur].end[k]);
                    } else {
                        const int r = __ldcg(queue + base + k);
                        span[base + k] = make_int2(dptr[r], dptr[r + 1]);
                    }
                }
                if (threadIdx.x == 0) {
                    ctl[0] = (int)base;
                    ctl[1] = size;
                    ctl[2] = level;
                    cnt[0] = cnt[1] = cnt[2] = 0;
                }
            }
            if (!grid_barrier(words, gen++, 0, &total, limit, status, level)) return;
            int st[3];
#pragma unroll
            for (int k = 0; k < 3; ++k)
                asm volatile("ld.relaxed.gpu.global.b32 %0, [%1];" : "=r"(st[k]) : "l"(ctl + k)
                             : "memory");
            base = st[0];
            size = st[1];
            level = st[2];
            spans = true;
            continue;
        }
        if (blockIdx.x == 0 && threadIdx.x == 0) cnt[(level + 2) % 3] = 0;
        int* tail = cnt + (level + 1) % 3;
        int* next = queue + base + size;
        int2* next_span = span + base + size;
        const long long room = (long long)n - base - size;  // places that are left
        for (long long w = wid; w * per < size; w += warps) {
            const long long f = w * per + lane / lanes;
            if (f >= size) continue;
            const int i = __ldcg(queue + base + f);
            int2 s;
            if (spans) s = __ldcg(span + base + f);
            else s = make_int2(dptr[i], dptr[i + 1]);
            kahn_remove_row(didx, count, lev, level, i, s.x, s.y, sl, lanes, g[0],
                            [&](int, int r) {
                                const int at = atomicAdd(tail, 1);
                                if (at < room) {
                                    next[at] = r;
                                    next_span[at] = make_int2(dptr[r], dptr[r + 1]);
                                } else {
                                    report(status, r, kCodeInternal);
                                }
                            });
        }
        __syncthreads();
        const int mine = g[0].cnt < kGather ? g[0].cnt : kGather;
        const int found = g[0].cnt;  // with the ones queued one by one
        if (threadIdx.x == 0 && mine > 0) g[0].at = atomicAdd(tail, mine);
        int beg = 0, end = 0;  // of this thread's first root, while the place comes
        if ((int)threadIdx.x < mine) {
            beg = dptr[g[0].row[threadIdx.x]];
            end = dptr[g[0].row[threadIdx.x] + 1];
        }
        __syncthreads();
        for (int k = threadIdx.x; k < mine; k += blockDim.x) {
            const int r = g[0].row[k];
            if (k != (int)threadIdx.x) {
                beg = dptr[r];
                end = dptr[r + 1];
            }
            const int at = g[0].at + k;
            if (at < room) {
                next[at] = r;
                next_span[at] = make_int2(beg, end);
            } else {
                report(status, r, kCodeInternal);
            }
        }
        __syncthreads();
        if (threadIdx.x == 0) g[0].cnt = 0;
        if (!grid_barrier(words, gen++, found, &total, limit, status, level)) return;
        base += size;
        size = total;
        ++level;
        spans = true;
    }
    if (blockIdx.x == 0 && threadIdx.x == 0) {
        *nlev_out = level;
        cnt[3] = (int)base;  // rows leveled, checked by the host
    }
}

// Shared memory of the kernel: 48 KB and a little, so it is opted in to.
static cudaError_t kahn_attr() {
    return cudaFuncSetAttribute(kahn_persistent_k, cudaFuncAttributeMaxDynamicSharedMemorySize,
                                (int)(2 * sizeof(Gather)));
}

int kahn_persistent_blocks_per_sm(int block) {
    int nb = 0;
    if (kahn_attr() != cudaSuccess ||
        cudaOccupancyMaxActiveBlocksPerMultiprocessor(&nb, kahn_persistent_k, block,
                                                      2 * sizeof(Gather)) != cudaSuccess ||
        nb < 1)
        return 1;
    return nb;
}

cudaError_t launch_kahn_persistent(const int* dptr, const int* didx, int* count, int* lev,
                                   int* queue, int2* span, int* cnt, int* ctl, int n, int narrow,
                                   int lanes, int probe_level, int probe_min_avg,
                                   unsigned long long* words, int* nlev_out,
                                   unsigned long long* status, long long limit, int grid,
                                   int block, cudaStream_t s) {
    cudaError_t e = kahn_attr();
    if (e != cudaSuccess) return e;
    void* args[] = {(void*)&dptr,   (void*)&didx,        (void*)&count,         (void*)&lev,
                    (void*)&queue,  (void*)&span,        (void*)&cnt,           (void*)&ctl,
                    (void*)&n,      (void*)&narrow,      (void*)&lanes,         (void*)&probe_level,
                    (void*)&probe_min_avg, (void*)&words, (void*)&nlev_out,     (void*)&status,
                    (void*)&limit};
    return cudaLaunchCooperativeKernel((const void*)kahn_persistent_k, dim3(grid), dim3(block),
                                       args, 2 * sizeof(Gather), s);
}

}  // namespace sptrsv
