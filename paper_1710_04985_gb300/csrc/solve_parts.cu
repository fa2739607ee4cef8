// Part-ordered copy for the partitioned solve (SPTRSV_ALGO_SELF_PARTITIONED):
// level-scheduled order inside a part of consecutive rows.
//
// Parts are runs of consecutive rows in order of substitution (ascending for
// a lower system, descending for an upper one), so every dependency of a
// part lies in the part itself or in an earlier part of the same run.  The
// copy lists the parts one after another and, inside a part, its rows by
// level (Sec. 4.1), then row; every column index is renumbered to its
// position in that order, or in its part (the sliced copy, below).  A dependency then points to an earlier position,
// one inside the part to a row of a lower level of the same part.  The
// partitioned kernel (solve_partitioned.cuh) runs on this copy, one part per
// thread block: the block holds its part's unknowns in shared memory,
// where dependencies inside the part are served, and waits for earlier parts
// through the published values as in Alg. 3.  On a structured grid in natural
// order a part is a slab of whole grid lines, so the dependency hops along
// the lines stay in shared memory and only the hops between slabs go through
// L2; with levels as the order inside a part its rows are taken as they
// become ready.
//
// How the rows are cut into parts.  The substitution order is first split
// where the matrix decouples: position t starts an independent block when no
// row at or after t depends on a row before t (a block-diagonal batch of
// systems decouples at every system boundary).  These boundaries come from
// one difference array: a row at position u whose farthest dependency is at
// position f < u covers the positions f+1 .. u, and the positions no row
// covers are the block starts.  A block longer than half the part size S is
// cut into ceil(len/S) pieces of balanced length; shorter blocks that start
// in the same window of S/2 positions share one part (so a part never holds
// more than S rows).  A part never straddles two blocks unless all of them
// fit in it whole.  The parts are then handed out latest start first: a
// part's key is the level at which it must start at the latest for its
// block to finish with the deepest one -- the block's slack (deepest level
// of the matrix minus the block's own depth) plus the piece's share of the
// block's levels (piece index times levels per piece) -- and parts with
// equal keys go in order of substitution.  Keys do not decrease along a
// block's pieces, so every part still depends only on parts handed out
// before it.  The pieces of the deepest systems of a batch are taken as the
// frontier reaches them, and short systems, which have slack, fill the
// blocks in between; handing out every system's first piece before any
// second piece (the previous order) left the deepest system's later pieces
// queued behind hundreds of short systems (batch of 512: 5.06 -> 4.64 ms).
#include "internal.h"

namespace sptrsv {

namespace {

int grid_for(long long m) {
    long long g = (m + 255) / 256;
    if (g > 8192) g = 8192;
    return g < 1 ? 1 : (int)g;
}

}  // namespace

// diff[f + 1] += 1 and diff[t + 1] -= 1 for the row at substitution position
// t whose farthest dependency sits at position f < t.
__global__ void part_spans_k(int n, const int* __restrict__ ptr, const int* __restrict__ idx,
                             int upper, int* diff) {
    for (long long r = (long long)blockIdx.x * blockDim.x + threadIdx.x; r < n;
         r += (long long)gridDim.x * blockDim.x) {
        const int beg = ptr[r], end = ptr[r + 1];
        if (beg >= end) continue;
        // columns ascend inside a row: the farthest dependency is the first
        // entry of a lower row and the last entry of an upper one
        const int c = upper ? idx[end - 1] : idx[beg];
        if (c == (int)r) continue;  // only the diagonal
        const long long t = upper ? n - 1 - r : r;
        const long long f = upper ? n - 1 - c : c;
        atomicAdd(diff + f + 1, 1);
        atomicAdd(diff + t + 1, -1);
    }
}

// flag[t] = 1 where no dependency span covers t (t = 0 always): a block start.
__global__ void block_flags_k(int n, const int* __restrict__ cover, int* flag) {
    for (long long t = (long long)blockIdx.x * blockDim.x + threadIdx.x; t < n;
         t += (long long)gridDim.x * blockDim.x)
        flag[t] = (t == 0 || cover[t + 1] == 0) ? 1 : 0;
}

// start[scan[t]] = t where flag[t]; start[scan[n]] = n.
__global__ void flag_scatter_k(int n, const int* __restrict__ flag, const int* __restrict__ scan,
                               int* start) {
    for (long long t = (long long)blockIdx.x * blockDim.x + threadIdx.x; t < n;
         t += (long long)gridDim.x * blockDim.x)
        if (flag[t]) start[scan[t]] = (int)t;
    if (blockIdx.x == 0 && threadIdx.x == 0) start[scan[n]] = n;
}

// depth[b] = largest level of the rows of block b (an atomic max per warp
// when its lanes hold one block, which is the common case).
__global__ void block_depth_k(int n, int upper, const int* __restrict__ lev,
                              const int* __restrict__ bscan, int* depth) {
    for (long long t0 = (long long)blockIdx.x * blockDim.x; t0 < n;
         t0 += (long long)gridDim.x * blockDim.x) {
        const long long t = t0 + threadIdx.x;
        const bool in = t < n;
        const int b = in ? bscan[t + 1] - 1 : -1;
        const int l = in ? lev[upper ? n - 1 - t : t] : -1;
        const unsigned peers = __match_any_sync(0xffffffffu, b);
        const int m = __reduce_max_sync(peers, l);
        if (in && (threadIdx.x & 31) == __ffs(peers) - 1) atomicMax(depth + b, m);
    }
}

// flag[t] = 1 where a part starts: at the pieces of a long block (longer than
// h = S/2, cut into ceil(len/S) balanced pieces) and at a short block that
// follows a long one or starts in another window of h positions than the
// short block before it.
__global__ void part_flags_k(int n, int S, const int* __restrict__ bscan,
                             const int* __restrict__ bstart, int* flag) {
    const long long h = S / 2 > 0 ? S / 2 : 1;
    for (long long t = (long long)blockIdx.x * blockDim.x + threadIdx.x; t < n;
         t += (long long)gridDim.x * blockDim.x) {
        const int b = bscan[t + 1] - 1;
        const long long st = bstart[b], len = bstart[b + 1] - st;
        int f;
        if (len > h) {
            const long long np = (len + S - 1) / S;
            f = (t == st || (t - st) * np / len != (t - 1 - st) * np / len) ? 1 : 0;
        } else if (t != st) {
            f = 0;
        } else if (b == 0) {
            f = 1;
        } else {
            const long long pst = bstart[b - 1];
            f = (st - pst > h || st / h != pst / h) ? 1 : 0;
        }
        flag[t] = f;
    }
}

// key[p] = deepest level minus the depth of the block part p starts in, so
// that an ascending stable sort hands the deepest blocks out first.
__global__ void part_depth_keys_k(int np, int maxdepth, const int* __restrict__ pstart,
                                  const int* __restrict__ bscan, const int* __restrict__ depth,
                                  int* key) {
    for (long long p = (long long)blockIdx.x * blockDim.x + threadIdx.x; p < np;
         p += (long long)gridDim.x * blockDim.x)
        key[p] = maxdepth - depth[bscan[pstart[p] + 1] - 1];
}

// piece[p] = index of part p among the parts of its block (0 for the first).
__global__ void part_piece_k(int np, const int* __restrict__ pstart,
                             const int* __restrict__ bscan, const int* __restrict__ bstart,
                             const int* __restrict__ pscan, int* piece) {
    for (long long p = (long long)blockIdx.x * blockDim.x + threadIdx.x; p < np;
         p += (long long)gridDim.x * blockDim.x) {
        const int b = bscan[pstart[p] + 1] - 1;
        piece[p] = (int)p - (pscan[bstart[b] + 1] - 1);
    }
}

// key[p] = the estimated latest level at which part p can start: its
// block's slack (deepest level minus the block's depth) plus its piece's
// share of the block's levels (piece index times levels per piece).  Keys do
// not decrease along a block's pieces, so a stable sort keeps them in order.
__global__ void part_alap_keys_k(int np, int maxdepth, const int* __restrict__ pstart,
                                 const int* __restrict__ bscan, const int* __restrict__ bstart,
                                 const int* __restrict__ pscan, const int* __restrict__ depth,
                                 const int* __restrict__ piece, int* key) {
    for (long long p = (long long)blockIdx.x * blockDim.x + threadIdx.x; p < np;
         p += (long long)gridDim.x * blockDim.x) {
        const int b = bscan[pstart[p] + 1] - 1;
        const int d = depth[b];
        const int first = pscan[bstart[b] + 1] - 1;  // the block's first part
        const int cnt = pscan[bstart[b + 1]] - first;  // parts starting in the block
        const long long share = cnt > 1 ? (long long)piece[p] * (d + 1) / cnt : 0;
        key[p] = (maxdepth - d) + (int)share;
    }
}

// size[r] and row[r] = rows and lowest row of the part handed out r-th; atomic
// max of the sizes.
__global__ void part_sizes_k(int n, int np, int upper, const int* __restrict__ horder,
                             const int* __restrict__ pstart, int* size, int* row, int* maxsize) {
    int m = 0;
    for (long long r = (long long)blockIdx.x * blockDim.x + threadIdx.x; r < np;
         r += (long long)gridDim.x * blockDim.x) {
        const int p = horder[r];
        const int s = pstart[p + 1] - pstart[p];
        size[r] = s;
        row[r] = upper ? n - pstart[p + 1] : pstart[p];
        m = max(m, s);
    }
    m = __reduce_max_sync(0xffffffffu, m);
    if ((threadIdx.x & 31) == 0) atomicMax(maxsize, m);
}

// key[k] = hand-out rank of the part of row jlev[k].
__global__ void row_part_keys_k(int n, const int* __restrict__ jlev, int upper,
                                const int* __restrict__ pscan, const int* __restrict__ prank,
                                int* key) {
    for (long long k = (long long)blockIdx.x * blockDim.x + threadIdx.x; k < n;
         k += (long long)gridDim.x * blockDim.x) {
        const int i = jlev[k];
        const long long t = upper ? n - 1 - i : i;
        key[k] = prank[pscan[t + 1] - 1];
    }
}

// Runs of equal level inside a part, and groups of at most R rows of a run:
// the rows a warp of the partitioned kernel takes at once.  Rows of one group
// never depend on one another.
__global__ void run_flags_k(int n, const int* __restrict__ qord, const int* __restrict__ lev,
                            int* flag) {
    for (long long k = (long long)blockIdx.x * blockDim.x + threadIdx.x; k < n;
         k += (long long)gridDim.x * blockDim.x)
        flag[k] = (k == 0 || lev[qord[k]] != lev[qord[k - 1]]) ? 1 : 0;
}

__global__ void part_flag_starts_k(int np, const int* __restrict__ part_ptr, int* flag) {
    for (long long j = (long long)blockIdx.x * blockDim.x + threadIdx.x; j < np;
         j += (long long)gridDim.x * blockDim.x)
        flag[part_ptr[j]] = 1;
}

__global__ void group_flags_k(int n, int R, const int* __restrict__ rscan,
                              const int* __restrict__ rstart, int* flag) {
    for (long long k = (long long)blockIdx.x * blockDim.x + threadIdx.x; k < n;
         k += (long long)gridDim.x * blockDim.x)
        flag[k] = ((int)k - rstart[rscan[k + 1] - 1]) % R == 0 ? 1 : 0;
}

__global__ void part_groups_k(int np, const int* __restrict__ part_ptr,
                              const int* __restrict__ gscan, int* grp_ptr) {
    for (long long j = (long long)blockIdx.x * blockDim.x + threadIdx.x; j <= np;
         j += (long long)gridDim.x * blockDim.x)
        grp_ptr[j] = gscan[part_ptr[j]];
}

// ---- the sliced copy
// What the partitioned kernel reads (one copy per sub-warp width W).  A group
// (at most 32/W rows of one level of one part) is stored as slices of 32
// slots, slot = lane of the warp that solves it, so that every load of an
// entry is coalesced and needs nothing but the group's descriptor
//   { first position, first slice, X, I << 12 | span << 6 | rows }.
// Lane sl of a row holds the row's entries sl, sl + W, ... in fold order, the
// diagonal left out (it comes last and is kept as 1/d(i) by position).  The
// first X slices hold entries of earlier parts (a column is a position, -1: no
// entry), the next I slices entries of the part itself (a column is the offset
// of the unknown in the part; no entry: max_part, a word that reads 0, with
// value 0).  An entry of an earlier part never follows one of the part itself
// in a lane's order, because parts are runs of consecutive rows and rows fold
// farthest dependency first.  span: the most lanes of a row that hold entries
// (at least 1).
__device__ __forceinline__ int part_of_group(const SliceParams& p, int g) {
    int lo = 0, hi = p.nparts - 1;  // last part whose first group is <= g
    while (lo < hi) {
        const int mid = (lo + hi + 1) >> 1;
        if (p.grp_ptr[mid] <= g) lo = mid;
        else hi = mid - 1;
    }
    return lo;
}

// Row of this lane group in fold order: entries t = 0 .. m - 1 at CSR entry
// upper ? q0 - t : q0 + t, the diagonal (if stored) left out.
struct FoldRow {
    int i, q0, m, len;
};
// (stored: a diagonal is known to be)
__device__ __forceinline__ FoldRow fold_row(const SliceParams& p, int k, bool has,
                                            bool stored = false) {
    FoldRow r = {-1, 0, 0, 0};
    if (!has) return r;
    r.i = p.qord[k];
    const int beg = p.ptr[r.i], end = p.ptr[r.i + 1];
    r.len = end - beg;
    r.q0 = p.upper ? end - 1 : beg;
    r.m = r.len;
    if (r.len > 0 && (stored || p.idx[p.upper ? beg : end - 1] == r.i)) --r.m;
    return r;
}

// more[0] and more[1] add up the chunks of every group beyond its first, of earlier
// parts' slots and of the part's own.
template <int W>
__global__ void group_shapes_k(SliceParams p, const int* __restrict__ gstart, int4* grp,
                               int* nslices, unsigned long long* more) {
    constexpr unsigned FULL = 0xffffffffu;
    __shared__ unsigned long long s_more[2];
    if (threadIdx.x < 2) s_more[threadIdx.x] = 0;
    __syncthreads();
    unsigned long long more_x = 0, more_i = 0;
    const int lane = threadIdx.x & 31, grow = lane / W, sl = lane % W;
    const long long warps = ((long long)gridDim.x * blockDim.x) >> 5;
    for (long long g = ((long long)blockIdx.x * blockDim.x + threadIdx.x) >> 5; g < p.ngroups;
         g += warps) {
        const int j = part_of_group(p, (int)g);
        const int r0 = p.part_row[j], r1 = r0 + (p.part_ptr[j + 1] - p.part_ptr[j]);
        const int k0 = gstart[g], cnt = gstart[g + 1] - k0;
        const FoldRow r = fold_row(p, k0 + grow, grow < cnt);
        int ext = 0, all = 0;
        for (int t = sl; t < r.m; t += W, ++all) {
            const int c = p.idx[p.upper ? r.q0 - t : r.q0 + t];
            if (c < r0 || c >= r1) {
                if (ext != all) report(p.status, r.i, kCodeInternal);  // not a prefix
                ++ext;
            }
        }
        const int X = __reduce_max_sync(FULL, ext);
        const int I = __reduce_max_sync(FULL, all - ext);
        int span = W == 1 ? 1 : __reduce_max_sync(FULL, r.m < W ? r.m : W);
        if (span < 1) span = 1;
        if (lane == 0) {
            grp[g] = make_int4(k0, 0, X, (I << 12) | (span << 6) | cnt);
            nslices[g] = X + I;
            if (X > kExtChunk) more_x += (X - 1) / kExtChunk;
            if (I > kOwnChunk) more_i += (I - 1) / kOwnChunk;
        }
    }
    if (lane == 0) {
        if (more_x) atomicAdd(s_more, more_x);
        if (more_i) atomicAdd(s_more + 1, more_i);
    }
    __syncthreads();
    if (threadIdx.x < 2 && s_more[threadIdx.x]) atomicAdd(more + threadIdx.x, s_more[threadIdx.x]);
}

__global__ void group_bases_k(int ngroups, const int* __restrict__ base, int4* grp) {
    for (long long g = (long long)blockIdx.x * blockDim.x + threadIdx.x; g < ngroups;
         g += (long long)gridDim.x * blockDim.x)
        grp[g].y = base[g];
}

// A warp per group writes the group's slices and the 1/d(i) of its rows; checks
// that every entry names an earlier position outside the group.
template <typename T, int W>
__global__ void fill_slices_k(SliceParams p, const int4* __restrict__ grp,
                              const T* __restrict__ vals, int* cols, T* out, T* dinv) {
    const int lane = threadIdx.x & 31, grow = lane / W, sl = lane % W;
    const long long warps = ((long long)gridDim.x * blockDim.x) >> 5;
    for (long long g = ((long long)blockIdx.x * blockDim.x + threadIdx.x) >> 5; g < p.ngroups;
         g += warps) {
        const int j = part_of_group(p, (int)g);
        const int p0 = p.part_ptr[j];
        const int r0 = p.part_row[j], r1 = r0 + (p.part_ptr[j + 1] - p0);
        const int4 d = grp[g];
        const int cnt = d.w & 63, I = d.w >> 12, k = d.x + grow;
        const FoldRow r = fold_row(p, k, grow < cnt);
        T di = T(1);
        if (dinv && r.len > 0) {
            const int qd = p.upper ? r.q0 - r.m : r.q0 + r.m;  // the diagonal folds last
            di = T(1) / vals[p.vmap ? p.vmap[qd] : qd];
            if (sl == 0) dinv[k] = di;
        }
        int t = sl;
        long long at = (long long)d.y * 32 + lane;
        for (int s = 0; s < d.z + I; ++s, at += 32) {
            int c = s < d.z ? -1 : p.max_part;
            T a = T(0);
            if (t < r.m) {
                const int q = p.upper ? r.q0 - t : r.q0 + t;
                const int col = p.idx[q];
                const bool ext = col < r0 || col >= r1;
                if (ext == (s < d.z)) {
                    const T v = vals[p.vmap ? p.vmap[q] : q];
                    a = dinv ? v * di : v;
                    t += W;
                    if (cols) {
                        const int pos = p.qipos[col];
                        if (pos < 0 || pos >= d.x || (!ext && pos < p0) || (ext && pos >= p0))
                            report(p.status, r.i, kCodeInternal);
                        c = ext ? pos : pos - p0;
                    }
                }
            }
            if (cols) cols[at] = c;
            out[at] = a;
        }
        if (t < r.m) report(p.status, r.i, kCodeInternal);  // an entry found no slice
    }
}

// The values alone, into slices that are there: the columns say which slots hold an
// entry, so that a batch of a lane's entries is loaded at once and the next batch's
// columns meanwhile (fill_slices_k looks at one entry after the other to tell which
// slice it belongs to, a load's latency per slice of a long row).  Values of one copy,
// both kernels, us: general 3001 rows FP64, 4 and 8 lanes 141 -> 69 and 94 -> 41, of
// 100001 rows 195 -> 97 and 134 -> 65; band of 40, 4 lanes 49 -> 34.  Where rows take a few
// slices of a large system, the columns are traffic on top (5-point 1024 x 1024 FP32, one
// lane 101 and 141; 7-point 96^3, 4 lanes 74 and 101): those keep fill_slices_k.
template <typename T, int W>
__global__ void refill_slices_k(SliceParams p, const int4* __restrict__ grp,
                                const T* __restrict__ vals, const int* __restrict__ cols, T* out,
                                T* dinv) {
    constexpr int U = 8;
    const int lane = threadIdx.x & 31, grow = lane / W, sl = lane % W;
    const long long warps = ((long long)gridDim.x * blockDim.x) >> 5;
    for (long long g = ((long long)blockIdx.x * blockDim.x + threadIdx.x) >> 5; g < p.ngroups;
         g += warps) {
        const int4 d = grp[g];
        const int cnt = d.w & 63, X = d.z, S = d.z + (d.w >> 12), k = d.x + grow;
        const FoldRow r = fold_row(p, k, grow < cnt, dinv != nullptr);
        T di = T(1);
        if (dinv && r.len > 0) {
            const int qd = p.upper ? r.q0 - r.m : r.q0 + r.m;  // the diagonal folds last
            di = T(1) / vals[p.vmap ? p.vmap[qd] : qd];
            if (sl == 0) dinv[k] = di;
        }
        int t = sl, c[U], cn[U];
        const long long at = (long long)d.y * 32 + lane;
        auto load_cols = [&](int s) {  // the warp's slices s, s + 1, ...
#pragma unroll
            for (int u = 0; u < U; ++u) {
                if (s + u >= S) break;
                cn[u] = cols[at + 32ll * (s + u)];
            }
        };
        load_cols(0);
        for (int s = 0; s < S; s += U) {
            int q[U];
            T v[U];
#pragma unroll
            for (int u = 0; u < U; ++u) {
                if (s + u >= S) break;
                c[u] = cn[u];
            }
            load_cols(s + U);
#pragma unroll
            for (int u = 0; u < U; ++u) {
                if (s + u >= S) break;
                q[u] = -1;
                if (c[u] != (s + u < X ? -1 : p.max_part)) {
                    q[u] = p.upper ? r.q0 - t : r.q0 + t;
                    t += W;
                }
            }
            if (p.vmap) {
#pragma unroll
                for (int u = 0; u < U; ++u) {
                    if (s + u >= S) break;
                    if (q[u] >= 0) q[u] = p.vmap[q[u]];
                }
            }
#pragma unroll
            for (int u = 0; u < U; ++u) {
                if (s + u >= S) break;
                v[u] = q[u] >= 0 ? vals[q[u]] : T(0);
            }
#pragma unroll
            for (int u = 0; u < U; ++u) {
                if (s + u >= S) break;  // an FP64 multiply takes 64 cycles, needed or not
                const T a = dinv ? v[u] * di : v[u];
                if (q[u] >= 0) out[at + 32ll * (s + u)] = a;
            }
        }
    }
}

#define SPTRSV_LAUNCH(kernel, m, ...)                        \
    do {                                                     \
        kernel<<<grid_for(m), 256, 0, s>>>(__VA_ARGS__);     \
        cudaError_t _e = cudaGetLastError();                 \
        if (_e != cudaSuccess) return _e;                    \
    } while (0)

cudaError_t launch_part_spans(int n, const int* ptr, const int* idx, bool upper, int* diff,
                              cudaStream_t s) {
    if (n <= 0) return cudaSuccess;
    SPTRSV_LAUNCH(part_spans_k, n, n, ptr, idx, upper ? 1 : 0, diff);
    return cudaSuccess;
}

cudaError_t launch_block_flags(int n, const int* cover, int* flag, cudaStream_t s) {
    if (n <= 0) return cudaSuccess;
    SPTRSV_LAUNCH(block_flags_k, n, n, cover, flag);
    return cudaSuccess;
}

cudaError_t launch_flag_scatter(int n, const int* flag, const int* scan, int* start,
                                cudaStream_t s) {
    SPTRSV_LAUNCH(flag_scatter_k, n, n, flag, scan, start);
    return cudaSuccess;
}

cudaError_t launch_block_depth(int n, bool upper, const int* lev, const int* bscan, int* depth,
                               cudaStream_t s) {
    if (n <= 0) return cudaSuccess;
    SPTRSV_LAUNCH(block_depth_k, n, n, upper ? 1 : 0, lev, bscan, depth);
    return cudaSuccess;
}

cudaError_t launch_part_flags(int n, int S, const int* bscan, const int* bstart, int* flag,
                              cudaStream_t s) {
    if (n <= 0) return cudaSuccess;
    SPTRSV_LAUNCH(part_flags_k, n, n, S, bscan, bstart, flag);
    return cudaSuccess;
}

cudaError_t launch_part_depth_keys(int np, int maxdepth, const int* pstart, const int* bscan,
                                   const int* depth, int* key, cudaStream_t s) {
    if (np <= 0) return cudaSuccess;
    SPTRSV_LAUNCH(part_depth_keys_k, np, np, maxdepth, pstart, bscan, depth, key);
    return cudaSuccess;
}

cudaError_t launch_part_piece(int np, const int* pstart, const int* bscan, const int* bstart,
                              const int* pscan, int* piece, cudaStream_t s) {
    if (np <= 0) return cudaSuccess;
    SPTRSV_LAUNCH(part_piece_k, np, np, pstart, bscan, bstart, pscan, piece);
    return cudaSuccess;
}

cudaError_t launch_part_alap_keys(int np, int maxdepth, const int* pstart, const int* bscan,
                                  const int* bstart, const int* pscan, const int* depth,
                                  const int* piece, int* key, cudaStream_t s) {
    if (np <= 0) return cudaSuccess;
    SPTRSV_LAUNCH(part_alap_keys_k, np, np, maxdepth, pstart, bscan, bstart, pscan, depth, piece,
                  key);
    return cudaSuccess;
}

cudaError_t launch_part_sizes(int n, int np, bool upper, const int* horder, const int* pstart,
                              int* size, int* row, int* maxsize, cudaStream_t s) {
    if (np <= 0) return cudaSuccess;
    SPTRSV_LAUNCH(part_sizes_k, np, n, np, upper ? 1 : 0, horder, pstart, size, row, maxsize);
    return cudaSuccess;
}

cudaError_t launch_row_part_keys(int n, const int* jlev, bool upper, const int* pscan,
                                 const int* prank, int* key, cudaStream_t s) {
    if (n <= 0) return cudaSuccess;
    SPTRSV_LAUNCH(row_part_keys_k, n, n, jlev, upper ? 1 : 0, pscan, prank, key);
    return cudaSuccess;
}

cudaError_t launch_run_flags(int n, const int* qord, const int* lev, int* flag, cudaStream_t s) {
    if (n <= 0) return cudaSuccess;
    SPTRSV_LAUNCH(run_flags_k, n, n, qord, lev, flag);
    return cudaSuccess;
}

cudaError_t launch_part_flag_starts(int np, const int* part_ptr, int* flag, cudaStream_t s) {
    if (np <= 0) return cudaSuccess;
    SPTRSV_LAUNCH(part_flag_starts_k, np, np, part_ptr, flag);
    return cudaSuccess;
}

cudaError_t launch_group_flags(int n, int R, const int* rscan, const int* rstart, int* flag,
                               cudaStream_t s) {
    if (n <= 0) return cudaSuccess;
    SPTRSV_LAUNCH(group_flags_k, n, n, R, rscan, rstart, flag);
    return cudaSuccess;
}

cudaError_t launch_part_groups(int np, const int* part_ptr, const int* gscan, int* grp_ptr,
                               cudaStream_t s) {
    SPTRSV_LAUNCH(part_groups_k, (long long)np + 1, np, part_ptr, gscan, grp_ptr);
    return cudaSuccess;
}

static int warps_grid(long long warps) {  // 8 warps a block
    const long long g = (warps + 7) / 8;
    return g < 1 ? 1 : (g > 16384 ? 16384 : (int)g);
}

cudaError_t launch_group_shapes(const SliceParams& p, int lanes, const int* gstart, int4* grp,
                                int* nslices, unsigned long long* more, cudaStream_t s) {
    const int g = warps_grid(p.ngroups);
#define SPTRSV_SHAPES(W) group_shapes_k<W><<<g, 256, 0, s>>>(p, gstart, grp, nslices, more)
    switch (lanes) {
        case 1: SPTRSV_SHAPES(1); break;
        case 2: SPTRSV_SHAPES(2); break;
        case 4: SPTRSV_SHAPES(4); break;
        case 8: SPTRSV_SHAPES(8); break;
        case 16: SPTRSV_SHAPES(16); break;
        case 32: SPTRSV_SHAPES(32); break;
        default: return cudaErrorInvalidValue;
    }
#undef SPTRSV_SHAPES
    return cudaGetLastError();
}

cudaError_t launch_group_bases(int ngroups, const int* base, int4* grp, cudaStream_t s) {
    SPTRSV_LAUNCH(group_bases_k, ngroups, ngroups, base, grp);
    return cudaSuccess;
}

template <typename T>
static cudaError_t fill_t(const SliceParams& p, int lanes, const int4* grp, const void* vals,
                          int* cols, void* out, void* dinv, cudaStream_t s) {
    const int g = warps_grid(p.ngroups);
#define SPTRSV_FILL(W) \
    fill_slices_k<T, W><<<g, 256, 0, s>>>(p, grp, (const T*)vals, cols, (T*)out, (T*)dinv)
    switch (lanes) {
        case 1: SPTRSV_FILL(1); break;
        case 2: SPTRSV_FILL(2); break;
        case 4: SPTRSV_FILL(4); break;
        case 8: SPTRSV_FILL(8); break;
        case 16: SPTRSV_FILL(16); break;
        case 32: SPTRSV_FILL(32); break;
        default: return cudaErrorInvalidValue;
    }
#undef SPTRSV_FILL
    return cudaGetLastError();
}

cudaError_t launch_fill_slices(bool f64, const SliceParams& p, int lanes, const int4* grp,
                               const void* vals, int* cols, void* out, void* dinv,
                               cudaStream_t s) {
    return f64 ? fill_t<double>(p, lanes, grp, vals, cols, out, dinv, s)
               : fill_t<float>(p, lanes, grp, vals, cols, out, dinv, s);
}

template <typename T>
static cudaError_t refill_t(const SliceParams& p, int lanes, const int4* grp, const void* vals,
                            const int* cols, void* out, void* dinv, cudaStream_t s) {
    const int g = warps_grid(p.ngroups);
#define SPTRSV_REFILL(W) \
    refill_slices_k<T, W><<<g, 256, 0, s>>>(p, grp, (const T*)vals, cols, (T*)out, (T*)dinv)
    switch (lanes) {
        case 1: SPTRSV_REFILL(1); break;
        case 2: SPTRSV_REFILL(2); break;
        case 4: SPTRSV_REFILL(4); break;
        case 8: SPTRSV_REFILL(8); break;
        case 16: SPTRSV_REFILL(16); break;
        case 32: SPTRSV_REFILL(32); break;
        default: return cudaErrorInvalidValue;
    }
#undef SPTRSV_REFILL
    return cudaGetLastError();
}

cudaError_t launch_refill_slices(bool f64, const SliceParams& p, int lanes, int longest,
                                 const int4* grp, const void* vals, const int* cols, void* out,
                                 void* dinv, cudaStream_t s) {
    if (lanes <= 8 && longest <= 4 * lanes && p.n > 300000)
        return launch_fill_slices(f64, p, lanes, grp, vals, nullptr, out, dinv, s);
    return f64 ? refill_t<double>(p, lanes, grp, vals, cols, out, dinv, s)
               : refill_t<float>(p, lanes, grp, vals, cols, out, dinv, s);
}

#undef SPTRSV_LAUNCH

}  // namespace sptrsv
