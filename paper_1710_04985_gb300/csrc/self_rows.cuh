// What the single-RHS kernels of the in-place and level-ordered forms do with a row
// of a ticket (solve_self.cu, solve_cluster.cu): 32 / W rows per warp, W lanes each.
#pragma once
#include "cursor.h"
#include "internal.h"

namespace sptrsv {
namespace {

// Entries a lane holds at once: groups of 16 and 32 lanes hold an average row in one
// or two, and every further slot costs its instructions in each polling round
// (general 150001 rows, 32 lanes 4811 us with four, 4670 with two).
template <int W>
struct ChunkOf {
    static constexpr int E = W >= 16 ? 2 : kChunk;
    static_assert(cursor_ahead(W, E) <= kCursorAhead, "entry index");
};

__device__ __forceinline__ double lds_relaxed(const double* p) { return *(const volatile double*)p; }
__device__ __forceinline__ float lds_relaxed(const float* p) { return *(const volatile float*)p; }

// One row of a ticket as its lanes see it.
template <typename T>
struct Row {
    int i, beg, end, lev;
    long long k;
    bool has;
    T dinv, sum;
    double xbase;  // refinement: the solution the row's value is added to
};

template <typename T, int W, bool PERM>
__device__ __forceinline__ Row<T> take_row(const SolveParams& p, long long k) {
    Row<T> r;
    r.k = k;
    r.has = k < p.n;
    r.i = r.beg = r.end = r.lev = 0;
    r.dinv = T(1);
    r.sum = T(0);
    r.xbase = 0.0;
    if (r.has) {
        r.i = p.jlev[k];
        r.beg = p.ptr[PERM ? k : r.i];
        r.end = p.ptr[(PERM ? k : r.i) + 1];
        if (W < 32) r.lev = p.lev[r.i];
    }
    return r;
}

// Everything of a row that does not depend on x: SLFR computes 1/d(i) up front
// too; the row is scaled by it, so x(i) = b(i)/d(i) - sum of (a_ij/d(i)) x(j) and
// only the FMA fold and the lane reduction remain once the last value is there.
template <typename T, int W, bool MAP>
__device__ __forceinline__ void start_row(const SolveParams& p, Row<T>& r, int sl) {
    if (r.has && sl == 0) {
        const T* __restrict__ vals = (const T*)p.vals;
        if (!p.unit) {
            const int q = p.diag_first ? r.beg : r.end - 1;
            const T d = vals[MAP ? p.vmap[q] : q];
            r.dinv = p.prescaled ? d : T(1) / d;  // a pre-scaled copy holds 1/d(i)
        }
        r.sum = ((const T*)p.b)[(long long)r.i * p.ldb];
        if (!p.unit) r.sum *= r.dinv;
        r.xbase = accumulate_base(p, r.i, 0);
    }
    if (W > 1 && !p.unit && !p.prescaled)
        r.dinv = __shfl_sync(0xffffffffu, r.dinv, (threadIdx.x & 31) / W * W);
}

// Entries q0, q0 + W, ... of a row in fold order: the unknown to wait for (-1:
// none, the diagonal included) and the scaled value (0).
template <typename T, int W, bool MAP, bool PERM, int E>
__device__ __forceinline__ void load_entries(const SolveParams& p, const Row<T>& r, int q0,
                                             int (&c)[E], T (&a)[E]) {
    const T* __restrict__ vals = (const T*)p.vals;
    // every form folds farthest dependency first: a lower row in storage order,
    // an upper row from its last entry back (the copies already store it so)
    const bool rvs = !PERM && p.diag_first;
    const int self = PERM ? (int)r.k : r.i;
#pragma unroll
    for (int e = 0; e < E; ++e) {
        const int q = q0 + e * W;
        c[e] = -1;
        a[e] = T(0);
        if (q < r.end) {
            const int pq = rvs ? r.beg + r.end - 1 - q : q;
            c[e] = p.idx[pq];
            a[e] = vals[MAP ? p.vmap[pq] : pq];
        }
    }
#pragma unroll
    for (int e = 0; e < E; ++e)
        if (c[e] == self) {
            c[e] = -1;
            a[e] = T(0);
        }
}

// Scales the loaded values of a row that is not pre-scaled (slots that no lane
// uses are branched around: an FP64 multiply takes 64 cycles).
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

// group_sum_span (the same sums in the same order) with at most three branches
// instead of one per level of the butterfly.
template <int OFF, typename T>
__device__ __forceinline__ T sum_from(T v) {
    v += __shfl_xor_sync(0xffffffffu, v, OFF);
    if constexpr (OFF > 1) v = sum_from<OFF / 2>(v);
    return v;
}
template <int W, typename T>
__device__ __forceinline__ T row_sum(T v, int span) {
    if constexpr (W == 1) return v;
    if constexpr (W == 2) return span > 1 ? sum_from<1>(v) : v;
    if constexpr (W >= 4) {
        if (span > 4) {
            if constexpr (W >= 32)
                if (span > 16) return sum_from<16>(v);
            if constexpr (W >= 16)
                if (span > 8) return sum_from<8>(v);
            if constexpr (W >= 8) return sum_from<4>(v);
        }
        if (span > 2) return sum_from<2>(v);
        return span > 1 ? sum_from<1>(v) : v;
    }
}

}  // namespace
}  // namespace sptrsv
