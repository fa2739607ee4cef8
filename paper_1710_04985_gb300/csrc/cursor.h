// Index arithmetic of the solve kernels at the limit of their int indices (n and nnz
// up to SPTRSV_MAX_SIZE, 256 below 2^31).  Plain C++, so that it can be checked on the
// host with the limit's own numbers.
#pragma once

#ifdef __CUDACC__
#define SPTRSV_HD __host__ __device__ __forceinline__
#else
#define SPTRSV_HD inline
#endif

namespace sptrsv {

// A lane's cursor over the entries [.., end) of its row, `step` further on.  The lanes
// of a warp go through chunks together, for as long as its longest row lasts: the
// cursor of a lane whose row has ended stops 32 past the end instead of running on by the
// length of its neighbour's row.  (Stepping only lanes that are inside their row is the
// same, but cost the 27-point adjoint with one lane per row 10 %.)
SPTRSV_HD int advance(int cursor, int step, int end) {
    const int next = cursor + step, most = end + 32;
    return next < most ? next : most;
}

// An entry index that a kernel forms is at most this far past the end of its row (the
// kernels assert it for their chunks): it stays an int at the limit.
constexpr int kCursorAhead = 255;

// The furthest for chunks of `slots` slots of `lanes` entries: a cursor that has stopped,
// the chunk after its own, the last slot of it.
constexpr int cursor_ahead(int lanes, int slots) {
    return 32 + lanes * slots + lanes * (slots - 1);
}

// The start of the window of `rows` rows after the one at `base`, or n after the last
// (base + rows may be past the largest int).
SPTRSV_HD int next_window(int base, int rows, int n) {
    return n - base > rows ? base + rows : n;
}

}  // namespace sptrsv
