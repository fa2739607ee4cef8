// Partitioned solve, FP32 instances.
#include "solve_partitioned.cuh"

namespace sptrsv {

template cudaError_t part_any<float>(int, const SolveParams&, int, int, int, cudaStream_t, int,
                                   int*);

}  // namespace sptrsv
