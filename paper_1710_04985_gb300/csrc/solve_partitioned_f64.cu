// Partitioned solve, FP64 instances and the launch interface.
#include "solve_partitioned.cuh"

namespace sptrsv {

template cudaError_t part_any<double>(int, const SolveParams&, int, int, int, cudaStream_t, int,
                                   int*);
extern template cudaError_t part_any<float>(int, const SolveParams&, int, int, int, cudaStream_t,
                                            int, int*);

cudaError_t launch_part_k1(bool f64, int lanes, const SolveParams& p, int grid, int block,
                           int cluster, cudaStream_t s) {
    return f64 ? part_any<double>(lanes, p, grid, block, cluster, s, 0, nullptr)
               : part_any<float>(lanes, p, grid, block, cluster, s, 0, nullptr);
}

int part_resident_blocks(bool f64, int lanes, int cluster, int block, int part_rows, int num_sms) {
    int nb = 0;
    SolveParams p = {};
    p.max_part = part_rows;
    const cudaError_t e = f64 ? part_any<double>(lanes, p, 0, block, cluster, nullptr, num_sms, &nb)
                              : part_any<float>(lanes, p, 0, block, cluster, nullptr, num_sms, &nb);
    return e == cudaSuccess ? nb : 0;
}

}  // namespace sptrsv
