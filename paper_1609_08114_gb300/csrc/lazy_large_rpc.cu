// lazy_large_rpc.cu -- the pivots kept, FP32, the tableau kernel's arithmetic (m or n above 127), random entering rule.
#include "simplex_lazy.cuh"

namespace lpb {

namespace {
// Warps per LP, rows and columns per thread, CTAs per SM at least.
const LazyConfig kTable[] = {
    lazy_config<float, 4, 2, 4, true, kRandom>(),
    lazy_config<float, 8, 2, 2, true, kRandom>(),
    lazy_config<float, 8, 4, 1, true, kRandom>(),
};
}  // namespace

cudaError_t lazy_occupancy_large_rpc(const LazyShape &q, int dtype, int *ctas, int *threads, LazyLayout *lay) {
  return lazy_occ<float>(kTable, q, dtype, ctas, threads, lay);
}

cudaError_t launch_lazy_large_rpc(const TableauParams &p, const LazyLayout &lay, int grid, cudaStream_t s) {
  return lazy_launch(kTable, p, lay, grid, s);
}

}  // namespace lpb
