// lazy_small_rpc.cu -- the pivots kept, FP32, the register kernel's arithmetic (m, n <= 64), random entering rule.
#include "simplex_lazy.cuh"

namespace lpb {

namespace {
// Warps per LP, rows and columns per thread, CTAs per SM at least.  (Above 64 rows or
// columns the planner leaves this rule to the other kernels.)
const LazyConfig kTable[] = {
    lazy_config<float, 1, 1, 16, false, kRandom>(),
    lazy_config<float, 1, 2, 16, false, kRandom>(),
};
}  // namespace

cudaError_t lazy_occupancy_small_rpc(const LazyShape &q, int dtype, int *ctas, int *threads, LazyLayout *lay) {
  return lazy_occ<float>(kTable, q, dtype, ctas, threads, lay);
}

cudaError_t launch_lazy_small_rpc(const TableauParams &p, const LazyLayout &lay, int grid, cudaStream_t s) {
  return lazy_launch(kTable, p, lay, grid, s);
}

}  // namespace lpb
