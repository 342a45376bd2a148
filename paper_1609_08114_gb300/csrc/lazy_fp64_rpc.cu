// lazy_fp64_rpc.cu -- the pivots kept, FP64 tableau, random entering rule.
#include "simplex_lazy.cuh"

namespace lpb {

namespace {
// Warps per LP, rows and columns per thread, CTAs per SM at least.
const LazyConfig kTable[] = {
    lazy_config<double, 1, 1, 16, true, kRandom>(),
    lazy_config<double, 1, 2, 16, true, kRandom>(),
    lazy_config<double, 1, 4, 12, true, kRandom>(),
    lazy_config<double, 4, 2, 4, true, kRandom>(),
    lazy_config<double, 4, 3, 3, true, kRandom>(),
    lazy_config<double, 8, 2, 2, true, kRandom>(),
    lazy_config<double, 8, 4, 1, true, kRandom>(),
};
}  // namespace

cudaError_t lazy_occupancy_fp64_rpc(const LazyShape &q, int dtype, int *ctas, int *threads, LazyLayout *lay) {
  return lazy_occ<double>(kTable, q, dtype, ctas, threads, lay);
}

cudaError_t launch_lazy_fp64_rpc(const TableauParams &p, const LazyLayout &lay, int grid, cudaStream_t s) {
  return lazy_launch(kTable, p, lay, grid, s);
}

}  // namespace lpb
