// lazy_fp64.cu -- the pivots kept, FP64 tableau.
#include "simplex_lazy.cuh"

namespace lpb {

namespace {
// Warps per LP, rows and columns per thread, CTAs per SM at least.
const LazyConfig kTable[] = {
    lazy_config<double, 1, 1, 16, true>(),
    lazy_config<double, 1, 2, 16, true>(),
    lazy_config<double, 1, 4, 12, true>(),
    lazy_config<double, 4, 2, 4, true>(),
    lazy_config<double, 4, 3, 3, true>(),
    lazy_config<double, 8, 2, 2, true>(),
    lazy_config<double, 8, 4, 1, true>(),
};
}  // namespace

cudaError_t lazy_occupancy_fp64(const LazyShape &q, int dtype, int *ctas, int *threads, LazyLayout *lay) {
  return lazy_occ<double>(kTable, q, dtype, ctas, threads, lay);
}

cudaError_t launch_lazy_fp64(const TableauParams &p, const LazyLayout &lay, int grid, cudaStream_t s) {
  return lazy_launch(kTable, p, lay, grid, s);
}

}  // namespace lpb
