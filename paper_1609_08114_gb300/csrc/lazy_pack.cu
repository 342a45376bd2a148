// lazy_pack.cu -- the pivots kept, FP32, the several-LPs-per-warp kernel's arithmetic (m, n <= 31).
#include "simplex_lazy.cuh"

namespace lpb {

namespace {
// Warps per LP, rows and columns per thread, CTAs per SM at least: 32 (64 registers, no
// spills) hide the most latency (100,000 x 28: 353 us with 16, 289 with 24, 249 with 32).
const LazyConfig kTable[] = {lazy_config<float, 1, 1, 32, true, kPacked>()};
}  // namespace

cudaError_t lazy_occupancy_pack(const LazyShape &q, int dtype, int *ctas, int *threads, LazyLayout *lay) {
  return lazy_occ<float>(kTable, q, dtype, ctas, threads, lay);
}

cudaError_t launch_lazy_pack(const TableauParams &p, const LazyLayout &lay, int grid, cudaStream_t s) {
  return lazy_launch(kTable, p, lay, grid, s);
}

}  // namespace lpb
