// Stage-kernel specialisation for M = 5 modes with 2 partners a pair (see qb_block.cuh).
#include "qb_stage.cuh"

namespace qb {
int stage_launch_m5(const Tables& t, const DfArgs& a, int mode, int B, bool bil, int shape, cudaStream_t st, int* grid) {
  return blk_launch_kind<5, true>(t, a, mode, B, bil, shape, st, grid);
}
int resident_launch_m5(const Tables& t, const ResArgs& r, int threads, cudaStream_t st) {
  return resident_reg_launch<5>(t, r, threads, st);
}
int grid_launch_m5(const Tables& t, const ResArgs& r, cudaStream_t st) { return grid_reg_launch<5>(t, r, st); }
}  // namespace qb
