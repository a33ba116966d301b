// Stage-kernel specialisation for M = 9 modes with 4 partners a pair (see qb_block.cuh).
#include "qb_stage.cuh"

namespace qb {
int stage_launch_m9(const Tables& t, const DfArgs& a, int mode, int B, bool bil, int shape, cudaStream_t st, int* grid) {
  return blk_launch_kind<9, true>(t, a, mode, B, bil, shape, st, grid);
}
int resident_launch_m9(const Tables& t, const ResArgs& r, int threads, cudaStream_t st) {
  return resident_sparse(t) ? resident_launch_k<0, 4, false, true>(t, r, threads, st)
                            : resident_reg_launch<9>(t, r, threads, st);
}
}  // namespace qb
