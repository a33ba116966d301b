// Stage-kernel specialisation for M = 11 modes with 5 partners a pair (see qb_block.cuh).
#include "qb_stage.cuh"

namespace qb {
int stage_launch_m11(const Tables& t, const DfArgs& a, int mode, int B, bool bil, int shape, cudaStream_t st, int* grid) {
  return blk_launch_kind<11, true>(t, a, mode, B, bil, shape, st, grid);
}
int resident_launch_m11(const Tables& t, const ResArgs& r, int threads, cudaStream_t st) {
  return resident_sparse(t) ? resident_launch_k<0, 5, false, true>(t, r, threads, st)
                            : resident_launch_k<11, 5, false, false>(t, r, threads, st);
}
}  // namespace qb
