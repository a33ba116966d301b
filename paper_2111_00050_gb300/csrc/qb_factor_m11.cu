// Factored stages for M = 11 modes (see qb_factor.cuh).
#include "qb_factor.cuh"

namespace qb {
int fac_launch_m11(const Tables& t, const DfArgs& a, int mode, int B, bool bil, int shape, cudaStream_t st, int* grid) {
  if (t.fa_nt == 0) return fac_launch<11, 0>(t, a, mode, B, bil, shape, st, grid);  // exact momentum
  return fac_launch<11, 6>(t, a, mode, B, bil, shape, st, grid);
}
}  // namespace qb
