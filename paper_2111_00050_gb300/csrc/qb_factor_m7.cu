// Factored stages for M = 7 modes (see qb_factor.cuh).
#include "qb_factor.cuh"

namespace qb {
int fac_launch_m7(const Tables& t, const DfArgs& a, int mode, int B, bool bil, int shape, cudaStream_t st, int* grid) {
  if (t.fa_nt == 0) return fac_launch<7, 0>(t, a, mode, B, bil, shape, st, grid);  // exact momentum
  return fac_launch<7, 4>(t, a, mode, B, bil, shape, st, grid);
}
}  // namespace qb
