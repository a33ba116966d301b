// Factored stages for any M (see qb_factor.cuh).
#include "qb_factor.cuh"

namespace qb {
int fac_launch_any(const Tables& t, const DfArgs& a, int mode, int B, bool bil, int shape, cudaStream_t st, int* grid) {
  // the creation pairs unrolled (us a stage): M = 6, 593,775 kets 56.2 / 48.8; M = 8, 1.56M kets 183 / 150
  switch (t.M) {
    case 6: return fac_launch<6, 0>(t, a, mode, B, bil, shape, st, grid);
    case 8: return fac_launch<8, 0>(t, a, mode, B, bil, shape, st, grid);
    default: return fac_launch<0, 0>(t, a, mode, B, bil, shape, st, grid);
  }
}
}  // namespace qb
