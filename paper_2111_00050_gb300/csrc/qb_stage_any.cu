// Stage kernels for any M, exact momentum and complex couplings (see qb_block.cuh).
#include "qb_stage.cuh"

namespace qb {
int stage_launch_any(const Tables& t, const DfArgs& a, int mode, int B, bool cplx, bool bil, int shape, cudaStream_t st,
                     int* grid) {
  if (!cplx) return blk_launch_kind<0, false>(t, a, mode, B, bil, shape, st, grid);
  if (B != 1) return fail(QB_EUNSUPPORTED, "batched sweeps need a real coupling");
  if (mode < 0 || mode > 4) return fail(QB_EINTERNAL, "bad stage mode");
  if (mode == 4) return blk_launch<0, false, 1, true, KIND_DOT>(t, a, mode, shape, st, grid);
  if (bil) return blk_launch<0, false, 1, true, KIND_BIL>(t, a, mode, shape, st, grid);
  return blk_launch<0, false, 1, true, KIND_STAGE>(t, a, mode, shape, st, grid);
}
int resident_launch_any(const Tables& t, const ResArgs& r, int threads, cudaStream_t st) {
  return t.is_complex ? resident_launch_k<0, false, true>(t, r, threads, st)
                      : resident_launch_k<0, false, false>(t, r, threads, st);
}
}  // namespace qb
