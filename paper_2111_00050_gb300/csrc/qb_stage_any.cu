// Stage kernels for any M, exact momentum and complex couplings (see qb_block.cuh).
#include "qb_stage.cuh"

namespace qb {
// The RK4 stage of one state with the mode count known: the occupations in the words they
// need, their unpacking and the epilogue unrolled.  Against the kernel for any M (us a stage, the
// same bit for bit): M = 4, 1.66M kets 106 / 101; M = 6, 230,230 kets, complex 48.7 / 46.6, real 35.2 /
// 34.1; M = 8, 1.56M kets 325 / 313; exact momentum, M = 7, 1.56M kets 176 / 171.
template <bool CPLX>
static int stage_of(const Tables& t, const DfArgs& a, int mode, int shape, cudaStream_t st, int* grid) {
  switch (t.M) {
    case 4: return blk_launch<4, false, 1, CPLX, KIND_STAGE>(t, a, mode, shape, st, grid);
    case 5: return blk_launch<5, false, 1, CPLX, KIND_STAGE>(t, a, mode, shape, st, grid);
    case 6: return blk_launch<6, false, 1, CPLX, KIND_STAGE>(t, a, mode, shape, st, grid);
    case 7: return blk_launch<7, false, 1, CPLX, KIND_STAGE>(t, a, mode, shape, st, grid);
    case 8: return blk_launch<8, false, 1, CPLX, KIND_STAGE>(t, a, mode, shape, st, grid);
    default: return blk_launch<0, false, 1, CPLX, KIND_STAGE>(t, a, mode, shape, st, grid);
  }
}
int stage_launch_any(const Tables& t, const DfArgs& a, int mode, int B, bool cplx, bool bil, int shape, cudaStream_t st,
                     int* grid) {
  if (!cplx && B == 1 && !bil && mode >= 0 && mode < 4) return stage_of<false>(t, a, mode, shape, st, grid);
  if (!cplx) return blk_launch_kind<0, false>(t, a, mode, B, bil, shape, st, grid);
  if (B != 1) return fail(QB_EUNSUPPORTED, "batched sweeps need a real coupling");
  if (mode < 0 || mode > 4) return fail(QB_EINTERNAL, "bad stage mode");
  if (mode == 4) return blk_launch<0, false, 1, true, KIND_DOT>(t, a, mode, shape, st, grid);
  if (bil) return blk_launch<0, false, 1, true, KIND_BIL>(t, a, mode, shape, st, grid);
  return stage_of<true>(t, a, mode, shape, st, grid);
}
int resident_launch_any(const Tables& t, const ResArgs& r, int threads, cudaStream_t st) {
  if (resident_sparse(t))
    return t.is_complex ? resident_launch_k<0, 0, true, true>(t, r, threads, st)
                        : resident_launch_k<0, 0, false, true>(t, r, threads, st);
  return t.is_complex ? resident_launch_k<0, 0, true, false>(t, r, threads, st)
                      : resident_launch_k<0, 0, false, false>(t, r, threads, st);
}
}  // namespace qb
