// Step kernels of small grids: 8 x 8-cell tiles in 2D (variant 9: every precision, both expansions) and 30-cell
// tiles in 1D (variant 3).  A grid of a few thousand cells is bound by the latency of one CTA, and what
// shortens it is fewer cells per CTA on more of the SMs; the rule is in tile_candidates.
#include "gks_dispatch.h"
#include "gks_step.cuh"

namespace gks {

cudaError_t prepare_step_small() {
  cudaError_t e = cudaSuccess, r;
#define GKS_PREP(P)                                                       \
  if ((r = prepare_step<1, P, false, 3>()) != cudaSuccess) e = r;         \
  if ((r = prepare_step<2, P, false, 9>()) != cudaSuccess) e = r;         \
  if ((r = prepare_step<2, P, true, 9>()) != cudaSuccess) e = r;
  GKS_PREP(PREC_F64)
  GKS_PREP(PREC_F32)
  GKS_PREP(PREC_F32D)
#undef GKS_PREP
  return e;
}

template <int PREC>
void launch_small(int D, bool multid, const StepArgs& A, int nblocks, cudaStream_t s) {
  if (D == 1)
    launch_step<1, PREC, false, 3>(A, nblocks, s);
  else if (multid)
    launch_step<2, PREC, true, 9>(A, nblocks, s);
  else
    launch_step<2, PREC, false, 9>(A, nblocks, s);
}

void launch_step_small(int D, int prec, bool multid, const StepArgs& A, int nblocks, cudaStream_t s) {
  if (prec == PREC_F64)
    launch_small<PREC_F64>(D, multid, A, nblocks, s);
  else if (prec == PREC_F32)
    launch_small<PREC_F32>(D, multid, A, nblocks, s);
  else
    launch_small<PREC_F32D>(D, multid, A, nblocks, s);
}

}  // namespace gks
