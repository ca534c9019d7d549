// Batched ensemble step of the 3-D elastic family with the Cauchy-Kowalevski predictor (FP64 and
// mixed precision), orders 4 and 5 (one cell per block): one launch per phase for all runs, as for
// the Picard predictor.  The predictor's blocks take the concatenated cells of the runs (one each)
// and call the per-context kernels' block function with the cell's run; the Riemann solver and
// the corrector are the ensemble's shared persistent kernels.  For these runs the per-run
// launches on forked streams are faster (74.9 against 87.3 ms per step of the 16-run ensemble);
// the autotuner chooses between them.
#include "kernels_ensemble.cuh"

namespace ader {

// prec: 0 FP64, 1 mixed; orders 4 and 5
cudaError_t ens_step_ck_elastic3(const StepArgs* R, const EnsTable& E, const Tables& T,
                                 const TablesF& F, int prec, int order, cudaStream_t s) {
  if (prec == 1) {
    if (order == 4) return ens_step_n<4, true, false>(R, E, T, F, E.blk0[E.nr], s);
    if (order == 5) return ens_step_n<5, true, false>(R, E, T, F, E.blk0[E.nr], s);
  } else if (prec == 0) {
    if (order == 4) return ens_step_n<4, false, false>(R, E, T, F, E.blk0[E.nr], s);
    if (order == 5) return ens_step_n<5, false, false>(R, E, T, F, E.blk0[E.nr], s);
  }
  return cudaErrorInvalidValue;
}

}  // namespace ader
