// Batched ensemble step of the 3-D elastic family with the mixed-precision Picard predictor, orders 1-5 (one
// persistent launch per phase for all runs, or one launch for whole steps).
#include "kernels_ensemble.cuh"

namespace ader {

cudaError_t ens_step_elastic3_mixed(const StepArgs* R, const EnsTable& E, const Tables& T,
                                   const TablesF& F, int order, cudaStream_t s) {
  switch (order) {
    case 1: return ens_step_n<1, true, true>(R, E, T, F, E.pblocks, s);
    case 2: return ens_step_n<2, true, true>(R, E, T, F, E.pblocks, s);
    case 3: return ens_step_n<3, true, true>(R, E, T, F, E.pblocks, s);
    case 4: return ens_step_n<4, true, true>(R, E, T, F, E.pblocks, s);
    case 5: return ens_step_n<5, true, true>(R, E, T, F, E.pblocks, s);
  }
  return cudaErrorInvalidValue;
}

cudaError_t ens_fused_elastic3_mixed(const StepArgs* R, const EnsTable& E, const Tables& T, const TablesF& F, int order,
               int steps, void* bar, long long limit, int bps, cudaStream_t s) {
  GridBar* b = static_cast<GridBar*>(bar);
  switch (order) {
    case 1: return ens_fused_n<1, true>(R, E, T, F, steps, b, limit, bps, s);
    case 2: return ens_fused_n<2, true>(R, E, T, F, steps, b, limit, bps, s);
    case 3: return ens_fused_n<3, true>(R, E, T, F, steps, b, limit, bps, s);
    case 4: return ens_fused_n<4, true>(R, E, T, F, steps, b, limit, bps, s);
    case 5: return ens_fused_n<5, true>(R, E, T, F, steps, b, limit, bps, s);
  }
  return cudaErrorInvalidValue;
}

}  // namespace ader
