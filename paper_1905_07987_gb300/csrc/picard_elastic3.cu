// Picard predictor of the 3-D elastic family, orders 1-6, FP64 and mixed precision: the linear
// system's iterates in their polynomial form (kernels_ck.cuh).
#include "kernels_ck_fx.cuh"

namespace ader {

cudaError_t predictor_picard_elastic3(const StepArgs& a, const Tables& t, const TablesF& f,
                                      int prec, cudaStream_t s) {
  if (!a.lin) return cudaErrorInvalidValue;
  if (prec == 1) {
    switch (a.g.order) {
      case 1: return launch_predictor_elastic_mixed_n<1, true>(a, t, f, s);
      case 2: return launch_predictor_elastic_mixed_n<2, true>(a, t, f, s);
      case 3: return launch_predictor_elastic_mixed_n<3, true>(a, t, f, s);
      case 4: return launch_predictor_elastic_mixed_n<4, true>(a, t, f, s);
      case 5: return launch_predictor_elastic_mixed_n<5, true>(a, t, f, s);
      case 6: return launch_predictor_elastic_mixed_n<6, true>(a, t, f, s);
    }
    return cudaErrorInvalidValue;
  }
  switch (a.g.order) {
    case 1: return launch_predictor_elastic_n<1, true>(a, t, f, s);
    case 2: return launch_predictor_elastic_n<2, true>(a, t, f, s);
    case 3: return launch_predictor_elastic_n<3, true>(a, t, f, s);
    case 4: return launch_predictor_elastic_n<4, true>(a, t, f, s);
    case 5: return launch_predictor_elastic_n<5, true>(a, t, f, s);
    case 6: return launch_predictor_elastic_n<6, true>(a, t, f, s);
  }
  return cudaErrorInvalidValue;
}

}  // namespace ader
