// The flat two-phase Arnoldi kernel instantiated for the advdiff2d operator: both
// precisions, and the augmented operator (float64).
#include "lsa_flat.cuh"

namespace lsa {

cudaError_t launch_arnoldi_flat_advdiff2d(const ArnoldiParams& P, int precision, int G, cudaStream_t s) {
  if (P.naug > 0) return launch_arnoldi_flat_t<OpAdvDiff2D, double, true>(P, G, s);
  return precision == LSA_FP64 ? launch_arnoldi_flat_t<OpAdvDiff2D, double, false>(P, G, s)
                               : launch_arnoldi_flat_t<OpAdvDiff2D, float, false>(P, G, s);
}
int flat_blocks_per_sm_advdiff2d(int precision, int aug) {
  if (aug) return flat_blocks_per_sm_t<OpAdvDiff2D, double, true>();
  return precision == LSA_FP64 ? flat_blocks_per_sm_t<OpAdvDiff2D, double, false>() : flat_blocks_per_sm_t<OpAdvDiff2D, float, false>();
}

}  // namespace lsa
