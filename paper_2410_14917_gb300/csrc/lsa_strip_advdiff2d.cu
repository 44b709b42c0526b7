// The float32 two-phase Arnoldi kernel with the streaming kernel's sums, for the advdiff2d operator.
#include "lsa_strip.cuh"

namespace lsa {

cudaError_t launch_arnoldi_strip_advdiff2d(const ArnoldiParams& P, int G, int ranks, cudaStream_t s) {
  return launch_arnoldi_strip_t<OpAdvDiff2D>(P, G, ranks, s);
}
int strip_blocks_per_sm_advdiff2d() { return strip_blocks_per_sm_t<OpAdvDiff2D>(); }

}  // namespace lsa
