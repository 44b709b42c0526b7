// The batched kernel instantiated for the advdiff2d operator (a translation unit of
// its own: it holds the tile and the flat passes).
#include "lsa_batched.cuh"

namespace lsa {

cudaError_t launch_batched_advdiff2d(const BatchParams& BP, int precision, int G, cudaStream_t s) {
  return launch_batched_op<OpAdvDiff2D>(BP, precision, G, s);
}
int batched_blocks_per_sm_advdiff2d(int precision) { return batched_blocks_per_sm_op<OpAdvDiff2D>(precision); }

}  // namespace lsa
