// The batched kernel instantiated for the grayscott2d operator (a translation unit of
// its own: it holds the tile and the flat passes).
#include "lsa_batched.cuh"

namespace lsa {

cudaError_t launch_batched_grayscott2d(const BatchParams& BP, int precision, int G, cudaStream_t s) {
  return launch_batched_op<OpGrayScott2D>(BP, precision, G, s);
}
int batched_blocks_per_sm_grayscott2d(int precision) { return batched_blocks_per_sm_op<OpGrayScott2D>(precision); }

}  // namespace lsa
