// The batched kernel instantiated for the adr3d operator (a translation unit of
// its own: it holds the tile and the flat passes).
#include "lsa_batched.cuh"

namespace lsa {

cudaError_t launch_batched_adr3d(const BatchParams& BP, int precision, int G, cudaStream_t s) {
  return launch_batched_op<OpADR3D>(BP, precision, G, s);
}
int batched_blocks_per_sm_adr3d(int precision) { return batched_blocks_per_sm_op<OpADR3D>(precision); }

}  // namespace lsa
