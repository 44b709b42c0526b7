// The float32 two-phase Arnoldi kernel with the streaming kernel's sums, for the adr3d operator.
#include "lsa_strip.cuh"

namespace lsa {

cudaError_t launch_arnoldi_strip_adr3d(const ArnoldiParams& P, int G, int ranks, cudaStream_t s) {
  return launch_arnoldi_strip_t<OpADR3D>(P, G, ranks, s);
}
int strip_blocks_per_sm_adr3d() { return strip_blocks_per_sm_t<OpADR3D>(); }

}  // namespace lsa
