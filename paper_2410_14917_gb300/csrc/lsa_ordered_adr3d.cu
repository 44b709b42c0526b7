// The float32 two-phase Arnoldi kernel with the tile passes' sums, for the adr3d operator.
#include "lsa_ordered.cuh"

namespace lsa {

cudaError_t launch_arnoldi_ordered_adr3d(const ArnoldiParams& P, int G, cudaStream_t s) {
  return launch_arnoldi_ordered_t<OpADR3D>(P, G, s);
}
int ordered_blocks_per_sm_adr3d() { return ordered_blocks_per_sm_t<OpADR3D>(); }

}  // namespace lsa
