// The flat two-phase Arnoldi kernel for the operators of the Gray-Scott
// gradient (float64 form only): the transposed Jacobian and the block operator
// of the Frechet derivative.
#include "lsa_flat.cuh"

namespace lsa {

cudaError_t launch_arnoldi_flat_grayscott2d_t(const ArnoldiParams& P, int G, cudaStream_t s) {
  return launch_arnoldi_flat_t<OpGrayScott2DT, double, false>(P, G, s);
}
int flat_blocks_per_sm_grayscott2d_t() { return flat_blocks_per_sm_t<OpGrayScott2DT, double, false>(); }

cudaError_t launch_arnoldi_flat_grayscott2d_frechet(const ArnoldiParams& P, int G, cudaStream_t s) {
  return launch_arnoldi_flat_t<OpGrayScottFrechet2D, double, false>(P, G, s);
}
int flat_blocks_per_sm_grayscott2d_frechet() { return flat_blocks_per_sm_t<OpGrayScottFrechet2D, double, false>(); }

}  // namespace lsa
