// Polar resampling and ring FFT launchers with 16-bit (BF16 / FP16) output
// for the precision-split path (mma.sync fragments).  The kernel itself is in
// polar_impl.cuh.
#include "polar_impl.cuh"

namespace mra {

cudaError_t launch_polar16(const Geometry &g, const PolarArgs &a, cudaStream_t st) {
  return launch_polar_out<kOut16>(g, a, st);
}

}  // namespace mra
