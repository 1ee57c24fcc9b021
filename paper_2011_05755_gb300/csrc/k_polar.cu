// Polar resampling and ring FFT launchers: the FP32-output instantiations
// and the dispatcher (the 16-bit-output ones are in k_polar16.cu).  The
// kernel itself is in polar_impl.cuh.
#include "polar_impl.cuh"

namespace mra {

cudaError_t launch_polar16(const Geometry &g, const PolarArgs &a, cudaStream_t st);

size_t polar_smem_one_row(const Geometry &g, int mode, bool out16) { return polar_smem_bytes(g, mode, out16, 1); }

int polar_rows_per_cta(const Geometry &g, int mode, bool out16) { return polar_cta_rows(g, mode, out16); }

cudaError_t launch_polar(const Geometry &g, const PolarArgs &a, cudaStream_t st) {
  if (a.n_imgs <= 0 || a.rows_per_img <= 0) return cudaSuccess;
  return a.out16 ? launch_polar16(g, a, st) : launch_polar_out<kOutF32>(g, a, st);
}

}  // namespace mra
