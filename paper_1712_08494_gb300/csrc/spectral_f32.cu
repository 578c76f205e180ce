// Spectral solve: kernel variants of one precision and size class (spectral_dev.cuh).
#include "spectral_dev.cuh"

namespace lbeh {
const void *spectral_kernel_f32(bool mix) {
  return mix ? (const void *)k_spectral<float, true, true, false> : (const void *)k_spectral<float, true, false, false>;
}
}  // namespace lbeh
