// Spectral solve: kernel variants of one precision and size class (spectral_dev.cuh).
#include "spectral_dev.cuh"

namespace lbeh {
const void *spectral_kernel_f64(bool mix) {
  return mix ? (const void *)k_spectral<double, false, true, true> : (const void *)k_spectral<double, false, false, true>;
}
}  // namespace lbeh
