// Spectral solve: kernel variants of one precision and size class (spectral_dev.cuh).
#include "spectral_dev.cuh"

namespace lbeh {
const void *spectral_kernel_f32_big() { return (const void *)k_spectral<float, true, false, true>; }
}  // namespace lbeh
