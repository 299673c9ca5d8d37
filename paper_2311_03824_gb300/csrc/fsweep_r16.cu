// The DFT sweep for ranks up to 16.
#include "fourier_sweep.cuh"

namespace lrs {
void* fsweep_kernel_r16(bool pow2) {
  return pow2 ? reinterpret_cast<void*>(&fourier::fsweep_kernel<16, true>)
              : reinterpret_cast<void*>(&fourier::fsweep_kernel<16, false>);
}
}  // namespace lrs
