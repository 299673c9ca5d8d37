// The DFT sweep for ranks up to 8.
#include "fourier_sweep.cuh"

namespace lrs {
void* fsweep_kernel_r8(bool pow2) {
  return pow2 ? reinterpret_cast<void*>(&fourier::fsweep_kernel<8, true>)
              : reinterpret_cast<void*>(&fourier::fsweep_kernel<8, false>);
}
}  // namespace lrs
