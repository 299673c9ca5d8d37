// The DFT sweep for ranks up to 4.
#include "fourier_sweep.cuh"

namespace lrs {
void* fsweep_kernel_r4(bool pow2) {
  return pow2 ? reinterpret_cast<void*>(&fourier::fsweep_kernel<4, true>)
              : reinterpret_cast<void*>(&fourier::fsweep_kernel<4, false>);
}
}  // namespace lrs
