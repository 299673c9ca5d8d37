// The DFT sweep for ranks up to 6.
#include "fourier_sweep.cuh"

namespace lrs {
void* fsweep_kernel_r6(bool pow2) {
  return pow2 ? reinterpret_cast<void*>(&fourier::fsweep_kernel<6, true>)
              : reinterpret_cast<void*>(&fourier::fsweep_kernel<6, false>);
}
}  // namespace lrs
