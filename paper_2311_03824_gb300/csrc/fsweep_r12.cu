// The DFT sweep for ranks up to 12.
#include "fourier_sweep.cuh"

namespace lrs {
void* fsweep_kernel_r12(bool pow2) {
  return pow2 ? reinterpret_cast<void*>(&fourier::fsweep_kernel<12, true>)
              : reinterpret_cast<void*>(&fourier::fsweep_kernel<12, false>);
}
}  // namespace lrs
