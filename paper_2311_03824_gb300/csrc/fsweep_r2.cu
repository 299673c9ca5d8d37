// The DFT sweep for ranks up to 2.
#include "fourier_sweep.cuh"

namespace lrs {
void* fsweep_kernel_r2(bool pow2) {
  return pow2 ? reinterpret_cast<void*>(&fourier::fsweep_kernel<2, true>)
              : reinterpret_cast<void*>(&fourier::fsweep_kernel<2, false>);
}
}  // namespace lrs
