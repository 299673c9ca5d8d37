// Instantiation of the streaming engine for rank width 12 (all stored forms
// of A_k).
#include "stream_impl.cuh"

namespace lrs {
void* stream_w_kernel_r12(int et) {
  using namespace stream;
  switch (et) {
    case 1: return reinterpret_cast<void*>(&w_kernel<12, 1>);
    case 2: return reinterpret_cast<void*>(&w_kernel<12, 2>);
    case 3: return reinterpret_cast<void*>(&w_kernel<12, 3>);
    default: return reinterpret_cast<void*>(&w_kernel<12, 0>);
  }
}
void* stream_step_kernel_r12(int next, int variant) {
  using namespace stream;
  switch (variant) {
    case 0: return next ? reinterpret_cast<void*>(&step_next_kernel<12, 0>)
                        : reinterpret_cast<void*>(&step_first_kernel<12, 0>);
    case 1: return next ? reinterpret_cast<void*>(&step_next_kernel<12, 1>)
                        : reinterpret_cast<void*>(&step_first_kernel<12, 1>);
    default: return next ? reinterpret_cast<void*>(&step_next_kernel<12, 2>)
                         : reinterpret_cast<void*>(&step_first_kernel<12, 2>);
  }
}
}  // namespace lrs
