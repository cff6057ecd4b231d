// The layer kernel's instances for byte and packed 2-bit codes.
#include "conv_tc.cuh"

namespace pq {

const void* conv_kernel_f8(bool lu) {
  return lu ? reinterpret_cast<const void*>(pq_conv_tc_kernel<false, true>)
            : reinterpret_cast<const void*>(pq_conv_tc_kernel<false, false>);
}

}  // namespace pq
