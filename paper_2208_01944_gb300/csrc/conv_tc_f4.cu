// The layer kernel's instances for packed FP4 codes.
#include "conv_tc.cuh"

namespace pq {

const void* conv_kernel_f4(bool lu) {
  return lu ? reinterpret_cast<const void*>(pq_conv_tc_kernel<true, true>)
            : reinterpret_cast<const void*>(pq_conv_tc_kernel<true, false>);
}

}  // namespace pq
