// Launch of the layer kernel (conv_tc.cuh): picks the instance that a call needs.  The
// instances are compiled in translation units of their own, in parallel.
#include <cuda_runtime.h>

#include "pq_internal.h"

namespace pq {

const void* conv_kernel_f8(bool lu);
const void* conv_kernel_f4(bool lu);

int launch_conv_tc(const ConvParams& p, const CUtensorMap& tma_a, const CUtensorMap& tma_w, int grid,
                   cudaStream_t stream) {
  // the attribute is set once per instance and device
  static int attr_set_for_device[4][64] = {{0}};
  int dev = 0;
  if (cudaGetDevice(&dev) != cudaSuccess) return -1;
  const int need = static_cast<int>(p.smem_bytes) + 1024;
  const bool f4 = p.codes_f4 != 0, lu = p.q_lu != 0;
  const int v = (f4 ? 2 : 0) + (lu ? 1 : 0);
  const void* fn = f4 ? conv_kernel_f4(lu) : conv_kernel_f8(lu);
  if (dev >= 64 || attr_set_for_device[v][dev] < need) {
    if (cudaFuncSetAttribute(fn, cudaFuncAttributeMaxDynamicSharedMemorySize, kMaxSmem) != cudaSuccess) return -1;
    if (dev < 64) attr_set_for_device[v][dev] = kMaxSmem;
  }
  cudaLaunchConfig_t cfg = {};
  cfg.gridDim = dim3(grid);
  cfg.blockDim = dim3(kConvThreads);
  cfg.dynamicSmemBytes = static_cast<size_t>(need);
  cfg.stream = stream;
  cudaLaunchAttribute attr[1];
  attr[0].id = cudaLaunchAttributeProgrammaticStreamSerialization;
  attr[0].val.programmaticStreamSerializationAllowed = 1;
  cfg.attrs = attr;
  cfg.numAttrs = p.pdl ? 1 : 0;
  void* args[] = {const_cast<ConvParams*>(&p), const_cast<CUtensorMap*>(&tma_a), const_cast<CUtensorMap*>(&tma_w)};
  const cudaError_t e = cudaLaunchKernelExC(&cfg, fn, args);
  return e == cudaSuccess && cudaGetLastError() == cudaSuccess ? 0 : -1;
}

}  // namespace pq
