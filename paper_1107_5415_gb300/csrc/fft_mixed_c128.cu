// The mixed-radix passes of complex128 elements.
#include "fft_mixed.cuh"

namespace pfft {

int launch_mixed_c128(const MixDesc& a, cudaStream_t s) {
  static const bool ok = cudaFuncSetAttribute(reinterpret_cast<const void*>(mixed_kernel<double2>),
                                              cudaFuncAttributeMaxDynamicSharedMemorySize, 227 * 1024) == cudaSuccess;
  if (!ok) return -1;
  mixed_kernel<double2><<<dim3(a.groups, a.kind == MIX_WHOLE ? 1 : a.batch), a.nthreads, a.smem_bytes, s>>>(a);
  return cudaGetLastError() == cudaSuccess ? 0 : -1;
}

}  // namespace pfft
