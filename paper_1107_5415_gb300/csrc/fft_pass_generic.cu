// Dispatch of the split-precision passes with odd prime radices (fft_kernels.cuh;
// every other pass with odd radices runs in fft_mixed.cuh).
#include "fft_plan.hpp"

namespace pfft {

int launch_generic_c64_e32(const PassArgs& a, cudaStream_t s);  // fft_pass_generic_c64_e32{,u}.cu

int launch_pass_generic(const PassArgs& a, int dtype, cudaStream_t s) {
  return dtype == 0 && a.tc ? launch_generic_c64_e32(a, s) : -1;
}

}  // namespace pfft
