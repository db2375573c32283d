// The low-rank FP32 iteration kernel (ssm_lowrank.cuh) for padded ranks up to 16.
#define SSM_LOWRANK_KERNEL
#include "ssm_lowrank.cuh"

namespace ssm {

LowrankKernel lowrank_kernel_small(int R, int naxes) {
  switch (R) {
    case 4: return kernel_of<4>(naxes);
    case 8: return kernel_of<8>(naxes);
    case 12: return kernel_of<12>(naxes);
    case 16: return kernel_of<16>(naxes);
    default: return LowrankKernel{nullptr, nullptr};
  }
}

}  // namespace ssm
