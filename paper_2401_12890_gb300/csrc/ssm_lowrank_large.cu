// The low-rank FP32 iteration kernel (ssm_lowrank.cuh) for padded ranks 40 to 64.
#define SSM_LOWRANK_KERNEL
#include "ssm_lowrank.cuh"

namespace ssm {

LowrankKernel lowrank_kernel_large(int R, int naxes) {
  switch (R) {
    case 40: return kernel_of<40>(naxes);
    case 48: return kernel_of<48>(naxes);
    case 56: return kernel_of<56>(naxes);
    case 64: return kernel_of<64>(naxes);
    default: return LowrankKernel{nullptr, nullptr};
  }
}

}  // namespace ssm
