// The low-rank FP32 iteration kernel (ssm_lowrank.cuh) for padded ranks 20 to 32.
#define SSM_LOWRANK_KERNEL
#include "ssm_lowrank.cuh"

namespace ssm {

LowrankKernel lowrank_kernel_mid(int R, int naxes) {
  switch (R) {
    case 20: return kernel_of<20>(naxes);
    case 24: return kernel_of<24>(naxes);
    case 28: return kernel_of<28>(naxes);
    case 32: return kernel_of<32>(naxes);
    default: return LowrankKernel{nullptr, nullptr};
  }
}

}  // namespace ssm
