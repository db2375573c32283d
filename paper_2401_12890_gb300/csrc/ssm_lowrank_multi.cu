// The low-rank FP32 iteration kernel (ssm_lowrank.cuh) with a dictionary per voxel label.
#define SSM_LOWRANK_KERNEL
#include "ssm_lowrank.cuh"

namespace ssm {

LowrankKernel lowrank_kernel_multi(int R, int naxes) {
  switch (R) {
    case 4: return kernel_of<4, true>(naxes);
    case 8: return kernel_of<8, true>(naxes);
    case 12: return kernel_of<12, true>(naxes);
    case 16: return kernel_of<16, true>(naxes);
    default: return LowrankKernel{nullptr, nullptr};
  }
}

}  // namespace ssm
