// musr_kernels_fp64.cu -- instantiates the FP64-path kernels of musr_kernels.cuh.
#include "musr_kernels.cuh"

namespace musr {

int launch_group_fp64(int mode, int grad, const LaunchHead& h, int sms, cudaStream_t s, LaunchInfo* info) {
  return kern::dispatch_mode<0, 0>(mode, grad, h, sms, s, info);
}
int occupancy_group_fp64(int mode, int grad) { return kern::occupancy_mode<0, 0>(mode, grad); }

}  // namespace musr
