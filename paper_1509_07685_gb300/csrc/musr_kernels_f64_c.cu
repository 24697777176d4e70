// musr_kernels_f64_c.cu -- instantiates the FP64 basis kernels (kShapeT2m, kShapeT2N1m) of musr_kernels_f64.cuh.
#include "musr_kernels_f64.cuh"

namespace musr {

int launch_group_f64_c(int shape, int mode, int grad, const LaunchHead& h, int sms, cudaStream_t s,
                       LaunchInfo* info) {
  switch (shape) {
    case kShapeT2m:
      return kern::dispatch64<kShapeT2m>(mode, grad, h, sms, s, info);
    case kShapeT2N1m:
      return kern::dispatch64<kShapeT2N1m>(mode, grad, h, sms, s, info);
    default:
      return -1;
  }
}

}  // namespace musr
