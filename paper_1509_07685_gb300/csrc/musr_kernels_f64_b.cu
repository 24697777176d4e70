// musr_kernels_f64_b.cu -- instantiates the FP64 basis kernels (kShapeT2, kShapeT2N1) of musr_kernels_f64.cuh.
#include "musr_kernels_f64.cuh"

namespace musr {

int launch_group_f64_b(int shape, int mode, int grad, const LaunchHead& h, int sms, cudaStream_t s,
                       LaunchInfo* info) {
  switch (shape) {
    case kShapeT2:
      return kern::dispatch64<kShapeT2>(mode, grad, h, sms, s, info);
    case kShapeT2N1:
      return kern::dispatch64<kShapeT2N1>(mode, grad, h, sms, s, info);
    default:
      return -1;
  }
}

}  // namespace musr
