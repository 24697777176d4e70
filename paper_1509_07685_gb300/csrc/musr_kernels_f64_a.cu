// musr_kernels_f64_a.cu -- instantiates the FP64 basis kernels (kShapeGeneric, kShapeT1, kShapeN1, kShapeT1N1) of musr_kernels_f64.cuh.
#include "musr_kernels_f64.cuh"

namespace musr {

int launch_group_f64_a(int shape, int mode, int grad, const LaunchHead& h, int sms, cudaStream_t s,
                       LaunchInfo* info) {
  switch (shape) {
    case kShapeGeneric:
      return kern::dispatch64<kShapeGeneric>(mode, grad, h, sms, s, info);
    case kShapeT1:
      return kern::dispatch64<kShapeT1>(mode, grad, h, sms, s, info);
    case kShapeN1:
      return kern::dispatch64<kShapeN1>(mode, grad, h, sms, s, info);
    case kShapeT1N1:
      return kern::dispatch64<kShapeT1N1>(mode, grad, h, sms, s, info);
    default:
      return -1;
  }
}

}  // namespace musr
