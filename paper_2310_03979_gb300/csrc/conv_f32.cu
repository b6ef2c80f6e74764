// conv_f32.cu - the self-convolution pair sum in FP32 (separable bispectra of FP32 plans).
#include "conv_launch.cuh"

namespace srm3 {

int conv_run_f32(const ConvJob &j) { return conv_run<float2>(j); }

}  // namespace srm3
