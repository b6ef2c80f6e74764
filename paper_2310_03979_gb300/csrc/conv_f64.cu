// conv_f64.cu - the self-convolution pair sum in FP64 (separable bispectra of FP64 plans).
#include "conv_launch.cuh"

namespace srm3 {

int conv_run_f64(const ConvJob &j) { return conv_run<double2>(j); }

}  // namespace srm3
