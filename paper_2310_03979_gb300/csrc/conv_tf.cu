// conv_tf.cu - the self-convolution pair sum in triple-float (FP64 plans, Gaussian envelope).
#include "conv_launch.cuh"

namespace srm3 {

int conv_run_tf(const ConvJob &j) { return conv_run<tf2>(j); }

}  // namespace srm3
