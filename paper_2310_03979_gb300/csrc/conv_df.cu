// conv_df.cu - the self-convolution pair sum in double-float (FP32 plans, Gaussian envelope).
#include "conv_launch.cuh"

namespace srm3 {

int conv_run_df(const ConvJob &j) { return conv_run<df2>(j); }

}  // namespace srm3
