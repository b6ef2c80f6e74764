// solve_tf.cu - the whole-lattice solve of Eq. pure in triple-float.
#include "solve_launch.cuh"

namespace srm3 {

int solve_iterate_tf(const SolveArgs &A, int it, int device, int nsm, cudaStream_t st) {
  return solve_iterate<tf2>(A, it, device, nsm, st);
}

}  // namespace srm3
