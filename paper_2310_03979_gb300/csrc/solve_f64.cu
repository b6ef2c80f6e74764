// solve_f64.cu - the whole-lattice solve of Eq. pure in FP64.
#include "solve_launch.cuh"

namespace srm3 {

int solve_iterate_f64(const SolveArgs &A, int it, int device, int nsm, cudaStream_t st) {
  return solve_iterate<double2>(A, it, device, nsm, st);
}

}  // namespace srm3
