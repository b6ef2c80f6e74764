// solve_df.cu - the whole-lattice solve of Eq. pure in double-float.
#include "solve_launch.cuh"

namespace srm3 {

int solve_iterate_df(const SolveArgs &A, int it, int device, int nsm, cudaStream_t st) {
  return solve_iterate<df2>(A, it, device, nsm, st);
}

}  // namespace srm3
