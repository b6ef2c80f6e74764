// solve_launch.cuh - one iteration of the whole-lattice solve of Eq. pure
// (kernels in solve.cuh) for one number type; one translation unit per type
// instantiates it (solve_df.cu, solve_tf.cu).
#pragma once

#include <algorithm>
#include <atomic>
#include <type_traits>

#include "solve.cuh"
#include "srm3_internal.cuh"

namespace srm3 {
namespace {

template <int L0, int L1, class F>
void solve_with_log2(int v, F &&f) {
  if constexpr (L0 <= L1) {
    if (v == L0)
      f(std::integral_constant<int, L0>{});
    else
      solve_with_log2<L0 + 1, L1>(v, f);
  }
}

constexpr int kSolveSmemMax = 224 * 1024;  // beside the kernels' static words

// The kernel's dynamic shared memory limit raised once per device.
template <auto K>
cudaError_t solve_prepare(int dev) {
  static std::atomic<unsigned long long> done{0};
  const unsigned long long bit = dev >= 0 && dev < 64 ? 1ull << dev : 0ull;
  if (bit && (done.load(std::memory_order_relaxed) & bit)) return cudaSuccess;
  const cudaError_t e =
      cudaFuncSetAttribute(K, cudaFuncAttributeMaxDynamicSharedMemorySize, kSolveSmemMax);
  if (e == cudaSuccess) done.fetch_or(bit, std::memory_order_relaxed);
  return e;
}

// A launch whose CTAs may be placed before the kernel ahead of it in the stream
// has completed (its kernels wait for that themselves, solve_turn), where it has
// at most one CTA per SM: early CTAs of larger launches settle unevenly on the
// SMs.  Without / with / with this rule: 32 x 32 FP64 plan and sample 913 / 822 /
// 817 us, 40 x 70 mixed with 16 samples 1028 / 867 / 864 us, 256 x 512 with 64
// samples 3514 / 3617 / 3424 us.
template <class... P, class... Q>
cudaError_t solve_launch(void (*k)(P...), int nsm, int grid, int threads, size_t smem,
                         cudaStream_t st, Q... args) {
  cudaLaunchConfig_t c = {};
  c.gridDim = dim3(grid);
  c.blockDim = dim3(threads);
  c.dynamicSmemBytes = smem;
  c.stream = st;
  cudaLaunchAttribute at[1];
  at[0].id = cudaLaunchAttributeProgrammaticStreamSerialization;
  at[0].val.programmaticStreamSerializationAllowed = 1;
  c.attrs = at;
  c.numAttrs = grid <= nsm ? 1 : 0;
  return cudaLaunchKernelEx(&c, k, P(args)...);
}

// Column pairs per CTA: two where that still leaves two CTAs per SM, else one
// (a pass is short: the spread over the SMs counts for more than the width of
// its 16- or 32-byte accesses, which stay in L2).
template <typename T2>
int solve_iterate(SolveArgs A, int it, int device, int nsm, cudaStream_t st) {
  int lk = 0, lm = 0;
  while ((1 << lk) < A.Nk) ++lk;
  while ((1 << lm) < A.M) ++lm;
  // rows per CTA: what 64 threads hold, fewer where that leaves SMs idle; whole warps
  const int tpt = solve_tpt(lm), most = std::max(1, 64 / tpt);
  A.rows = std::min(most, std::max(1, (A.nk + nsm - 1) / nsm));
  const int rthreads = (A.rows * tpt + 31) / 32 * 32, rb = rthreads / tpt;
  const size_t srow = (size_t)rb * (tx_len(A.M) + 1) * sizeof(T2);
  const size_t sout = srow + (A.mixed ? (size_t)rthreads * sizeof(typename RealOf<T2>::type) : 0);
  const int wf = sizeof(T2) == 24 ? 4 : (int)(128 / sizeof(T2));
  const int pairs = A.M / 2 + 1;
  int TC = 2;
  while (TC > 1 && ((pairs + TC - 1) / TC < 2 * nsm || 2 * TC * solve_tpt(lk) > solve_col_threads(lk)))
    TC >>= 1;
  const int cs = (tx_len(A.Nk) + wf - 1) / wf * wf + wf / (2 * TC);
  const size_t scol = (size_t)2 * TC * cs * sizeof(T2);
  const int rows = (A.nk + A.rows - 1) / A.rows;
  cudaError_t err = cudaSuccess;
  solve_with_log2<1, 12>(lm, [&](auto c) {
    constexpr int L = decltype(c)::value;
    err = solve_prepare<k_solve_rows<L, T2>>(device);
    if (err == cudaSuccess) err = solve_launch(k_solve_rows<L, T2>, nsm, rows, rthreads, srow, st, A, it);
  });
  if (err == cudaSuccess) err = cudaGetLastError();
  if (err != cudaSuccess) return cuda_fail(err, "whole-lattice solve, rows");
  solve_with_log2<1, 12>(lk, [&](auto c) {
    constexpr int L = decltype(c)::value;
    err = solve_prepare<k_solve_cols<L, T2>>(device);
    if (err == cudaSuccess)
      err = solve_launch(k_solve_cols<L, T2>, nsm, (pairs + TC - 1) / TC, 2 * TC * solve_tpt(L), scol, st,
                         A, it, TC, cs);
  });
  if (err == cudaSuccess) err = cudaGetLastError();
  if (err != cudaSuccess) return cuda_fail(err, "whole-lattice solve, columns");
  solve_with_log2<1, 12>(lm, [&](auto c) {
    constexpr int L = decltype(c)::value;
    err = solve_prepare<k_solve_out<L, T2>>(device);
    if (err == cudaSuccess) err = solve_launch(k_solve_out<L, T2>, nsm, rows, rthreads, sout, st, A, it);
  });
  if (err == cudaSuccess) err = cudaGetLastError();
  if (err != cudaSuccess) return cuda_fail(err, "whole-lattice solve, output rows");
  return SRM3_OK;
}

}  // namespace
}  // namespace srm3
