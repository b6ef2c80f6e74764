// conv_launch.cuh - launches of the self-convolution pair sum (kernels in
// conv.cuh) for one number type; one translation unit per type instantiates
// it (conv_f32.cu, conv_f64.cu, conv_df.cu).
#pragma once

#include <algorithm>
#include <atomic>
#include <cmath>
#include <cstring>

#include "conv.cuh"
#include "srm3_internal.cuh"

namespace srm3 {
namespace {

int conv_cdiv(long long a, long long b) { return (int)((a + b - 1) / b); }

// f(std::integral_constant<int, l>) for the l in [L0, L1] equal to v.
template <int L0, int L1, class F>
void conv_with_log2(int v, F &&f) {
  if constexpr (L0 <= L1) {
    if (v == L0)
      f(std::integral_constant<int, L0>{});
    else
      conv_with_log2<L0 + 1, L1>(v, f);
  }
}

constexpr int kConvSmemMax = 227 * 1024;

// The kernel's dynamic shared memory limit raised once per device.
template <auto K>
cudaError_t conv_prepare(int dev) {
  static std::atomic<unsigned long long> done{0};
  const unsigned long long bit = dev >= 0 && dev < 64 ? 1ull << dev : 0ull;
  if (bit && (done.load(std::memory_order_relaxed) & bit)) return cudaSuccess;
  const cudaError_t e =
      cudaFuncSetAttribute(K, cudaFuncAttributeMaxDynamicSharedMemorySize, kConvSmemMax);
  if (e == cudaSuccess) done.fetch_or(bit, std::memory_order_relaxed);
  return e;
}

// The pair sum of n samples into C, as many samples at a time as the work
// block holds (grid rows and phasors of two sheet-samples each).
//
// Which plans take it: every separable bispectrum, and the Gaussian envelope
// with W recomputed at every size.  Both sides measured (GB300, FP32 plans,
// pair sum with its phases): 256 x 512, 64 samples 44.4 -> 1.74 ms; 512 x
// 1024, 16 samples 183 -> 2.13 ms; 32 spectra on lattices of 32..256 per axis
// in one captured batch 22.7 -> 2.4 ms; one sample on 32 x 32, with its field,
// 60 -> 26 us.  FP64 plans: 90 x 117, 4 samples 1.64 -> 0.070 ms (in FP64 0.097 ms).
// Against 64-bit coefficients the FP32 fields' relative error went 1.9e-7 -> 1.8e-7
// (2.1e-7 -> 1.9e-7 on 512 x 1024).  FP64 coefficients against the oracle's, direct
// sums / triple-float / FP64 transforms: 90 x 117 2.96e-16 / 2.96e-16 / 9.6e-16,
// sigma_g = 0.2237 2.91e-16 / 2.90e-16 / 1.9e-15, 24 x 37 mixed 2.98e-16 / 2.93e-16 /
// 4.3e-16 in the norm.
//
// What bounds it: the FP32 pipe.  A point and level of a transform costs ~28
// FP32 operations in double-float (2 two-sums of 8 per sum, 32 a complex
// product), ~46e9 for the 256 x 512 case = 1.2 ms at the pipe's peak.  The column
// pass takes TC columns per CTA (at most 16, within its threads and 100 KB),
// the column stride chosen so that the TC columns of one access fall on
// distinct banks.
template <typename T2>
int conv_run(const ConvJob &j) {
  using Y2 = typename ConvNum<T2>::Y2;
  const srm3_plan *p = j.plan;
  const int lk = p->log2cNk, lw = p->log2cNw, Nk = p->cNk, Nw = p->cNw;
  const size_t zrow = (size_t)p->nk * Nw * sizeof(T2), yrow = (size_t)p->nk * p->nw * sizeof(Y2);
  int per = (int)std::min<size_t>((size_t)j.n, j.work_bytes / (2 * (zrow + yrow)));
  per = std::min(per, 16384);
  if (!j.dseeds) per = std::min(per, kMaxChunk);
  if (per < 1) return fail(SRM3_ERR_INVALID_ARG, "pair sum: workspace too small");
  // rows per CTA: what 64 threads hold, fewer where that leaves SMs idle; whole warps
  int nsm = 0;
  cudaDeviceGetAttribute(&nsm, cudaDevAttrMultiProcessorCount, p->device);
  const int tpt = conv_tpt<T2>(lw), most = std::max(1, 64 / tpt);
  if (j.max_ctas > 0) {
    const long long threads = 2LL * p->nk * tpt;  // of one sample's rows
    per = (int)std::min<long long>(per, std::max<long long>(1, 1024LL * j.max_ctas / threads));
  }
  const long long allrows = (long long)p->nk * 2 * per;
  const int rows = (int)std::min<long long>(most, std::max<long long>(1, allrows / (4 * nsm)));
  const int rthreads = (rows * tpt + 31) / 32 * 32, rb = rthreads / tpt;
  const int copies = p->mixed ? 2 : 1;
  const size_t stage = (size_t)rb * (tx_len(Nw) + 1) * sizeof(T2);
  const size_t srow = conv_align(stage) + (size_t)rb * copies * p->nw * sizeof(Y2);
  const size_t sout = stage + (p->mixed ? (size_t)rthreads * sizeof(T2) : 0);
  // lanes of one shared-memory wavefront (triple-floats: of their 32-byte spacing)
  const int wf = sizeof(T2) == 24 ? 4 : (int)(128 / sizeof(T2));
  auto colstride = [&](int tc) {
    const int len = (tx_len(Nk) + wf - 1) / wf * wf;
    return len + (tc >= wf ? 1 : wf / tc);
  };
  int TC = 16;
  while (TC > 1 && (TC > Nw || (size_t)TC * colstride(TC) * sizeof(T2) > 100 * 1024 ||
                    TC * conv_tpt<T2>(lk) > conv_col_threads<T2>(lk) ||
                    (long long)(Nw / TC) * 2 * per < nsm))
    TC >>= 1;
  const int cs = colstride(TC);
  const size_t scol = (size_t)TC * cs * sizeof(T2);
  if (std::max({srow, sout, scol}) > (size_t)kConvSmemMax)
    return fail(SRM3_ERR_NOT_SUPPORTED,
                "pair sum: a padded row or column does not fit in shared memory");
  ConvArgs A;
  std::memset(static_cast<void *>(&A), 0, sizeof(A));
  A.nk = p->nk;
  A.nw = p->nw;
  A.Nk = Nk;
  A.Nw = Nw;
  A.mixed = p->mixed ? 1 : 0;
  constexpr bool f32 = std::is_same<T2, float2>::value;
  constexpr bool gauss = !kPlainNum<T2>;  // the others: separable bispectra alone
  if (p->sep) {
    A.e = f32 ? (const void *)p->env_e32 : (const void *)p->env_e;
    A.eb = f32 ? (const void *)p->env_b32 : (const void *)p->env_b;
  } else {
    const size_t es = sizeof(typename ConvNum<T2>::F);
    const char *f = static_cast<const char *>(p->conv_fac);  // aK, bK, aW, bW
    A.aK = f;
    A.bK = f + es * p->nk;
    A.aW = f + es * 2 * p->nk;
    A.bW = f + es * (2 * p->nk + 2 * p->nw - 1);
  }
  A.sqq = p->sqq;
  A.Pk = p->Pk;
  A.ck = p->ck;
  A.sqq_of = j.sqq_of;
  A.pk_of = j.pk_of;
  A.ck_of = j.ck_of;
  A.dseeds = j.dseeds;
  A.twk = p->tw_conv;
  A.tww = static_cast<const T2 *>(p->tw_conv) + tx_twlen(lk, conv_lv<T2>(lk));
  A.cb = std::cos(p->beta);
  A.sb = std::sin(p->beta);
  A.row_lo = p->row_lo;
  A.row_hi = p->row_hi;
  A.rows = rows;
  A.Z = j.work;
  SeedChunk sc;
  std::memset(&sc, 0, sizeof(sc));
  for (int n0 = 0; n0 < j.n; n0 += per) {
    const int ns = std::min(per, j.n - n0);
    A.n0 = n0;
    A.y = static_cast<char *>(j.work) + 2 * ns * zrow;
    A.C = static_cast<char *>(j.C) + 2 * n0 * yrow;
    if (!j.dseeds) std::memcpy(sc.s, j.seeds + n0, sizeof(uint64_t) * ns);
    cudaError_t err = cudaSuccess;
    conv_with_log2<1, kConvMaxLog2<T2>>(lw, [&](auto c) {
      constexpr int L = decltype(c)::value;
      const dim3 grid(conv_cdiv(p->nk, rows), 2 * ns);
      if constexpr (gauss) {
        if (p->mixed) {
          err = conv_prepare<k_conv_rows<L, T2, true>>(p->device);
          if (err == cudaSuccess)
            k_conv_rows<L, T2, true><<<grid, rthreads, srow, j.stream>>>(A, sc);
          return;
        }
      }
      err = conv_prepare<k_conv_rows<L, T2, false>>(p->device);
      if (err == cudaSuccess)
        k_conv_rows<L, T2, false><<<grid, rthreads, srow, j.stream>>>(A, sc);
    });
    if (err == cudaSuccess) err = cudaGetLastError();
    if (err != cudaSuccess) return cuda_fail(err, "pair sum, rows");
    conv_with_log2<1, kConvMaxLog2<T2>>(lk, [&](auto c) {
      constexpr int L = decltype(c)::value;
      err = conv_prepare<k_conv_cols<L, T2>>(p->device);
      if (err == cudaSuccess)
        k_conv_cols<L, T2><<<dim3(Nw / TC, 2 * ns), TC * conv_tpt<T2>(L), scol, j.stream>>>(
            p->nk, Nw, TC, cs, static_cast<const T2 *>(A.twk), static_cast<T2 *>(A.Z));
    });
    if (err == cudaSuccess) err = cudaGetLastError();
    if (err != cudaSuccess) return cuda_fail(err, "pair sum, columns");
    conv_with_log2<1, kConvMaxLog2<T2>>(lw, [&](auto c) {
      constexpr int L = decltype(c)::value;
      const dim3 grid(conv_cdiv(p->row_hi - p->row_lo, rows), 2 * ns);
      if constexpr (gauss) {
        if (p->mixed) {
          err = conv_prepare<k_conv_out<L, T2, true>>(p->device);
          if (err == cudaSuccess) k_conv_out<L, T2, true><<<grid, rthreads, sout, j.stream>>>(A);
          return;
        }
      }
      err = conv_prepare<k_conv_out<L, T2, false>>(p->device);
      if (err == cudaSuccess) k_conv_out<L, T2, false><<<grid, rthreads, sout, j.stream>>>(A);
    });
    if (err == cudaSuccess) err = cudaGetLastError();
    if (err != cudaSuccess) return cuda_fail(err, "pair sum, output rows");
  }
  return SRM3_OK;
}

}  // namespace
}  // namespace srm3
