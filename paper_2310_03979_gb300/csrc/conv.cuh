// conv.cuh - the pair sum of an envelope that factors on i + j = k, g(i,j) =
// a(i) a(j) b(i+j), as an FFT self-convolution (a3 + a4 + a5: phases, pair
// sum, coefficients).  Included by the conv_*.cu units.
//
// With W_ij = c_k a_i a_j b_k the pair part of C_k is
//   c_k e^{i beta} b_k sum_{Pi(k)} z_i z_j,   z = a y  (z_0 = 0),
// and over unordered pairs {i, j}, i + j = k,
//   sum_{Pi(k)} z_i z_j = ((z * z)_k + [k even] z_{k/2}^2) / 2,
// with (z * z) the linear 2-D self-convolution on the quadrant lattice.  It
// is taken on a zero-padded Nk x Nw grid (powers of two, Nk >= 2 n_kappa - 1,
// Nw >= 2 n_omega - 1): three passes per sheet-sample -- rows of z
// (k_conv_rows), columns, square, columns again (k_conv_cols), rows and the
// coefficient epilogue (k_conv_out) -- all with the e^{+} transform of the
// output stage, the second one as conj(G(conj(G(z)^2))).  The inputs of the
// first row and column transforms are zero past n_omega, n_kappa <= half the
// length and the outputs of the second ones are needed up to there: the first
// passes skip the upper half of their input blocks (tx_mask_low_half), the
// last ones the upper half of their outputs.
//
// Two envelopes take this form: the tables of a separable bispectrum, and the
// Gaussian envelope, g = exp(-1/2 ((ik - jk)/sk)^2 - 1/2 ((iw - jw)/sw)^2):
// for any centre c, (i - j)^2 = 2 (i - c)^2 + 2 (j - c)^2 - (k - 2c)^2, so
// a = exp(-((ik - ck)/sk)^2 - ((iw - cw)/sw)^2) and b = exp(1/2 ((kk -
// 2ck)/sk)^2 + 1/2 ((kw - 2cw)/sw)^2).  c is a quarter of the lattice: 2c is
// the middle of the outputs' range, where b = 1, and b <= exp(E / 8) at its
// corners (E the exponent range of k_gauss_sep; e^4 for sigma_g = 0.25,
// against e^16 with c in the middle of the lattice).  A transform's rounding
// is relative to its largest values, so b_k is what it costs an output: the
// FP32 plans run it in double-float (df.cuh), whose 2^-46 leaves every output
// far below the FP32 rounding of y, FP64 plans in triple-float (tf.cuh), which
// leaves the rounding of the outputs alone.
//
// Mixed-sign interactions (Gaussian envelope): on the axis of signed omega
// the sheet's own y sits at +omega and the other sheet's at -omega (omega >=
// 1), and the sum and the difference pairs of k = (kk, kw), kw >= 1, together
// are one self-convolution of that sequence (a difference pair is i at kw +
// jw, j at -jw; the envelope is that of the signed difference).  Nw >= 3
// n_omega - 2 keeps the outputs kw < n_omega free of aliases.  At kw = 0 the
// pairs that cancel in omega do not count: those outputs are summed directly
// over the omega = 0 column.
//
// Cost, and the O(N^2) pair sum's: see conv_run (conv_launch.cuh).
#pragma once

#include <type_traits>

#include "fft.cuh"
#include "philox.cuh"

namespace srm3 {
namespace {

// Number types of a transform: T2 complex, F the real type of its factors
// (and of the twiddles' parts), Y the stored phasors and coefficients.
template <typename T2>
struct ConvNum;
template <>
struct ConvNum<float2> {
  using F = float;
  using Y2 = float2;
};
template <>
struct ConvNum<double2> {
  using F = double;
  using Y2 = double2;
};
template <>
struct ConvNum<df2> {
  using F = df;
  using Y2 = float2;
};
template <>
struct ConvNum<tf2> {
  using F = tf;
  using Y2 = double2;
};

__device__ __forceinline__ float conv_scale(float y, float a) { return y * a; }
__device__ __forceinline__ double conv_scale(double y, double a) { return y * a; }
__device__ __forceinline__ df conv_scale(float y, df a) {  // the exact product, rounded to a df
  const float p = __fmul_rn(y, a.h);
  return df(p, __fmaf_rn(y, a.l, __fmaf_rn(y, a.h, -p)));
}
__device__ __forceinline__ tf conv_scale(double y, tf a) { return tf(y) * a; }
__device__ __forceinline__ float conv_round(float v) { return v; }
__device__ __forceinline__ double conv_round(double v) { return v; }
__device__ __forceinline__ float conv_round(df v) { return v.h + v.l; }
__device__ __forceinline__ double conv_round(tf v) { return (double)v.h + ((double)v.m + (double)v.l); }
template <typename F>
__device__ __forceinline__ F conv_pow2(F v, float s) { return v * (F)s; }
__device__ __forceinline__ df conv_pow2(df v, float s) { return df(v.h * s, v.l * s); }
__device__ __forceinline__ tf conv_pow2(tf v, float s) { return tf(v.h * s, v.m * s, v.l * s); }
// the phasor rows of a row kernel follow its transforms, 16-byte aligned
__host__ __device__ constexpr size_t conv_align(size_t b) { return (b + 15) / 16 * 16; }

}  // namespace

// One launch sequence over sheet-samples [0, 2 ns) of samples n0 .. n0 + ns - 1.
struct ConvArgs {
  int nk, nw, Nk, Nw;
  int mixed;
  int n0;                       // first sample: dseeds, fac_of
  // factors of the envelope: tables over the lattice (separable bispectra),
  // or per axis (aW at signed omega index + n_omega - 1)
  const void *e, *eb;
  const void *aK, *aW, *bK, *bW;
  // sqrt(q), pure and pair factors: one plan's, or per sample (batches)
  const void *sqq, *Pk, *ck;
  const void *const *sqq_of, *const *pk_of, *const *ck_of;
  const uint64_t *dseeds;       // seeds in device memory, else SeedChunk
  void *y;                      // [2 ns][nk][nw] phasors (Y2)
  void *Z;                      // [2 ns][nk][Nw] grid rows (T2)
  void *C;                      // [2 ns][nk][nw] coefficients (Y2), of sample n0 on
  const void *twk, *tww;        // pass twiddles of lengths Nk, Nw
  double cb, sb;                // cos, sin of the biphase
  int row_lo, row_hi;           // lattice rows whose coefficients are written
  int rows;                     // lattice rows per CTA of the row kernels
};

namespace {

// log2 of the values a thread holds of a length-2^l transform: 8, fewer for
// the short transforms of small lattices, whose passes are bound by the latency
// of a thread's own instructions, more for the longest, whose threads would not
// fit in a CTA.  4 / 8 / 16 values everywhere measured, in us (pair sum with
// phases): one sample of 32 x 32 19.4 / 22.4 / 31.7, 4 mixed ones of 29 x 12 in FP64
// 37 / 46 / 67; 64 samples of 256 x 512 2213 / 1931 / 2193, 16 of 512 x 1024 2589 /
// 2561 / 2384, 64 separable ones of 256 x 512 907 / 624 / 662, 50 of 256 x 128
// 192 / 139 / 180 (202 with separate phases and 16 values).  Triple-floats: 4,
// whose passes hold 64 registers or so and need no rotations within.
template <typename T2>
__host__ __device__ constexpr int conv_lv(int l) {
  return l <= 6 || sizeof(T2) == 24 ? 2 : l <= 12 ? 3 : 4;
}
// log2 of the longest transform: a row or column has to fit in shared memory.
template <typename T2>
constexpr int kConvMaxLog2 = sizeof(T2) == 24 ? 12 : 13;
template <typename T2>
__host__ __device__ constexpr int conv_tpt(int l) { return tx_tpt(1 << l, conv_lv<T2>(l)); }
// Threads of a row CTA at most (64 unless one row takes more; whole warps, of
// which A.rows rows are in use) and of a column CTA.
template <typename T2>
__host__ __device__ constexpr int conv_row_threads(int lw) {
  return conv_tpt<T2>(lw) >= 64 ? conv_tpt<T2>(lw) : 64;
}
// The column pass holds its CTAs to 64 registers a thread, 1024 threads per SM:
// with the 68 that lengths past 512 took, one CTA of 512 was all an SM held, its
// loads, transforms and stores one after the other.  Up to length 512 the CTAs
// are of 256 threads, so that four of them overlap.  512 threads without the
// limit / with it / 256 threads with it, ms: 16 samples of 512 x 1024 2.60 / 2.31 /
// 2.34, 256 x 512 plan and 64 samples 3.58 / 3.54 / 3.52, 32 uneven spectra 2.46 /
// 2.46 / 2.39; with the two as here 2.31, 3.51 and 2.39.  (Length 4096 would
// spill.)
template <typename T2>
__host__ __device__ constexpr int conv_col_threads(int lk) {
  return conv_tpt<T2>(lk) > 512 ? conv_tpt<T2>(lk) : lk <= 9 ? 256 : 512;
}
// (Triple-floats: no limit but the CTA's own.)
template <typename T2>
__host__ __device__ constexpr int conv_col_ctas(int lk) {
  return lk <= 11 && sizeof(T2) != 24 ? 1024 / conv_col_threads<T2>(lk) : 1;
}

template <typename T2>
__device__ __forceinline__ typename ConvNum<T2>::F conv_a(const ConvArgs &A, int kk, int m) {
  using F = typename ConvNum<T2>::F;
  if (A.e) return static_cast<const F *>(A.e)[(size_t)kk * A.nw + m];
  return static_cast<const F *>(A.aK)[kk] * static_cast<const F *>(A.aW)[A.nw - 1 + m];
}
template <typename T2>
__device__ __forceinline__ typename ConvNum<T2>::F conv_b(const ConvArgs &A, int kk, int kw) {
  using F = typename ConvNum<T2>::F;
  if (A.eb) return static_cast<const F *>(A.eb)[(size_t)kk * A.nw + kw];
  return static_cast<const F *>(A.bK)[kk] * static_cast<const F *>(A.bW)[kw];
}
template <typename T>
__device__ __forceinline__ const T *conv_table(const void *one, const void *const *of, int n) {
  return static_cast<const T *>(of ? of[n] : one);
}

// The phasors y = sqrt(q) z of lattice row kk on sheet s of sample n into
// row[kw] (shared; 0 at k = 0, which takes part in no pair), by the row's
// tpt threads; a thread takes a Philox counter (four consecutive entries) at
// a time.  store: also to global memory, for the epilogue (k = 0 included).
template <typename Y2>
__device__ __forceinline__ void conv_phases(const ConvArgs &A, uint64_t seed, int n, int s, int kk,
                                            int tpt, int jt, Y2 *row, Y2 *store) {
  using T = decltype(Y2::x);
  const T *sqq = conv_table<T>(A.sqq, A.sqq_of, n) + (size_t)kk * A.nw;
  const uint64_t e0 = ((uint64_t)s * A.nk + kk) * A.nw;
  const int first = (int)(e0 & 3), nc = (first + A.nw + 3) / 4;
  for (int c = jt; c < nc; c += tpt) {
    const uint64_t ctr = (e0 >> 2) + c;
    const uint4 o = philox4x32_10(make_uint4((uint32_t)ctr, (uint32_t)(ctr >> 32), 0u, 0u),
                                  make_uint2((uint32_t)seed, (uint32_t)(seed >> 32)));
    const uint32_t w[4] = {o.x, o.y, o.z, o.w};
#pragma unroll
    for (int l = 0; l < 4; ++l) {
      const int kw = 4 * c + l - first;
      if (kw < 0 || kw >= A.nw) continue;
      Y2 v = phasor(w[l], T());
      const T a = sqq[kw];
      v.x *= a;
      v.y *= a;
      if (store) store[kw] = v;
      if (kk == 0 && kw == 0) v.x = v.y = 0;
      row[kw] = v;
    }
  }
}

// Pass 1: phases, z = a y along lattice row kk < n_kappa (zero-padded to Nw),
// transformed; rb rows of one sheet-sample per CTA (blockIdx.y = ss).
// Threads of rows past n_kappa take part in the barriers only.
template <int LW, typename T2, bool MIXED>
__global__ void __launch_bounds__(conv_row_threads<T2>(LW)) k_conv_rows(const ConvArgs A,
                                                                    const SeedChunk seeds) {
  using Y2 = typename ConvNum<T2>::Y2;
  extern __shared__ __align__(16) unsigned char conv_smem[];
  constexpr int Nw = 1 << LW, tpt = conv_tpt<T2>(LW), LV = conv_lv<T2>(LW);
  const int rb = blockDim.x / tpt;  // rows that fit; A.rows of them are in use
  const int row = threadIdx.x / tpt, jt = threadIdx.x & (tpt - 1), ss = blockIdx.y;
  const int kk = blockIdx.x * A.rows + row, nw = A.nw;
  const bool live = row < A.rows && kk < A.nk;
  T2 *buf = reinterpret_cast<T2 *>(conv_smem) + row * (tx_len(Nw) + 1);
  // the row's phasors (and the other sheet's): up to Nw / 2 entries each
  Y2 *yr = reinterpret_cast<Y2 *>(conv_smem + conv_align(rb * (tx_len(Nw) + 1) * sizeof(T2))) +
           (size_t)row * (MIXED ? 2 : 1) * nw;
  T2 *out = static_cast<T2 *>(A.Z) + ((size_t)ss * A.nk + kk) * Nw;
  if (live) {
    const int n = A.n0 + (ss >> 1), s = ss & 1;
    const uint64_t seed = A.dseeds ? A.dseeds[n] : seeds.s[ss >> 1];
    conv_phases<Y2>(A, seed, n, s, kk, tpt, jt, yr,
                    static_cast<Y2 *>(A.y) + ((size_t)ss * A.nk + kk) * nw);
    if constexpr (MIXED)
      conv_phases<Y2>(A, seed, n, 1 - s, kk, tpt, jt, yr + nw, (Y2 *)nullptr);
  }
  __syncthreads();
  auto src = [&](int m) -> T2 {
    if (!live) return c_zero<T2>();
    int w = m;
    const Y2 *y = yr;
    if constexpr (MIXED) {
      if (m > Nw / 2) {  // omega = m - Nw < 0: the other sheet
        w = m - Nw;
        y = yr + nw;
      }
    }
    const int aw = w < 0 ? -w : w;
    if (aw >= nw) return c_zero<T2>();
    const Y2 yv = y[aw];
    const auto a = conv_a<T2>(A, kk, w);
    return c_make<T2>(conv_scale(yv.x, a), conv_scale(yv.y, a));
  };
  auto dst = [&](int i, T2 v) {
    if (live) out[i] = v;
  };
  stockham_passes<LW, 0, MIXED ? 0u : tx_mask_low_half<LW, LV>(), false, false, false, LV>(
      1, 0, tpt, jt, static_cast<const T2 *>(A.tww), buf, src, dst);
}

// Pass 2: TC columns of one sheet-sample per CTA, thread (c, jt) = (t mod TC,
// t / TC): the column transformed along kappa (rows >= n_kappa zero) within
// shared memory, squared and conjugated as the second transform reads it,
// transformed again, and the n_kappa rows the lattice needs stored.  In place
// in Z ([ss][n_kappa][Nw]: the grid's rows past n_kappa are zero and not
// stored).  Shared memory: colstride entries per column.
template <int LK, typename T2>
__global__ void __launch_bounds__(conv_col_threads<T2>(LK), conv_col_ctas<T2>(LK))
    k_conv_cols(int nk, int Nw, int TC, int colstride, const T2 *__restrict__ tw,
                T2 *__restrict__ Z) {
  extern __shared__ __align__(16) unsigned char conv_smem[];
  constexpr int Nk = 1 << LK, tpt = conv_tpt<T2>(LK), LV = conv_lv<T2>(LK);
  const int c = threadIdx.x & (TC - 1), jt = threadIdx.x / TC, ss = blockIdx.y;
  T2 *col = reinterpret_cast<T2 *>(conv_smem) + c * colstride;
  T2 *base = Z + (size_t)ss * nk * Nw + blockIdx.x * TC + c;
  auto src1 = [&](int kk) -> T2 {
    return kk < nk ? base[(size_t)kk * Nw] : c_zero<T2>();
  };
  auto none = [](int, T2) {};
  stockham_passes<LK, 0, tx_mask_low_half<LK, LV>(), false, true, false, LV>(1, 0, tpt, jt, tw, col,
                                                                          src1, none);
  auto src2 = [&](int i) -> T2 {
    const T2 v = col[sp16(i)];
    return c_conj(cmul(v, v));
  };
  auto dst2 = [&](int kk, T2 v) {
    if (kk < nk) base[(size_t)kk * Nw] = v;
  };
  stockham_passes<LK, 0, 0u, true, false, true, LV>(1, 0, tpt, jt, tw, col, src2, dst2);
}

// Pass 3: lattice row kk of the twice-transformed grid, transformed along
// omega; the conjugate of its entry kw over Nk Nw is the ordered
// self-convolution at (kk, kw), taken straight from the last pass.  Epilogue
// as in the O(N^2) pair sums:
//   C_k = P_k y_k + c_k e^{i beta} b_k ((z * z)_k + [k even] z_{k/2}^2) / 2.
template <int LW, typename T2, bool MIXED>
__global__ void __launch_bounds__(conv_row_threads<T2>(LW)) k_conv_out(const ConvArgs A) {
  using F = typename ConvNum<T2>::F;
  using Y2 = typename ConvNum<T2>::Y2;
  using T = decltype(Y2::x);
  extern __shared__ __align__(16) unsigned char conv_smem[];
  constexpr int Nw = 1 << LW, tpt = conv_tpt<T2>(LW), LV = conv_lv<T2>(LW);
  const int rb = blockDim.x / tpt;  // rows that fit; A.rows of them are in use
  const int row = threadIdx.x / tpt, jt = threadIdx.x & (tpt - 1), ss = blockIdx.y;
  const int kk = A.row_lo + blockIdx.x * A.rows + row, nw = A.nw;
  const bool live = row < A.rows && kk < A.row_hi;
  T2 *buf = reinterpret_cast<T2 *>(conv_smem) + row * (tx_len(Nw) + 1);
  const T2 *in = static_cast<const T2 *>(A.Z) + ((size_t)ss * A.nk + (live ? kk : 0)) * Nw;
  const Y2 *y = static_cast<const Y2 *>(A.y) + (size_t)ss * A.nk * nw;
  const int n = A.n0 + (ss >> 1);
  const T *Pk = conv_table<T>(A.Pk, A.pk_of, n), *ck = conv_table<T>(A.ck, A.ck_of, n);
  Y2 *C = static_cast<Y2 *>(A.C) + (size_t)ss * A.nk * nw;
  const float inv = 1.0f / ((float)A.Nk * (float)Nw);  // a power of two
  const T cb = (T)A.cb, sb = (T)A.sb;
  auto z_at = [&](int hk, int hw) -> T2 {
    if (hk == 0 && hw == 0) return c_zero<T2>();
    const Y2 yh = y[(size_t)hk * nw + hw];
    const F a = conv_a<T2>(A, hk, hw);
    return c_make<T2>(conv_scale(yh.x, a), conv_scale(yh.y, a));
  };
  T2 *part = buf + tx_len(Nw);  // MIXED: the kw = 0 sum of the row, past the transform
  if constexpr (MIXED) {
    T2 *psum = reinterpret_cast<T2 *>(conv_smem) + rb * (tx_len(Nw) + 1) + row * tpt;
    T2 s = c_zero<T2>();
    if (live)
      for (int a = jt; a <= kk; a += tpt) s = c_add(s, cmul(z_at(a, 0), z_at(kk - a, 0)));
    psum[jt] = s;
    __syncthreads();
    if (jt == 0) {
      s = psum[0];
      for (int j = 1; j < tpt; ++j) s = c_add(s, psum[j]);
      *part = s;
    }
    __syncthreads();
  }
  auto src = [&](int i) -> T2 { return in[i]; };
  auto dst = [&](int kw, T2 cv) {
    if (!live || kw >= nw) return;
    T2 t = c_make<T2>(conv_pow2(c_re(cv), inv), conv_pow2(-c_im(cv), inv));
    if constexpr (MIXED) {
      if (kw == 0) t = *part;
    }
    if (((kk | kw) & 1) == 0) {  // the diagonal pair {k/2, k/2}
      const T2 z = z_at(kk >> 1, kw >> 1);
      t = c_add(t, cmul(z, z));
    }
    const T ar = (T)0.5 * conv_round(c_re(t)), ai = (T)0.5 * conv_round(c_im(t));
    const size_t k = (size_t)kk * nw + kw;
    const Y2 yk = y[k];
    const T f = ck[k] * conv_round(conv_b<T2>(A, kk, kw)), P = Pk[k];
    Y2 o;
    o.x = P * yk.x + f * (ar * cb - ai * sb);
    o.y = P * yk.y + f * (ar * sb + ai * cb);
    C[k] = o;
  };
  // the upper half of the outputs is never needed: n_omega <= Nw / 2
  stockham_passes<LW, 0, 0u, false, false, true, LV>(1, 0, tpt, jt,
                                                 static_cast<const T2 *>(A.tww), buf, src, dst);
}

}  // namespace
}  // namespace srm3
