// solve.cuh - Eq. pure on the whole lattice at once, for envelopes that
// factor on i + j = k (g^2 = a_i^2 a_j^2 b_k^2): the sums of every point by one
// real 2-D FFT self-convolution per iteration, instead of level after level.
// Included by the solve_*.cu units.
//
// With h = a^2 q, q = 1/(1 - s) (0 where S = 0, h = 0 at the origin) and
//   g_k = b_k^2 sum_{Pi(k)} h_i h_j,   s = X g,   X = eps^2 dk dw,
// the tables of Eq. pure are the fixed point of s -> X g(s).
//  * Given X (a fixed eps): plain iterations from s = 0.  A point's sum takes
//    lower points only, so the error's dependence is strictly triangular and
//    the iterations converge faster than geometrically (about ten).
//  * Given the target of max_k s: X = target / max_k g at every iteration.  The
//    normalisation turns the search for eps into the same iteration, whose one
//    slow mode is X itself; it overshoots by a factor of about -0.45.  Moving s
//    3/4 of the way to X g (damping) converges at 0.25-0.3 an iteration, about
//    20 iterations to 3e-12; Anderson's mixing of the last three (J. ACM 12,
//    1965; solve_mix) takes 9-16 for the Gaussian envelope, whatever the lattice
//    (numpy simulation, 17 x 300 to 128 x 128, targets 0.15-0.95; 10 to 14
//    measured at 0.28-0.53).  Tables of a separable bispectrum keep the damping:
//    their weight can sit in a few points that the fit does not see (the
//    wind-field envelope on 94 x 603: 24 iterations to 1e-8 against about 14).
//    So do iterations past kSolveMixIt.  The last g gives X and s = X g meets
//    the target by construction: a move in X to first order.
//    256 x 512 plan and 64 samples 3.42 -> 3.29 ms, 40 x 70 mixed plan and 16
//    samples 864 -> 739 us, 32 x 32 FP64 plan and sample 817 -> 801 us.
// Iterations that do not converge (extreme targets with sparse supports), and
// sums close to 1 (kSolveTop), leave the plan to the level passes
// (recursion.cuh).
//
// The convolution.  h is real: its omega axis is packed two to a complex
// entry, z(m) = h(2m) + i h(2m + 1), on a zero-padded nk x M grid (M = Nw / 2,
// powers of two Nk >= 2 nk - 1, Nw >= 2 nw - 1, or 3 nw - 2 on the signed axis of
// mixed interactions).  With Z the transform of z, E and O those of the even
// and odd parts and W = e^{2 pi i f / M},
//   O(f1, f) = -i (Z(f1, f) - conj Z(-f1, -f)) / 2,
//   V = Z^2 + (1 + W) O^2 = E^2 + W O^2 + 2 i E O
// is the transform of c(2m) + i c(2m + 1), c = h * h.  Per iteration:
// k_solve_rows (s, h, row transforms), k_solve_cols (column pairs f and M - f:
// transform, V, transform back), k_solve_out (rows back, g and its maximum);
// the second transforms are conj(G(conj(V))) as in conv.cuh.
//
// Rounding.  A transform's error is relative to its largest values, here the
// largest pair sums, and a point multiplies it by b_k^2 / b^2 there: for the
// Gaussian envelope, centred at a quarter of the lattice as in conv.cuh, at
// most e^{E/4} (e^8 for sigma_g = 0.25) at the lattice's corners.  In
// double-float (the search, and the tables of FP32 plans with the Gaussian
// envelope) s is good to ~1e-11 there and 1e-14 in the middle; where tables were
// those of FP64 passes the solve finishes in triple-float, whose rounding is below
// FP64's everywhere.  (In FP64, which takes the FP64 pipe longer, the sums of the
// wind-field envelope were off by 2.7e-14 on 256 x 128, and by 9e-13 on 486 x 202.)
// The points with few pairs, whose sums are small, are summed directly at the end
// (k_solve_low), which keeps them accurate relative to themselves.
#pragma once

#include "fft.cuh"

namespace srm3 {

constexpr int kSolveMaxIt = 96;
constexpr int kSolveMixIt = 40;       // iterations with Anderson mixing at most
constexpr int kSolveMixPoints = 256;  // lattice points its coefficients are fitted on
// An iterate's s enters q as min(s, kSolveClip).  Points above it at the fixed
// point would feed others a q too small: a solve counts only where every s ends
// below kSolveTop (the margin is far above the rounding of s), and targets from
// there on go to the level passes at once.
constexpr double kSolveClip = 0.99, kSolveTop = 0.9899;
// A transform's rounding is relative to sum h^2 (the largest sum there can be, by
// Cauchy and Schwarz), times b_k^2 at a point.  Supports whose pairs are few or
// weak, or that have none, can leave max_k g anywhere below that, down to the
// rounding itself.  A solve counts where X max b^2 sum h^2 stays below kSolveSpread
// (double-float, Gaussian envelope: 3e4 at most on full lattices and on ones with
// nine of ten points empty, sigma_g >= 0.2237) or kSolveSpreadSep (separable
// tables, finished in triple-float: 3 times the number of points); where X comes
// from rounding alone it is 2^36 and above.
constexpr double kSolveSpread = 0x1p22, kSolveSpreadSep = 0x1p26;
constexpr double kSolveH2Unit = 0x1p-24;

// Control words of a solve, zeroed before it: the bits of max_k g and of the
// largest change of s, per iteration; then the results (k_solve_final).
struct SolveCtl {
  unsigned long long maxg[kSolveMaxIt];
  unsigned long long chg[kSolveMaxIt];
  double X;                    // eps^2 dk dw
  unsigned long long gmax;     // bits: max_k g, the directly summed points' included
  unsigned long long max_sb2;  // bits
  unsigned long long hmax, bmax;  // bits: max h and max b_k^2 where S > 0
  unsigned long long h2;       // sum of (h / hmax)^2, in units of kSolveH2Unit
  int last;                    // the iteration g is from
  int converged;
  int err;                     // some sum_b2 >= 1
};

struct SolveArgs {
  int nk, nw, Nk, M;
  int mixed;
  int rows;                 // lattice rows per CTA of the row kernels
  const double *S;
  // a^2 and b^2: tables over the lattice (separable bispectra), or per axis
  // (aW at signed omega index + nw - 1), in the transform's real type F
  const void *e2, *b2;
  const void *aK, *bK, *aW, *bW;
  // F [nk][nw]: g of iteration n in g[n % 3]; the iterate of iteration n in s[n & 3]
  // (of -1, in s[3]: the warm start)
  void *g[3], *s[4];
  void *Z;                  // [nk][M] complex
  const void *twk, *twm, *twz;  // pass twiddles of Nk and M; e^{pi i m / M}
  SolveCtl *ctl;
  double target;            // > 0: of max_k s; else X is given
  double X, w, tol, accept;
  int warm;                 // s[3] holds the first iterate (else it is 0)
  int hold;                 // the first updates take X as given, undamped
};

namespace {

__device__ __forceinline__ double as_double(unsigned long long b) {
  return __longlong_as_double((long long)b);
}
// Whether iteration it was the last that counts: its change within tol, or
// within accept and no longer falling (the transform's rounding: it keeps the
// sums of some bispectra moving by a few 1e-11 in double-float, at points of large
// b_k^2, which are summed directly at the end).  The words of skipped iterations
// stay 0.
__device__ __forceinline__ bool solve_last(const SolveArgs &A, int it) {
  if (it < A.hold + 1) return false;
  const double c = as_double(A.ctl->chg[it]);
  if (c <= A.tol) return true;
  if (it < A.hold + (A.e2 ? 2 : 4) || c > A.accept) return false;
  double m = as_double(A.ctl->chg[it - 1]);
  if (!A.e2)  // mixed iterations fall less evenly
    m = fmin(m, fmin(as_double(A.ctl->chg[it - 2]), as_double(A.ctl->chg[it - 3])));
  return c >= 0.5 * m;
}
__device__ __forceinline__ bool solve_done(const SolveArgs &A, int it) {
  return it >= 1 && solve_last(A, it - 1);
}
__device__ __forceinline__ double solve_X(const SolveArgs &A, int it) {
  if (!(A.target > 0.0) || it < A.hold) return A.X;
  const double m = as_double(A.ctl->maxg[it]);
  return m > 0.0 ? A.target / m : 0.0;
}
// S_k > 0 by its bits (an FP64 comparison would go through the FP64 pipe)
__device__ __forceinline__ bool solve_pos(const SolveArgs &A, size_t k) {
  return reinterpret_cast<const long long *>(A.S)[k] > 0;
}
template <typename F>
__device__ __forceinline__ F solve_a2(const SolveArgs &A, int kk, int w) {
  return A.e2 ? static_cast<const F *>(A.e2)[(size_t)kk * A.nw + w]
              : static_cast<const F *>(A.aK)[kk] * static_cast<const F *>(A.aW)[A.nw - 1 + w];
}
template <typename F>
__device__ __forceinline__ F solve_b2(const SolveArgs &A, int kk, int kw) {
  return A.b2 ? static_cast<const F *>(A.b2)[(size_t)kk * A.nw + kw]
              : static_cast<const F *>(A.bK)[kk] * static_cast<const F *>(A.bW)[kw];
}
// The per-point arithmetic stays in the transform's type: an FP64 operation
// takes a warp 16 cycles of its SM's FP64 pipe, and the first form of these
// kernels, with s, g and h in FP64, spent 25 us a launch on a 32 x 32 lattice.
// q from s: 1/(1 - s), s kept below kSolveClip while the iterations are on their
// way; a fixed point that reaches it is not Eq. pure's (kSolveTop).
__device__ __forceinline__ df solve_q(df s) {
  const df d = s.h < (float)kSolveClip ? df(1.0f, 0.0f) - s : df(1.0 - kSolveClip);
  const float r = __frcp_rn(d.h);  // one Newton step on it: error r (1 - d r)^2
  const float e = __fmaf_rn(-d.l, r, __fmaf_rn(-d.h, r, 1.0f));
  return df(r, __fmul_rn(r, e));
}
__device__ __forceinline__ tf solve_q(tf s) {
  const tf one(1.0f, 0.0f, 0.0f), d = s.h < (float)kSolveClip ? one - s : tf(1.0 - kSolveClip);
  const tf r0(__frcp_rn(d.h), 0.0f, 0.0f);  // two Newton steps
  const tf r1 = r0 + r0 * (one - d * r0);
  return r1 + r1 * (one - d * r1);
}
__device__ __forceinline__ df solve_num(float v, df) { return df(v, 0.0f); }
__device__ __forceinline__ tf solve_num(float v, tf) { return tf(v, 0.0f, 0.0f); }
__device__ __forceinline__ double solve_real(df v) { return (double)v.h + (double)v.l; }
__device__ __forceinline__ double solve_real(tf v) {
  return (double)v.h + ((double)v.m + (double)v.l);
}
// v, 0 if negative, its parts not overlapping (so that h orders first)
__device__ __forceinline__ df solve_clip(df v) {
  const float h = __fadd_rn(v.h, v.l), l = __fsub_rn(v.l, __fsub_rn(h, v.h));
  return h > 0.0f ? df(h, l) : df(0.0f, 0.0f);
}
__device__ __forceinline__ tf solve_clip(tf v) {
  float t, e, m, l;
  t = two_sum(v.m, v.l, e);
  const float h = two_sum(v.h, t, m);
  m = two_sum(m, e, l);
  return h > 0.0f ? tf(h, m, l) : tf(0.0f, 0.0f, 0.0f);
}
__device__ __forceinline__ df solve_max(df a, df b) {
  return (b.h > a.h || (b.h == a.h && b.l > a.l)) ? b : a;
}
__device__ __forceinline__ tf solve_max(tf a, tf b) {
  return (b.h > a.h || (b.h == a.h && (b.m > a.m || (b.m == a.m && b.l > a.l)))) ? b : a;
}
__device__ __forceinline__ float solve_abs(df v) { return fabsf(v.h + v.l); }
__device__ __forceinline__ float solve_abs(tf v) { return fabsf(v.h + (v.m + v.l)); }

__device__ __forceinline__ void warp_atomic_max(unsigned long long *p, double v) {
  for (int o = 16; o > 0; o >>= 1) v = fmax(v, __shfl_xor_sync(0xffffffffu, v, o));
  if ((threadIdx.x & 31) == 0 && v > 0.0)
    atomicMax(p, (unsigned long long)__double_as_longlong(v));
}

// Anderson mixing.  With G_n = X_n g(s_n), f_n = G_n - s_n, the next iterate is
// G_n + c1 (G_{n-1} - G_n) + c2 (G_{n-2} - G_n), the coefficients those that
// make the same combination of the f smallest.  The few slow modes are smooth: a
// fit on 256 points spread over the lattice (golden-ratio steps) takes the
// iterations that one over all points does (numpy), and every CTA makes it for
// itself, in the same order, with no reduction over the grid.  past: 1 or 2.
template <typename F>
__device__ __forceinline__ void solve_mix(const SolveArgs &A, int n, int past, float &c1, float &c2) {
  const unsigned nl = (unsigned)A.nk * A.nw;
  const F X0 = F(solve_X(A, n)), X1 = F(solve_X(A, n - 1)), X2 = F(past > 1 ? solve_X(A, n - 2) : 0.0);
  const F *g0 = static_cast<const F *>(A.g[n % 3]), *g1 = static_cast<const F *>(A.g[(n + 2) % 3]);
  const F *g2 = static_cast<const F *>(A.g[(n + 1) % 3]);
  const F *s0 = static_cast<const F *>(A.s[n & 3]), *s1 = static_cast<const F *>(A.s[(n - 1) & 3]);
  const F *s2 = static_cast<const F *>(A.s[(n - 2) & 3]);
  float v[5] = {0.f, 0.f, 0.f, 0.f, 0.f};  // d1.d1, d1.d2, d2.d2, d1.f0, d2.f0
  for (int j = threadIdx.x; j < kSolveMixPoints; j += blockDim.x) {
    // point floor(nl frac((j + 1/2) / golden ratio))
    const unsigned k = __umulhi((unsigned)(2 * j + 1) * 1327217885u, nl);
    const float f0 = (float)solve_real(X0 * g0[k] - s0[k]);
    const float d1 = f0 - (float)solve_real(X1 * g1[k] - s1[k]);
    const float d2 = past > 1 ? f0 - (float)solve_real(X2 * g2[k] - s2[k]) : 0.f;
    v[0] = fmaf(d1, d1, v[0]);
    v[1] = fmaf(d1, d2, v[1]);
    v[2] = fmaf(d2, d2, v[2]);
    v[3] = fmaf(d1, f0, v[3]);
    v[4] = fmaf(d2, f0, v[4]);
  }
  __shared__ float part[32][5];
#pragma unroll
  for (int i = 0; i < 5; ++i)
    for (int o = 16; o > 0; o >>= 1) v[i] += __shfl_xor_sync(0xffffffffu, v[i], o);
  if (blockDim.x > 32) {
    if ((threadIdx.x & 31) == 0)
      for (int i = 0; i < 5; ++i) part[threadIdx.x >> 5][i] = v[i];
    __syncthreads();
#pragma unroll
    for (int i = 0; i < 5; ++i) {
      v[i] = 0.f;
      for (unsigned w = 0; w < blockDim.x / 32; ++w) v[i] += part[w][i];
    }
  }
  c1 = c2 = 0.f;
  const float det = v[0] * v[2] - v[1] * v[1];
  if (past > 1 && det > 1e-6f * v[0] * v[2]) {
    c1 = (v[3] * v[2] - v[4] * v[1]) / det;
    c2 = (v[4] * v[0] - v[3] * v[1]) / det;
  } else if (v[0] > 0.f) {
    c1 = v[3] / v[0];
  }
  const float m = fmaxf(fabsf(c1), fabsf(c2));
  if (!(m <= 16.f)) c1 = c2 = 0.f;  // (NaN too)
}

// log2 of the values a thread holds of a length-2^l transform: 4 of them where
// the transform's threads then fit in a CTA twice over.  A pass is short --
// a lattice has a few points per thread of the GPU -- and bound by the latency
// of a thread's own instructions, ~30 a point and level: with 16 values a
// thread an iteration took 53 us on 32 x 32 and 92 us on 256 x 512.
__host__ __device__ constexpr int solve_lv(int l) { return l <= 10 ? 2 : 3; }
__host__ __device__ constexpr int solve_tpt(int l) { return tx_tpt(1 << l, solve_lv(l)); }

// Threads of a row CTA: whole warps of tpt threads a row, 64 at most unless
// one row takes more; A.rows of its rows are in use (fewer than fit, so that a
// small lattice spreads over the SMs).
__host__ __device__ constexpr int solve_row_threads(int lm) {
  return solve_tpt(lm) >= 64 ? solve_tpt(lm) : 64;
}
__host__ __device__ constexpr int solve_col_threads(int lk) {
  return 2 * solve_tpt(lk) > 256 ? 2 * solve_tpt(lk) : 256;
}

// The kernels of an iteration are launched as programmatic dependents
// (solve_launch.cuh): the next one's CTAs are placed while this one runs and wait
// here until it has completed and its writes are visible.
__device__ __forceinline__ void solve_turn() {
  asm volatile("griddepcontrol.launch_dependents;");
  asm volatile("griddepcontrol.wait;" ::: "memory");
}

// Rows: the iterate s (from g of the iteration before), h and its transform.
template <int LM, typename T2>
__global__ void __launch_bounds__(solve_row_threads(LM)) k_solve_rows(const SolveArgs A, int it) {
  using F = typename RealOf<T2>::type;
  solve_turn();
  if (solve_done(A, it)) return;
  extern __shared__ __align__(16) unsigned char solve_smem[];
  constexpr int M = 1 << LM, tpt = solve_tpt(LM), LV = solve_lv(LM);
  const int row = threadIdx.x / tpt, jt = threadIdx.x & (tpt - 1);
  const int kk = blockIdx.x * A.rows + row, nw = A.nw;
  const bool live = row < A.rows && kk < A.nk;
  T2 *buf = reinterpret_cast<T2 *>(solve_smem) + row * (tx_len(M) + 1);
  T2 *out = static_cast<T2 *>(A.Z) + (size_t)kk * M;
  // iteration n's results make the iterate of it = n + 1
  const int n = it - 1;
  const bool mix = A.target > 0.0 && !A.e2 && it < kSolveMixIt;
  const int past = mix && n > A.hold ? min(n - A.hold, 2) : 0;
  float c1 = 0.f, c2 = 0.f;
  if (past > 0) solve_mix<F>(A, n, past, c1, c2);
  const F m1 = solve_num(c1, F()), m2 = solve_num(c2, F());
  const F X = F(it > 0 ? solve_X(A, n) : 0.0);
  const F X1 = F(past > 0 ? solve_X(A, n - 1) : 0.0), X2 = F(past > 1 ? solve_X(A, n - 2) : 0.0);
  const F damp = F(it <= A.hold || mix ? 1.0 : A.w);
  const F *s_in = static_cast<const F *>(A.s[(it + 3) & 3]);
  const F *g = static_cast<const F *>(A.g[(it + 2) % 3]), *g1 = static_cast<const F *>(A.g[(it + 1) % 3]);
  const F *g2 = static_cast<const F *>(A.g[it % 3]);
  F *s_out = static_cast<F *>(A.s[it & 3]);
  float chg = 0.0f;
  auto h_at = [&](int p) -> F {  // position p of the row: omega = p, or p - 2 M
    int w = p;
    if (A.mixed && p > M) w = p - 2 * M;
    const int kw = w < 0 ? -w : w;
    if (!live || kw >= nw) return F(0.0);
    const size_t k = (size_t)kk * nw + kw;
    F s = F(0.0);
    if (it == 0) {
      if (A.warm) s = s_in[k];
    } else if (past > 0) {
      const F G = X * g[k];
      s = G + m1 * (X1 * g1[k] - G);
      if (past > 1) s = s + m2 * (X2 * g2[k] - G);
      s = solve_clip(s);
      if (w >= 0) chg = fmaxf(chg, solve_abs(s - s_in[k]));
    } else {
      const F s0 = s_in[k], d = (X * g[k] - s0) * damp;
      s = s0 + d;
      if (w >= 0) chg = fmaxf(chg, solve_abs(d));
    }
    if (w >= 0) s_out[k] = s;
    return (solve_pos(A, k) && k != 0) ? solve_a2<F>(A, kk, w) * solve_q(s) : F(0.0);
  };
  auto src = [&](int m) -> T2 {
    const F re = h_at(2 * m);
    return c_make<T2>(re, h_at(2 * m + 1));
  };
  auto dst = [&](int i, T2 v) {
    if (live) out[i] = v;
  };
  stockham_passes<LM, 0, 0u, false, false, false, LV>(1, 0, tpt, jt, static_cast<const T2 *>(A.twm), buf, src, dst);
  if (it > 0) warp_atomic_max(&A.ctl->chg[it], (double)chg);
}

// Column pairs f = p and M - p, p = 0 .. M / 2, TC of them per CTA: forward, V,
// and back, in place.
template <int LK, typename T2>
__global__ void __launch_bounds__(solve_col_threads(LK)) k_solve_cols(const SolveArgs A, int it,
                                                                      int TC, int colstride) {
  solve_turn();
  if (solve_done(A, it)) return;
  extern __shared__ __align__(16) unsigned char solve_smem[];
  constexpr int Nk = 1 << LK, tpt = solve_tpt(LK), LV = solve_lv(LK);
  const int M = A.M, nk = A.nk;
  const int c = threadIdx.x & (2 * TC - 1), jt = threadIdx.x / (2 * TC);
  const int p = blockIdx.x * TC + (c & (TC - 1));
  const bool live = p <= M / 2;
  const int f = c < TC ? p : (M - p) & (M - 1);
  T2 *col = reinterpret_cast<T2 *>(solve_smem) + c * colstride;
  const T2 *other = reinterpret_cast<T2 *>(solve_smem) + (c ^ TC) * colstride;
  T2 *base = static_cast<T2 *>(A.Z) + f;
  const T2 *tw = static_cast<const T2 *>(A.twk);
  auto src1 = [&](int kk) -> T2 {
    return live && kk < nk ? base[(size_t)kk * M] : c_zero<T2>();
  };
  auto none = [](int, T2) {};
  stockham_passes<LK, 0, tx_mask_low_half<LK, LV>(), false, true, false, LV>(1, 0, tpt, jt, tw, col,
                                                                          src1, none);
  using F = typename RealOf<T2>::type;
  T2 w1 = c_zero<T2>();  // 1 + e^{2 pi i f / M}; 0 at f = M / 2
  if (live && p < M / 2) {
    const T2 t = static_cast<const T2 *>(A.twz)[2 * p];
    w1 = c_make<T2>(c_re(t) + F(1.0), c >= TC && p > 0 ? -c_im(t) : c_im(t));
  }
  auto src2 = [&](int i) -> T2 {  // conj V
    const T2 z = col[sp16(i)], y = other[sp16((Nk - i) & (Nk - 1))];
    // -i (z - conj y) / 2
    const T2 o = c_make<T2>((c_im(z) + c_im(y)) * F(0.5), (c_re(y) - c_re(z)) * F(0.5));
    return c_conj(c_add(cmul(z, z), cmul(w1, cmul(o, o))));
  };
  auto dst2 = [&](int kk, T2 v) {
    if (live && kk < nk) base[(size_t)kk * M] = v;
  };
  stockham_passes<LK, 0, 0u, true, false, true, LV>(1, 0, tpt, jt, tw, col, src2, dst2);
}

// Rows back: g_k = b_k^2 ((h * h)_k + [k even] h_{k/2}^2) / 2 and its maximum.
// Mixed interactions at kw = 0: the pairs that cancel in omega do not count,
// the row's omega = 0 pairs are summed directly.
template <int LM, typename T2>
__global__ void __launch_bounds__(solve_row_threads(LM)) k_solve_out(const SolveArgs A, int it) {
  using F = typename RealOf<T2>::type;
  solve_turn();
  if (solve_done(A, it)) return;
  extern __shared__ __align__(16) unsigned char solve_smem[];
  constexpr int M = 1 << LM, tpt = solve_tpt(LM), LV = solve_lv(LM);
  const int row = threadIdx.x / tpt, jt = threadIdx.x & (tpt - 1);
  const int kk = blockIdx.x * A.rows + row, nw = A.nw;
  const bool live = row < A.rows && kk < A.nk;
  T2 *buf = reinterpret_cast<T2 *>(solve_smem) + row * (tx_len(M) + 1);
  const T2 *in = static_cast<const T2 *>(A.Z) + (size_t)(live ? kk : 0) * M;
  const F *s = static_cast<const F *>(A.s[it & 3]);
  F *g = static_cast<F *>(A.g[it % 3]);
  const F half_inv = F(0.5 / ((double)A.Nk * M)), half = F(0.5);  // powers of two
  F mx = F(0.0);
  auto h_of = [&](int hk, int hw) -> F {
    const size_t k = (size_t)hk * nw + hw;
    return (solve_pos(A, k) && k != 0) ? solve_a2<F>(A, hk, hw) * solve_q(s[k]) : F(0.0);
  };
  F c0 = F(0.0);
  if (A.mixed) {
    F *part = reinterpret_cast<F *>(reinterpret_cast<T2 *>(solve_smem) +
                                    (blockDim.x / tpt) * (tx_len(M) + 1)) + row * tpt;
    F t = F(0.0);
    if (live)
      for (int a = jt; a <= kk; a += tpt) t = t + h_of(a, 0) * h_of(kk - a, 0);
    part[jt] = t;
    __syncthreads();
    if (jt == 0)
      for (int j = 0; j < tpt; ++j) c0 = c0 + part[j];
    c0 = c0 * half;
  }
  auto put = [&](int kw, F c) {  // c: half the ordered sum
    if (!live || kw >= nw) return;
    const size_t k = (size_t)kk * nw + kw;
    if (A.mixed && kw == 0) c = c0;
    if (((kk | kw) & 1) == 0) {
      const F h = h_of(kk >> 1, kw >> 1);
      c = c + h * h * half;
    }
    // clipped: rounding below zero where every term is zero
    const F v = solve_pos(A, k) ? solve_clip(solve_b2<F>(A, kk, kw) * c) : F(0.0);
    g[k] = v;
    mx = solve_max(mx, v);
  };
  auto src = [&](int i) -> T2 { return in[i]; };
  auto dst = [&](int m, T2 v) {
    put(2 * m, c_re(v) * half_inv);
    put(2 * m + 1, -c_im(v) * half_inv);
  };
  stockham_passes<LM, 0, 0u, false, false, true, LV>(1, 0, tpt, jt, static_cast<const T2 *>(A.twm),
                                                 buf, src, dst);
  warp_atomic_max(&A.ctl->maxg[it], solve_real(mx));
}

}  // namespace
}  // namespace srm3
