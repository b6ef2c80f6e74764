// philox.cuh - the random phases: Philox4x32-10 words and unit phasors.
#pragma once

#include <cuda_runtime.h>
#include <stdint.h>

namespace srm3 {

// ---------------------------------------------------------------------------
// Philox4x32-10 (Salmon, Moraes, Dror & Shaw, SC'11): ten rounds of
// (hi, lo) = M * x on words 0 and 2, mixed with words 1 and 3 and the key;
// the key advances by the Weyl constants between rounds.
__device__ __forceinline__ uint4 philox4x32_10(uint4 c, uint2 k) {
#pragma unroll
  for (int r = 0; r < 10; ++r) {
    const uint32_t m0 = 0xD2511F53u, m1 = 0xCD9E8D57u;
    uint32_t hi0 = __umulhi(m0, c.x), lo0 = m0 * c.x;
    uint32_t hi1 = __umulhi(m1, c.z), lo1 = m1 * c.z;
    c = make_uint4(hi1 ^ c.y ^ k.x, lo1, hi0 ^ c.w ^ k.y, lo0);
    k.x += 0x9E3779B9u;
    k.y += 0xBB67AE85u;
  }
  return c;
}


// Unit phasor e^{i 2 pi (w + 1/2) 2^-32}.
__device__ __forceinline__ float2 phasor(uint32_t w, float) {
  float v = fmaf(__uint2float_rn(w), 0x1p-31f, 0x1p-32f);  // 2 (w + 1/2) 2^-32
  float s, c;
  sincospif(v, &s, &c);
  return make_float2(c, s);
}
__device__ __forceinline__ double2 phasor(uint32_t w, double) {
  double v = ((double)w + 0.5) * 0x1p-31;
  double s, c;
  sincospi(v, &s, &c);
  return make_double2(c, s);
}

}  // namespace srm3
