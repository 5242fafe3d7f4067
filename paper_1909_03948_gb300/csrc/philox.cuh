// philox.cuh -- the sampler's generator.
//
// Philox4x32-10 (Salmon, Moraes, Dror, Shaw, SC'11): 4 x 32-bit counter, 2 x 32-bit
// key, 10 rounds of  (c0,c1,c2,c3) <- (hi(M1 c2)^c1^k0, lo(M1 c2), hi(M0 c0)^c3^k1,
// lo(M0 c0))  with the key bumped by the Weyl constants between rounds.
// Normal t of sample j: call g = t/4 with counter (g, g>>32, j, j>>32) and key
// (seed, seed>>32); words (x0,x1), (x2,x3) give two Box-Muller pairs with
// u = ((x >> 8) + 1/2) 2^-24, r = sqrt(-2 ln u_a), z = r cos(2 pi u_b), r sin(2 pi u_b)
// in FP32. 
#pragma once
#include <cstdint>

namespace hp {

__device__ __forceinline__ uint4 philox4x32_10(uint4 c, uint2 k) {
#pragma unroll
  for (int r = 0; r < 10; ++r) {
    const unsigned lo0 = 0xD2511F53u * c.x, hi0 = __umulhi(0xD2511F53u, c.x);
    const unsigned lo1 = 0xCD9E8D57u * c.z, hi1 = __umulhi(0xCD9E8D57u, c.z);
    c = make_uint4(hi1 ^ c.y ^ k.x, lo1, hi0 ^ c.w ^ k.y, lo0);
    k.x += 0x9E3779B9u;
    k.y += 0xBB67AE85u;
  }
  return c;
}

__device__ __forceinline__ void box_muller(unsigned xa, unsigned xb, float *z0, float *z1) {
  const float ua = ((float)(xa >> 8) + 0.5f) * 5.9604644775390625e-08f;  // 2^-24
  const float ub = ((float)(xb >> 8) + 0.5f) * 5.9604644775390625e-08f;
  const float r = sqrtf(-2.0f * logf(ua));
  const float th = 6.2831853071795864769f * ub;
  *z0 = r * cosf(th);
  *z1 = r * sinf(th);
}

}  // namespace hp
