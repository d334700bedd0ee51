// Philox4x32-10 (Salmon, Moraes, Dror, Shaw, SC'11): ten rounds of two
// 32x32->64 multiplications with the Weyl key schedule.  Device-side
// implementation used for the features (Sec. 2.2) and the sketches (Sec. 4.1).
#pragma once
#include <stdint.h>

__device__ __forceinline__ void philox4x32_10(uint32_t c[4], uint32_t k0, uint32_t k1) {
#pragma unroll
  for (int r = 0; r < 10; ++r) {
    if (r) {
      k0 += 0x9E3779B9u;
      k1 += 0xBB67AE85u;
    }
    const uint32_t hi0 = __umulhi(0xD2511F53u, c[0]);
    const uint32_t lo0 = 0xD2511F53u * c[0];
    const uint32_t hi1 = __umulhi(0xCD9E8D57u, c[2]);
    const uint32_t lo1 = 0xCD9E8D57u * c[2];
    const uint32_t n0 = hi1 ^ c[1] ^ k0;
    const uint32_t n2 = hi0 ^ c[3] ^ k1;
    c[0] = n0;
    c[1] = lo1;
    c[2] = n2;
    c[3] = lo0;
  }
}

// 53-bit uniform on [0,1) from two words: ((a >> 5) * 2^26 + (b >> 6)) * 2^-53.
__device__ __forceinline__ double uniform53(uint32_t a, uint32_t b) {
  const uint64_t v = ((uint64_t)(a >> 5) << 26) + (uint64_t)(b >> 6);
  return (double)v * 0x1p-53;
}

// Nearest bfloat16 (ties to even) of a double in the bf16 normal range,
// returned as the 16 stored bits.
__device__ __forceinline__ uint16_t bf16_bits_rne(double x) {
  uint64_t b = (uint64_t)__double_as_longlong(x);
  b = (b + 0x0FFFFFFFFFFFull + ((b >> 45) & 1ull)) & ~((1ull << 45) - 1ull);
  const double r = __longlong_as_double((long long)b);
  const float f = (float)r;  // exact: r has 8 significant bits
  return (uint16_t)(__float_as_uint(f) >> 16);
}

__device__ __forceinline__ double bf16_bits_to_double(uint16_t h) {
  return (double)__uint_as_float(((uint32_t)h) << 16);
}

// Gaussian sketch entries rounded to the grid 2^-4: (rint(16 z0), rint(16 z1))
// for the Box-Muller pair z0 = r cos(t), z1 = r sin(t), r = sqrt(-2 log(w)),
// w = 1 - u1, t = 2 pi u2, by definition evaluated in FP64 and then rounded.
__device__ __forceinline__ void gauss_pair_q16_exact(const uint32_t c[4], float* d0, float* d1) {
  const double u1 = uniform53(c[0], c[1]);
  const double u2 = uniform53(c[2], c[3]);
  const double w = 1.0 - u1;  // exact
  const double rad = sqrt(-2.0 * log(w));
  const double th = 6.283185307179586 * u2;
  *d0 = (float)rint(16.0 * (rad * cos(th)));
  *d1 = (float)rint(16.0 * (rad * sin(th)));
}

// The same integers from FP32 with the hardware's log2, square root, sine and
// cosine; false where 16 z lies too near a rounding tie to be sure (0.2 % of
// the pairs) or w is below 2^-12.  No FP64 instruction (31 ns each on GB300).
// A tie needs |16 z| near 1/2 or more, so r >= 1/32 (below, 16 r < 1/2).  Errors of
// 16 z there: w from its top 32 bits, 1.2e-7 relative for w >= 1/2 and 6e-7 at most;
// log2 2^-22 absolute on [0.5, 2], 2 ulp elsewhere; so L = r^2 is within 8e-7 (L <=
// 1.4) or 5e-7 L, and 16 r within 8 dL / r <= 2.1e-4; the square root adds 16 r
// 2^-22; sine and cosine on [-pi, pi] within 6e-7 and their argument within 4e-7,
// times 16 r <= 66 (w >= 2^-12): 7e-5 where the first term is below 2e-5.  Below
// 2.5e-4 in all, half the margin of 5e-4.  For computed r < 0.01, r^2 is off by 8e-7
// at most, |16 z| < 0.2 and both are 0.
__device__ __forceinline__ bool gauss_pair_q16_fast(const uint32_t c[4], float* d0, float* d1) {
  const uint32_t wt = ~(((c[0] >> 5) << 5) | (c[1] >> 27));  // top 32 bits of 2^53 - (53 bits of u1), less one unit
  const float w = fmaf((float)wt, 0x1p-32f, 0x1p-33f);
  const float L = -1.3862944f * __log2f(w);
  float r;
  asm("sqrt.approx.f32 %0, %1;" : "=f"(r) : "f"(fmaxf(L, 0.0f)));
  const uint32_t a = ((c[2] >> 5) << 5) | (c[3] >> 27);  // top 32 bits of u2
  const float x = (float)(int)(a ^ 0x80000000u) * 1.4629180792671596e-9f;  // 2 pi (u2 - 1/2)
  const float r16 = -16.0f * r;  // cos(t) = -cos(x), sin(t) = -sin(x)
  const float t0 = r16 * __cosf(x), t1 = r16 * __sinf(x);
  const float q0 = rintf(t0), q1 = rintf(t1);
  const bool zero = r < 0.01f;
  *d0 = zero ? 0.0f : q0;
  *d1 = zero ? 0.0f : q1;
  const bool safe = fabsf(fabsf(t0 - q0) - 0.5f) > 5e-4f && fabsf(fabsf(t1 - q1) - 0.5f) > 5e-4f;
  return wt >= (1u << 20) && (zero || safe);
}

__device__ __forceinline__ void gauss_pair_q16(const uint32_t c[4], float* d0, float* d1) {
  if (!gauss_pair_q16_fast(c, d0, d1)) gauss_pair_q16_exact(c, d0, d1);
}
