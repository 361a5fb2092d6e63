// Quotient and square root of doubles, correctly rounded, on the integer pipe.
//
// An FP64 instruction holds a scheduler's pipe for 64 cycles on this GPU, so a
// division or square root (ten to twenty of them in a row) takes 1000 cycles or
// more.  The quotients of the two substitutions of the Hhat apply take div_rn; pivots of
// Cholesky, reflectors and tridiagonal eliminations were no faster with it.  sqrt_rn
// has no caller: it is kept with its test.  These versions use 64-bit
// integer products: a 23-bit approximation from the FP32 unit, two Newton steps
// in fixed point (62 bits), and the exact remainder, which decides the rounding to
// nearest even.  IEEE rounding leaves one possible result, so they return what the
// division and sqrt() return, bit for bit; operands or results outside the
// normal range go to the latter.
#pragma once

#include <cuda_runtime.h>
#include <math.h>
#include <stdint.h>
#include <string.h>

namespace sdpgb {

__host__ __device__ __forceinline__ uint64_t rd_bits(double x) {
#ifdef __CUDA_ARCH__
  return (uint64_t)__double_as_longlong(x);
#else
  uint64_t u;
  memcpy(&u, &x, 8);
  return u;
#endif
}
__host__ __device__ __forceinline__ double rd_double(uint64_t u) {
#ifdef __CUDA_ARCH__
  return __longlong_as_double((long long)u);
#else
  double x;
  memcpy(&x, &u, 8);
  return x;
#endif
}
__host__ __device__ __forceinline__ uint64_t rd_mulhi(uint64_t a, uint64_t b) {
#ifdef __CUDA_ARCH__
  return __umul64hi(a, b);
#else
  return (uint64_t)(((unsigned __int128)a * b) >> 64);
#endif
}
__host__ __device__ __forceinline__ int64_t rd_mulhi_s(int64_t a, int64_t b) {
#ifdef __CUDA_ARCH__
  return __mul64hi(a, b);
#else
  return (int64_t)(((__int128)a * b) >> 64);
#endif
}
// 24-bit significand of a positive float as an integer times 2^39, one more bit up
// when its exponent is above `e0` (the values here lie in [2^e0, 2^(e0 + 1)])
__host__ __device__ __forceinline__ uint64_t rd_fixed62(float f, int e0) {
#ifdef __CUDA_ARCH__
  const uint32_t u = __float_as_uint(f);
#else
  uint32_t u;
  memcpy(&u, &f, 4);
#endif
  const uint64_t m = (uint64_t)((u & 0x7FFFFFu) | 0x800000u) << 39;
  const int up = (int)(u >> 23) - 127 - e0;          // 0, rarely 1 or -1
  const uint64_t r = up > 0 ? m << 1 : (up < 0 ? m >> 1 : m);
  return r > 0x7FFFFFFFFFFFFFFFull ? 0x7FFFFFFFFFFFFFFFull : r;
}

// a / b
__host__ __device__ __forceinline__ double div_rn(double a, double b) {
  const uint64_t ua = rd_bits(a), ub = rd_bits(b);
  const int ea = (int)(ua >> 52) & 0x7FF, eb = (int)(ub >> 52) & 0x7FF;
  const uint64_t ma = (ua & 0xFFFFFFFFFFFFFull) | 0x10000000000000ull;
  const uint64_t mb = (ub & 0xFFFFFFFFFFFFFull) | 0x10000000000000ull;
  const int up = ma < mb ? 1 : 0;                    // quotient below one: one more bit
  const int E = ea - eb + 1023 - up;
  if (ea == 0 || ea == 0x7FF || eb == 0 || eb == 0x7FF || E < 1 || E > 2045) return a / b;
  // R = 2^126 / (mb 2^11) in (2^62, 2^63]
  const uint64_t D = mb << 11;
  const float f = (float)(uint32_t)(D >> 40);
#ifdef __CUDA_ARCH__
  float r;
  asm("rcp.approx.ftz.f32 %0, %1;" : "=f"(r) : "f"(f));
#else
  const float r = 1.0f / f;
#endif
  int64_t R = (int64_t)rd_fixed62(r, -24);
  const int64_t one = (int64_t)1 << 62;
#pragma unroll
  for (int it = 0; it < 2; ++it) {
    const int64_t e = one - (int64_t)rd_mulhi(D, (uint64_t)R);
    R += rd_mulhi_s(R, e << 2);
    if (R < 0) R = 0x7FFFFFFFFFFFFFFFll;             // b a power of two: R is 2^63
  }
  uint64_t q = rd_mulhi(ma << 11, (uint64_t)R) >> (10 - up);   // ma 2^(52 + up) / mb, off by a unit at most
  int64_t rem = (int64_t)((ma << (52 + up)) - q * mb);          // exact: small, so modulo 2^64
  if (rem < 0) {
    q -= 1;
    rem += (int64_t)mb;
  } else if (rem >= (int64_t)mb) {
    q += 1;
    rem -= (int64_t)mb;
  }
  const int64_t tw = 2 * rem - (int64_t)mb;
  if (tw > 0 || (tw == 0 && (q & 1))) q += 1;
  return rd_double(((ua ^ ub) & 0x8000000000000000ull) | (((uint64_t)E << 52) + (q - 0x10000000000000ull)));
}

// sqrt(p)
__host__ __device__ __forceinline__ double sqrt_rn(double p) {
  const uint64_t u = rd_bits(p);
  const int eb = (int)(u >> 52);
  if (eb == 0 || eb >= 0x7FF) return sqrt(p);        // zero, subnormal, negative, infinite, NaN
  const uint64_t m = (u & 0xFFFFFFFFFFFFFull) | 0x10000000000000ull;
  const int t = eb - 1075 + 53;                      // p = (m 2^-53) 2^t
  const int odd = t & 1;
  const uint64_t X = m << (11 - odd);                // x = X 2^-64 in [1/4, 1), p = x 2^(t + odd)
  const int h = (t + odd) / 2;                       // t + odd is even
  const float f = (float)(uint32_t)(X >> 40);
#ifdef __CUDA_ARCH__
  float y;
  asm("rsqrt.approx.ftz.f32 %0, %1;" : "=f"(y) : "f"(f));
#else
  const float y = 1.0f / sqrtf(f);
#endif
  int64_t Y = (int64_t)rd_fixed62(y, -12);           // 1 / sqrt(x) in units of 2^-62
  const int64_t one = (int64_t)1 << 62;
#pragma unroll
  for (int it = 0; it < 2; ++it) {
    const uint64_t A = rd_mulhi(X, (uint64_t)Y);     // x Y
    const int64_t e = one - (int64_t)rd_mulhi(A << 1, (uint64_t)Y << 1);
    Y += rd_mulhi_s(Y, e << 1);
    if (Y < 0) Y = 0x7FFFFFFFFFFFFFFFll;             // x = 1/4: 1 / sqrt(x) is 2^63 of these units
  }
  uint64_t q = rd_mulhi(X, (uint64_t)Y) >> 9;        // sqrt(x) 2^53, off by a unit at most
  int64_t rem = (int64_t)((X << 42) - q * q);
  if (rem < 0) {
    q -= 1;
    rem += (int64_t)(2 * q + 1);
  } else if (rem > (int64_t)(2 * q)) {
    rem -= (int64_t)(2 * q + 1);
    q += 1;
  }
  if (rem > (int64_t)q) q += 1;                      // above q + 1/2 (a square root is never midway)
  return rd_double(((uint64_t)(h + 1022) << 52) + (q - 0x10000000000000ull));
}

}  // namespace sdpgb
