// A double as seven signed bytes and a power of two: the operand format of the products in gemm_i8.cuh, which says what it
// is for and what it costs.
#pragma once

#include "common.cuh"

namespace rrf {

constexpr int kOzS = 7;                 // digits of an operand
constexpr int kOzBN = 32;               // columns of W in a tile of the update, of Z in an image
constexpr int kOzK = 32;                // contraction indices of one instruction
constexpr int kOzChunk = 32;            // steps of kOzK with one scale of the small operand (at most 32: see oz_join)
constexpr int kOzBad = 1 << 20;         // "exponent" of a row or column that is not finite

// Magnitude as an integer that orders like it (the high word), and the exponent e with |x| < 0.996 2^e for every x up to the
// magnitude given (the largest integer of seven balanced digits is 0.99608 2^55)
__device__ __forceinline__ uint32_t oz_mag(double x) { return (uint32_t)__double2hiint(x) & 0x7fffffffu; }
__device__ __forceinline__ int oz_exp(uint32_t mag) {
  if (mag >= 0x7ff00000u) return kOzBad;
  return max((int)((mag + 0x3000u) >> 20) - 1022, -960);
}
__device__ __forceinline__ double oz_pow2(int e) {      // 2^e, -1022 <= e <= 1023; NaN for the scale of what is not finite
  return e > 2000 ? __longlong_as_double(0x7ff8000000000000ll) : __hiloint2double((1023 + e) << 20, 0);
}
__device__ __forceinline__ double oz_scale(int e) { return oz_pow2(55 - min(e, 1024)); }      // to integers
// Four numbers -> a word of four bytes (x[0] in the low one) for each of the digits, most significant digit first.
// The bytes of x s rounded to an integer, 0x80 added to each: four high digits, three low ones.  `a` is x s rounded to a
// multiple of 2^24 with the high digits' bias in it (its low word counts multiples of 2^24), c what has to be added to x s to
// leave the rest beside 1.5 2^52; both are exact.
__device__ __forceinline__ void oz_words(const double (&x)[4], double s, uint32_t (&w)[kOzS]) {
  constexpr double m2 = 6755399441055744.0, m1 = m2 * 16777216.0 + 2155905152.0 * 16777216.0;     // 1.5 2^52; 1.5 2^76 + 0x80808080 2^24
  uint32_t hi[4], lo[4];
#pragma unroll
  for (int i = 0; i < 4; ++i) {
    const double a = fma(x[i], s, m1);
    const double c = (m1 + m2) - a;
    lo[i] = (uint32_t)__double2loint(fma(x[i], s, c)) + 0x808080u;
    hi[i] = (uint32_t)__double2loint(a) + (uint32_t)((int)lo[i] >> 24);
  }
  const uint32_t a = __byte_perm(hi[0], hi[1], 0x5140), b = __byte_perm(hi[2], hi[3], 0x5140);   // bytes 0, 1 of both
  const uint32_t c = __byte_perm(hi[0], hi[1], 0x7362), d = __byte_perm(hi[2], hi[3], 0x7362);   // bytes 2, 3
  w[3] = __byte_perm(a, b, 0x5410) ^ 0x80808080u;
  w[2] = __byte_perm(a, b, 0x7632) ^ 0x80808080u;
  w[1] = __byte_perm(c, d, 0x5410) ^ 0x80808080u;
  w[0] = __byte_perm(c, d, 0x7632) ^ 0x80808080u;
  const uint32_t e = __byte_perm(lo[0], lo[1], 0x5140), f = __byte_perm(lo[2], lo[3], 0x5140);
  const uint32_t g = __byte_perm(lo[0], lo[1], 0x0062), h = __byte_perm(lo[2], lo[3], 0x0062);
  w[6] = __byte_perm(e, f, 0x5410) ^ 0x80808080u;
  w[5] = __byte_perm(e, f, 0x7632) ^ 0x80808080u;
  w[4] = __byte_perm(g, h, 0x5410) ^ 0x80808080u;
}
__host__ __device__ constexpr uint32_t oz_at(uint32_t line, uint32_t k) {      // byte k of a line of an image
  return line * 32u + ((((k >> 4) ^ (line >> 2)) & 1u) << 4) + (k & 15u);
}

}  // namespace rrf
