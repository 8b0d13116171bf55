// Integer (fixed-point) evaluation of exponentials, logarithms and the
// exponents of rate constants.
//
// Why: an FP64 warp instruction occupies this part's FP64 pipe for 16 cycles
// per SM (2 lanes a clock), a 32 x 32 -> 64 multiply-add (IMAD.WIDE) about
// 1.1 and a plain integer instruction 0.3 to 0.5 (measured, cycles per warp
// instruction per SM).  A Horner step in 64-bit fixed point (three
// IMAD.WIDE) therefore costs a quarter of an FP64 FMA, and its 60 or more
// significant bits leave the final rounding to binary64 as the only error
// that matters (below 0.54 ulp in all).  Against the same method in nine FP64
// operations: 53-species source terms, 1 Mi states, 35.8 -> 22.3 ms; CSR
// Jacobian, 256 ki states, 22.8 -> 19.9 ms; VJP, 64 ki states, 10.3 -> 8.8 ms.
//
// Method: table-driven reduction after P. T. P. Tang, "Table-driven
// implementation of the exponential function in IEEE floating-point
// arithmetic", ACM TOMS 15 (1989), in base 2:
//   2^(n + j/256 + f) = 2^n T_j (1 + f c1 + f^2 c2 + .. + f^5 c5),
//   0 <= f < 2^-8, c_k = (ln 2)^k / k! (Taylor; truncation below 2^-60),
// with T_j = 2^(j/256) and the polynomial in unsigned fixed point.
#pragma once

#include <cstdint>

#include <cuda_runtime.h>

namespace pj {

// high 64 bits of a b, short of the exact value by at most 1 (the low
// partial product is left out)
__host__ __device__ __forceinline__ uint64_t mulhi_approx(uint64_t a, uint64_t b) {
  const uint32_t a0 = (uint32_t)a, a1 = (uint32_t)(a >> 32), b0 = (uint32_t)b, b1 = (uint32_t)(b >> 32);
  const uint64_t u = (uint64_t)a0 * b1;
  const uint64_t v = (uint64_t)a1 * b0 + (uint32_t)u;
  return (uint64_t)a1 * b1 + (u >> 32) + (v >> 32);
}

__host__ __device__ __forceinline__ uint32_t mulhi32(uint32_t a, uint32_t b) {
  return (uint32_t)(((uint64_t)a * b) >> 32);
}

// 2^(frac 2^-64) 2^63; tab[j] = round(2^63 2^(j/256)).  Short by at most
// 4.0e-18 relative: the three truncated Horner steps 2^-60 each, the series'
// end 2^-60.7, the rounding of c3 and c4 2^-61 each.
__host__ __device__ __forceinline__ uint64_t exp2_significand(uint64_t frac, const uint64_t* tab) {
  const uint64_t T = tab[(uint32_t)(frac >> 56)];
  const uint64_t F = frac << 8;                                  // f 2^72
  const uint32_t F1 = (uint32_t)(F >> 32);                       // f 2^40
  uint32_t q = 0x5762u;                                          // c5 2^24
  q = 0x00276557u + (mulhi32(F1, q) >> 4);                       // c4 2^28
  q = 0xe35846b8u + mulhi32(F1, q);                              // c3 2^36
  const uint32_t h = mulhi32(F1, q);                             // (c3 f + ..) 2^44
  const uint64_t s = 0x0f5fdeffc162c754ull + ((uint64_t)h << 18);  // c2 2^62
  const uint64_t P = 0xb17217f7d1cf79acull + (mulhi_approx(F, s) >> 6);  // c1 2^64
  const uint64_t v = mulhi_approx(F, P);                         // (2^f - 1) 2^72
  return T + (mulhi_approx(T, v) >> 8);                          // 2^63 2^(j/256 + f)
}

// bits of the double M 2^(n - 63), 2^63 <= M, -1022 <= n <= 1023, rounded to
// nearest (at n = 1023 up to infinity)
__host__ __device__ __forceinline__ uint64_t pack_double(int n, uint64_t M) {
  return (((M >> 10) + 1u) >> 1) + ((uint64_t)(int64_t)(n + 1022) << 52);
}

// the same for any n: subnormals, zero and infinity
__host__ __device__ __forceinline__ uint64_t pack_double_any(int n, uint64_t M) {
  if ((uint32_t)(n + 1022) < 2046u) return pack_double(n, M);
  if (n > 0) return 0x7ff0000000000000ull;
  const int sh = -1022 - n;
  return sh > 54 ? 0 : (((M >> 10) >> sh) + 1u) >> 1;
}

// bits of exp(x) for the double with bits b, |x| < 704: |x| and |x| log2(e)
// in 86 fractional bits (exact for |x| >= 2^-34), the sign applied to the
// fixed-point value.
__host__ __device__ __forceinline__ uint64_t exp_fixed_bits(uint64_t b, const uint64_t* tab) {
  const uint32_t hi = (uint32_t)(b >> 32);
  const int sh = 1032 - (int)((hi >> 20) & 0x7ffu);              // >= 0
  const int shc = sh > 63 ? 63 : sh;                             // |x| < 2^-54 (zero, subnormal): as 0
  const uint64_t m = (b << 11) | 0x8000000000000000ull;          // significand 2^63
  const uint64_t X = sh > 63 ? 0 : m >> shc;                     // |x| 2^54 ...
  const uint32_t r = sh > 63 ? 0u : (uint32_t)(((m << 1) << (63 - shc)) >> 32);  // ... and the 32 bits below
  // |x| (log2(e) - 1) from the constant's first 96 bits
  const uint32_t x0 = (uint32_t)X, x1 = (uint32_t)(X >> 32);
  const uint64_t u = (uint64_t)x0 * 0x71547652u;
  const uint64_t v = (uint64_t)x1 * 0xb82fe177u + (uint32_t)u;
  const uint64_t w = (uint64_t)r + (uint32_t)v + mulhi32(x1, 0x7d0ffda0u) + mulhi32(x0, 0xb82fe177u) + mulhi32(r, 0x71547652u);
  uint64_t Y = X + ((uint64_t)x1 * 0x71547652u + (u >> 32) + (v >> 32) + (w >> 32));
  uint32_t y = (uint32_t)w;
  int n = 0;
  if ((int32_t)hi < 0) {
    n = (Y | y) != 0 ? -1024 : 0;
    y = 0u - y;
    Y = ~Y + (y == 0u);
  }
  n += (int)(Y >> 54);
  return pack_double(n, exp2_significand((Y << 10) | (y >> 22), tab));
}

// One entry of the logarithm's table: r = ceil(2^15 / (1 + j/256)),
// t = round(2^62 log2(2^15 / r)).
struct LogEntry {
  uint64_t t;
  uint64_t r;
};

// log2 of the positive normal double with bits b as e + f 2^-62, e the
// exponent of b (returned in e), 0 <= f <= 2^62.  With m the significand and
// r from the table, z = m r 2^-15 - 1 lies in [0, 1.02 2^-8] and is exact in
// 64 bits (m r - 2^67 modulo 2^64); log2(m) = t + log2(1 + z) by the series
// z (k1 - z (k2 - ..)), k_i = 1 / (i ln 2), six terms.  Absolute error below
// 2^-54.
__host__ __device__ __forceinline__ uint64_t log2_fixed(uint64_t b, int& e, const LogEntry* __restrict__ tab) {
  const uint32_t hi = (uint32_t)(b >> 32);
  e = (int)(hi >> 20) - 1023;
  const LogEntry t = tab[(hi >> 12) & 255u];
  const uint64_t m = (b & 0x000fffffffffffffull) | 0x0010000000000000ull;
  const uint64_t F = (m * (uint32_t)t.r) << 4;                   // z 2^71
  const uint32_t F1 = (uint32_t)(F >> 32), z32 = F1 >> 7;        // z 2^39, z 2^32
  uint32_t q = 0x49ddb144u - mulhi32(z32, 0x3d8e13b8u);          // (k5 - z k6) 2^32
  q = 0x5c551d95u - mulhi32(z32, q);                             // k4
  q = 0x7b1c2771u - mulhi32(z32, q);                             // k3
  const uint64_t s = 0x5c551d94ae0bf85eull - (((uint64_t)F1 * q) >> 8);  // (k2 - ..) 2^63
  const uint64_t P = 0x5c551d94ae0bf85eull - (mulhi_approx(F, s) >> 8);  // (k1 - ..) 2^62
  return t.t + (mulhi_approx(F, P) >> 7);
}

// c b 2^-64 for a signed constant c and an unsigned b, short by at most 2
__host__ __device__ __forceinline__ int64_t mulhi_su(int64_t c, uint64_t b) {
  return (int64_t)(mulhi_approx((uint64_t)c, b) - (c < 0 ? b : 0));
}

__host__ __device__ __forceinline__ int clz64(uint64_t x) {
#ifdef __CUDA_ARCH__
  return __clzll((long long)x);
#else
  return x ? __builtin_clzll(x) : 64;
#endif
}

// bits of the double x 2^-s (rounded to nearest, ties up), |x| 2^-s within
// the normal range or 0; integer instructions where the hardware conversion
// would take an FP64-pipe slot
__host__ __device__ __forceinline__ uint64_t fixed_to_double(int64_t x, int s) {
  const uint64_t a = x < 0 ? 0 - (uint64_t)x : (uint64_t)x;
  const int lz = clz64(a);
  const uint64_t m = a << (lz & 63);
  const uint64_t r = (((m >> 10) + 1u) >> 1) + ((uint64_t)(1085 - lz - s) << 52);
  return a == 0 ? 0 : r | ((uint64_t)x & 0x8000000000000000ull);
}

// log2 of an Arrhenius rate constant, 2^51: A, beta and theta as packed in a
// reaction's record (fA holds 3/4 of a unit per product, their mean truncation),
// L = log2(T) 2^59, IT = 2^70 / T.  128 <= T < 65536 keeps both unsigned and
// below 2^63.
__host__ __device__ __forceinline__ int64_t arrhenius_fixed(int64_t fA, int64_t fB, int64_t fT, uint64_t L,
                                                            uint64_t IT) {
  return fA + mulhi_su(fB, L) + mulhi_su(fT, IT);
}

}  // namespace pj
