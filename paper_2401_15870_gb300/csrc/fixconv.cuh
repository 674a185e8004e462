// fixconv.cuh -- the epilogue's two conversions in integer arithmetic: a new
// contribution rounded to the nearest multiple of 2^-61, and a fixed-point sum
// as a double.
//
// The DF / DF-P epilogue turns every processed vertex's new rank times
// 2^61 / |out(v)| into the nearest integer (its next fixed-point
// contribution).  The epilogue is bound by GB300's narrow FP64 pipe, and this
// conversion is one of its FP64 instructions; doing it with integer
// instructions moves it to the integer pipes.  It follows the IEEE 754
// definition (IEEE 754-2019 Sec. 5.8 convertToIntegerTiesToEven, rounding
// direction roundTiesToEven of Sec. 4.3.1) for the non-negative values below
// 2^63 the sweep produces, so it gives the same integer as the hardware
// conversion; tests/test_fixconv.py checks it against the C library's llrint
// on every exponent and every kind of tie, and the GPU tests check that
// sweeps using it agree bit for bit with sweeps using the hardware
// conversion.
#pragma once
#include <cstdint>
#include <cstring>

#if defined(__CUDACC__)
#define FIXCONV_FN __host__ __device__ __forceinline__
#else
#define FIXCONV_FN inline
#endif

namespace fixconv {

FIXCONV_FN uint64_t bits_of(double x) {
#if defined(__CUDA_ARCH__)
  return (uint64_t)__double_as_longlong(x);
#else
  uint64_t b;
  std::memcpy(&b, &x, sizeof b);
  return b;
#endif
}

// y in [0, 2^63) (finite) to the nearest integer, ties to even
FIXCONV_FN int64_t f64_to_i64_rn(double y) {
  const uint64_t b = bits_of(y);
  const int ex = (int)(b >> 52);       // biased exponent (the sign bit is 0)
  if (ex < 1022) return 0;             // y < 0.5
  const uint64_t sig = (b & ((1ull << 52) - 1)) | (1ull << 52);
  const int sh = 1075 - ex;            // fraction bits of sig: 52 - (ex - 1023)
  if (sh <= 0) return (int64_t)(sig << -sh);   // already an integer
  const uint64_t q = sig >> sh;        // sh in [1, 53]
  const uint64_t rem = sig & ((1ull << sh) - 1);
  const uint64_t half = 1ull << (sh - 1);
  return (int64_t)(q + ((rem > half || (rem == half && (q & 1ull))) ? 1ull : 0ull));
}

// v to the nearest double, ties to even.  One or two of the FP64 pipe's
// instructions as hardware conversion: the Static / ND epilogue, which spent
// 67% of its time on that pipe, went from 93 to 76 us at 8.4M vertices with it,
// the DF-P epilogue from 424 to 407 at 33.5M.
FIXCONV_FN double i64_to_f64_rn(int64_t v) {
  const uint64_t sign = (uint64_t)v & (1ull << 63);
  const uint64_t u = v < 0 ? 0ull - (uint64_t)v : (uint64_t)v;
#if defined(__CUDA_ARCH__)
  const int lz = __clzll((long long)u);
#else
  const int lz = u ? __builtin_clzll(u) : 64;
#endif
  // the significand with its leading bit at 63: the 11 bits below the last one
  // kept decide the rounding
  const uint64_t m = u << (lz & 63);
  uint64_t q = m >> 11;
  const uint32_t rem = (uint32_t)m & 0x7ffu;
  q += (rem > 0x400u || (rem == 0x400u && (q & 1ull))) ? 1ull : 0ull;
  // exponent of the leading bit, 63 - lz; that bit itself adds one to the field
  const uint64_t b = u ? sign | (q + ((uint64_t)(1023 + 63 - lz - 1) << 52)) : 0ull;
#if defined(__CUDA_ARCH__)
  return __longlong_as_double((long long)b);
#else
  double d;
  std::memcpy(&d, &b, sizeof d);
  return d;
#endif
}

}  // namespace fixconv
