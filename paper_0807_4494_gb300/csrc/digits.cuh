// Fixed-point digits of FP64 numbers as FP16 tensor-core operands, shared by the torus products (torus_digits.cu)
// and the contractions (contract_digits.cu) of FP64 plans.
#pragma once

#include <cstdint>

#include "tc_common.cuh"

namespace ssht {
namespace {

using namespace tc;

constexpr int kDigits = 8;            // of a data row and of the torus products' matrices
constexpr int kNotFinite = 1 << 20;   // exponent of a row that holds an infinity or a NaN

// Exponent field of x (1 for denormals and zero), or kNotFinite.
__device__ __forceinline__ int exponent_of(double x) {
  const int e = (__double2hiint(x) >> 20) & 0x7ff;
  return e == 0x7ff ? kNotFinite : max(e, 1);
}

// x in units of 2^(e - 1075 - UP), rounded to nearest, e >= its own exponent field: at most 53 + UP bits.
template <int UP>
__device__ __forceinline__ long long fixed_point(double x, int e) {
  const unsigned long long u = (unsigned long long)__double_as_longlong(x);
  const int ex = (int)(u >> 52) & 0x7ff;
  unsigned long long m = (u & 0xfffffffffffffull) | (ex ? 1ull << 52 : 0ull);
  const int sh = e - max(ex, 1);
  m = sh > 53 + UP ? 0ull : sh > 0 ? ((m << UP) + (1ull << (sh - 1))) >> sh : m << UP;
  return (u >> 63) ? -(long long)m : (long long)m;
}

// DIGITS digits (8: of 55-bit numbers in units of 2^(e - 1077); 9: of 62-bit ones, 2^(e - 1084)) of eight
// consecutive k's of a row go to 16 bytes a digit: with 64 sum_i 128^i added, a digit is the plain field of seven
// bits less 64 (the top one takes 0 .. 128), and 0x6400 + n is the FP16 number 1024 + n.  Two digits share a part's
// 128-byte row.
template <int DIGITS, int PART_BYTES>
__device__ __forceinline__ void put_integers(uint8_t* tile, int row, int piece, unsigned long long (&v)[8]) {
  constexpr unsigned long long kMiddle = DIGITS == 8 ? 0x81020408102040ull : 0x4081020408102040ull;
#pragma unroll
  for (int k = 0; k < 8; ++k) v[k] += kMiddle;
  const __half2 bias = __float2half2_rn(1088.f);
#pragma unroll
  for (int i = 0; i < DIGITS; ++i) {
    const int sh = 7 * (DIGITS - 1 - i);
    uint32_t w[4];
#pragma unroll
    for (int k = 0; k < 4; ++k) {
      uint32_t a = (uint32_t)(v[2 * k] >> sh), b = (uint32_t)(v[2 * k + 1] >> sh);
      if (i > 0) {
        a &= 127u;
        b &= 127u;
      }
      const uint32_t bits = 0x64006400u + a + (b << 16);
      const __half2 h = __hsub2(*reinterpret_cast<const __half2*>(&bits), bias);
      w[k] = *reinterpret_cast<const uint32_t*>(&h);
    }
    *(uint4*)(tile + (i >> 1) * PART_BYTES + sw128(row, 64 * (i & 1) + 16 * piece)) = make_uint4(w[0], w[1], w[2], w[3]);
  }
}

template <int DIGITS, int PART_BYTES>
__device__ __forceinline__ void put_digits(uint8_t* tile, int row, int piece, const double (&x)[8], int e) {
  unsigned long long v[8];
#pragma unroll
  for (int k = 0; k < 8; ++k) v[k] = (unsigned long long)fixed_point<7 * DIGITS - 54>(x[k], e);
  put_integers<DIGITS, PART_BYTES>(tile, row, piece, v);
}

// (hi 2^28 + lo) 2^e, rounded to nearest.  Integer instructions: a conversion or product on the FP64 pipe takes a warp 64 clocks.
__device__ __forceinline__ double assemble(long long hi, long long lo, int e) {
  long long h = hi + (lo >> 28);
  unsigned l = (unsigned)lo & 0xfffffffu;
  const bool neg = h < 0;
  if (neg) {
    h = -h - (l ? 1 : 0);
    l = (0u - l) & 0xfffffffu;
  }
  const int z = min(__clzll(h), 28);
  unsigned long long m = ((unsigned long long)h << z) | (l >> (28 - z));
  const int c = __clzll((long long)m);
  if (m) m <<= c;
  m = (m >> 11) + ((m >> 10) & 1);
  const int E = e + (28 - z) - c + 63 + 1023;
  if (m == 0 && E < kNotFinite / 2) return 0.0;
  if (E >= 1 && E <= 2045) return __longlong_as_double((long long)(((unsigned long long)(E - 1) << 52) + m) | (neg ? (1ll << 63) : 0ll));
  if (E >= kNotFinite / 2) return __longlong_as_double(0x7ff8000000000000ll);
  return (neg ? -1.0 : 1.0) * scalbn((double)m, E - 1023 - 52);
}

// Whether the CTA still works, the same answer for the whole (converged) warp.
__device__ __forceinline__ bool going(volatile int* abort) { return !__any_sync(0xffffffffu, *abort); }

}  // namespace
}  // namespace ssht
