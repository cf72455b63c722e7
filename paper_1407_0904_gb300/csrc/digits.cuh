// Exact integer products of FP64 numbers on the f16 tensor cores: fixed-point digits, the issue of their
// MMAs, and the rounding of 64-bit integers to double. Shared by the FP64 assembly (k_fp64_tc.cu, which
// describes the method) and its adjoint (k_bwd_tc.cu).
#pragma once
#include <cuda_runtime.h>
#include <cuda_fp16.h>
#include <cstdint>
#include <cstdlib>
#include "coffee_internal.h"
#include "tc_common.cuh"

namespace coffee {
namespace tc {

// Shared-memory descriptor of a K-major operand without swizzle whose rows of 16 bytes (8 halves) are contiguous
// and whose second 16 bytes of a K step of 16 lie lbo bytes further.
__device__ __forceinline__ uint64_t f_desc(uint32_t saddr, uint32_t lbo) {
  return (uint64_t)((saddr >> 4) & 0x3FFFu) | (uint64_t)((lbo >> 4) & 0x3FFFu) << 16 | (uint64_t)(128u >> 4) << 32 |
         1ull << 46;
}

// Fixed point of x scaled by 2^(FB - X), FB = 61 (b = 9) or 62 (b = 8): X = biased exponent bound of the
// cell's factors (x < 2^(X-1022)), sh = X - (x's biased exponent) >= 0, plus the digits' bias.
template <uint64_t BIAS, int FB>
__device__ __forceinline__ uint64_t fixed_point(double x, int e20, int t20) {
  const uint32_t h = (uint32_t)__double2hiint(x), l = (uint32_t)__double2loint(x);
  const uint32_t ef = h & 0x7FF00000u;
  const uint32_t sh = min(((uint32_t)(e20 - t20) - ef) >> 20, 63u);
  uint64_t m = ((uint64_t)((h & 0xFFFFFu) | 0x100000u) << 32) | l;
  m = ef == 0u ? 0ull : (m << (FB - 53)) >> sh;  // subnormals count as zero (the largest factor is above 2^-900)
  return ((int)h < 0 ? 0ull - m : m) + BIAS;
}

// Eight numbers' digits p = 0 (leading) .. ND-1: 16 bytes each, PSTRIDE bytes apart.
template <int B, int ND, int PSTRIDE, bool CONSTANT>
__device__ __forceinline__ void store_digits(uint8_t* dst, const uint64_t (&U)[8]) {
  constexpr uint32_t mask = (1u << B) - 1u;
  // 0x6400 + u is the half 1024 + u, so one packed subtraction leaves the balanced digits
  const __half2 off = __halves2half2(__ushort_as_half(0x6400 + (1 << (B - 1))), __ushort_as_half(0x6400 + (1 << (B - 1))));
#pragma unroll
  for (int p = 0; p < ND; ++p) {
    const int sh = B * (ND - 1 - p);
    uint32_t w[4];
#pragma unroll
    for (int j = 0; j < 4; ++j) {
      const uint32_t a = (uint32_t)(U[2 * j] >> sh), b = (uint32_t)(U[2 * j + 1] >> sh);
      // the leading digit takes every bit left (b = 9: up to 2^9 at |g| = 2^62)
      const uint32_t u = (p ? a & mask : a) | ((p ? b & mask : b) << 16) | 0x64006400u;
      __half2 v = __hsub2(*reinterpret_cast<const __half2*>(&u), off);
      w[j] = *reinterpret_cast<uint32_t*>(&v);
    }
    // the constant's factor, 4096, in the last slot of the leading digit block
    if constexpr (CONSTANT) w[3] = (w[3] & 0xFFFFu) | (p == 0 ? 0x6C000000u : 0u);
    *reinterpret_cast<uint4*>(dst + p * PSTRIDE) = make_uint4(w[0], w[1], w[2], w[3]);
  }
}

// Integer multiply-adds. The compiler would turn multiplications by known powers of two into shifts, which
// share the ALU pipe (half a warp instruction per cycle) with everything else here; multiplications have
// a pipe of their own, so the powers are kept in registers whose values it does not see.
__device__ __forceinline__ uint32_t opaque(uint32_t x) {
  uint32_t r;
  asm("mov.u32 %0, %1;" : "=r"(r) : "r"(x));
  return r;
}
__device__ __forceinline__ uint32_t mad_lo(uint32_t a, uint32_t b, uint32_t c) {
  uint32_t r;
  asm("mad.lo.u32 %0, %1, %2, %3;" : "=r"(r) : "r"(a), "r"(b), "r"(c));
  return r;
}
__device__ __forceinline__ uint32_t mad_hi(uint32_t a, uint32_t b, uint32_t c) {
  uint32_t r;
  asm("mad.hi.u32 %0, %1, %2, %3;" : "=r"(r) : "r"(a), "r"(b), "r"(c));
  return r;
}
__device__ __forceinline__ uint64_t mad_wide(uint32_t a, uint32_t b, uint64_t c) {
  uint64_t r;
  asm("mad.wide.u32 %0, %1, %2, %3;" : "=l"(r) : "r"(a), "r"(b), "l"(c));
  return r;
}

// The double S 2^E, rounded to nearest (ties away), by integer instructions: S = hi:lo a two's complement
// number below 2^62 with a high word other than 0 or -1 (bit < 0 otherwise, the result void),
// e20 = (E + 1054) << 20; p22 = 2^22, p20 = 2^20. |S| is shifted to 2^62 <= m < 2^63, half a unit of the
// last place (2^9) added on the way, and m >> 10 is the significand with its leading one, which counts as
// one in the exponent field.
__device__ __forceinline__ double from_fixed(uint32_t hi, uint32_t lo, uint32_t e20, uint32_t p22, uint32_t p20,
                                             int& bit) {
  const uint32_t s = (uint32_t)((int)hi >> 31);
  asm("bfind.s32 %0, %1;" : "=r"(bit) : "r"(hi));  // the leading bit of |S| is 32 + bit
  uint32_t P;
  asm("shr.u32 %0, %1, %2;" : "=r"(P) : "r"(0x40000000u), "r"(bit));  // (0 for a bit of -1)
  const uint64_t m = mad_wide(lo ^ s, P, 0x200ull);
  const uint32_t mh = mad_lo(hi ^ s, P, (uint32_t)(m >> 32));
  const uint32_t qh = mad_hi(mh, p22, mad_lo((uint32_t)bit, p20, e20));
  return __hiloint2double((int)(qh | (s & 0x80000000u)), (int)__funnelshift_r((uint32_t)m, mh, 10));
}
// The same for any S below 2^62.
__device__ __forceinline__ double from_fixed_any(uint32_t hi, uint32_t lo, uint32_t e20) {
  int bit;
  const uint32_t s = (uint32_t)((int)hi >> 31);
  if ((hi ^ s) != 0u) return from_fixed(hi, lo, e20, 1u << 22, 1u << 20, bit);
  const uint32_t l = lo ^ s;  // |S|, or |S| - 1
  if (l < 4u) return 0.0;      // rounding of the digits
  // 32 places up: |S| < 2^32 becomes 2^30 times itself, so that the high word stays below 2^30
  return from_fixed(((l >> 2) ^ s), ((l << 30) ^ s), e20 - (30u << 20), 1u << 22, 1u << 20, bit);
}

inline uint16_t half_of_int(int v) {  // |v| <= 4096, exact in a half
  if (v == 0) return 0;
  const uint16_t s = v < 0 ? 0x8000 : 0;
  unsigned a = (unsigned)std::abs(v);
  int e = 0;
  while ((a >> e) > 1) ++e;
  return (uint16_t)(s | ((e + 15) << 10) | ((e <= 10 ? a << (10 - e) : a >> (e - 10)) & 0x3FFu));
}

}  // namespace tc
}  // namespace coffee
