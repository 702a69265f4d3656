// FP64 operands as 8-bit digits for the BF16 tensor cores (csrc/iedg_assemble.cu, the
// partial LU; csrc/iedg_assemble_dg.cu, the volume terms of the assembly).
//
// With emax the biased exponent of (a bound on) a row's or column's largest entry, an
// entry x becomes the integer X next to x 2^(61 - (emax - 1023)), |X| < 2^62, in balanced
// base 256: X = sum_s d_s 256^(7 - s), s = 0..7, -128 <= d_s <= 127 and |d_0| <= 64.  Digits
// are exact in BF16 and their products' sums exact in FP32 below 2^24.  X is in error by up to
// 2^-62 (rounded; 2^-61 cut off) of the largest entry, or of a bound on it: entries far below
// it keep fewer bits than FP64 holds.
#pragma once
#include <cstdint>
#include <cuda_runtime.h>

namespace iedg {
namespace dig {

constexpr int S = 8;                     // digits per operand, and product levels kept
constexpr int BAD_EXP = 1 << 13;         // exponent of a row or column with a non-finite entry

__host__ __device__ __forceinline__ int exponent_bits(long long b) { return (int)((b >> 52) & 0x7ff); }

// The digits of x, each with 128 added, most significant in the top byte.  Entries below
// 2^-62 of the scale and subnormals become 0.  NEAREST: rounded, not cut off (towards zero).
template <bool NEAREST = true>
__host__ __device__ __forceinline__ unsigned long long to_bytes(long long b, int emax) {
  const int e = exponent_bits(b), sh = emax - e;
  unsigned long long m = ((unsigned long long)b & 0xFFFFFFFFFFFFFull) | 0x10000000000000ull;
  m = (e == 0 || sh > 62 || sh < 0) ? 0ull : (NEAREST ? (((m << 10) >> sh) + 1) >> 1 : (m << 9) >> sh);
  return (b < 0 ? 0ull - m : m) + 0x8080808080808080ull;
}

#ifdef __CUDACC__
__device__ __forceinline__ int exponent_of(double x) { return (__double2hiint(x) >> 20) & 0x7ff; }
// biased exponent of a row's (column's) scale as the epilogue adds it
__device__ __forceinline__ int scale_of(int emax) { return emax >= 0x7ff ? BAD_EXP : emax; }

// Two values' digits s as packed BF16; w: the word of to_bytes that holds digit s (the upper
// one for s < 4).  byte -> float 2^23 + byte, minus 2^23 + 128: at most 8 significant
// bits, so the upper half of the FP32 pattern is the BF16 value; `scale`: a power of two.
__device__ __forceinline__ uint32_t bf16_pair(uint32_t w0, uint32_t w1, int s, float scale = 1.0f) {
  const uint32_t sel = 0x7440u | (uint32_t)(3 - (s & 3));
  const float f0 = (__uint_as_float(__byte_perm(w0, 0x4B000000u, sel)) - 8388736.0f) * scale;
  const float f1 = (__uint_as_float(__byte_perm(w1, 0x4B000000u, sel)) - 8388736.0f) * scale;
  return __byte_perm(__float_as_uint(f0), __float_as_uint(f1), 0x7632);
}

// +-mag 2^(field - 1086 + lz) normalised and rounded to FP64 from a 64-bit magnitude whose
// leading zeros are lz; field: biased exponent of the result; `odd` is set outside the
// normal range, where the caller replaces the result by special().
__device__ __forceinline__ double from_fixed(unsigned long long mag, int lz, int field, unsigned long long sign,
                                             bool& odd) {
  const unsigned long long mn = mag << lz;
  const unsigned long long r =
      ((mn >> 11) + ((mn >> 10) & 1ull) + ((unsigned long long)(unsigned)(field - 1) << 52)) | sign;
  odd = mag != 0 && (unsigned)(field - 1) >= 2045u;
  return __longlong_as_double(mag != 0 ? (long long)r : 0ll);
}
// the replacement, ef = row + column exponent: NaN of a non-finite operand, 0 below the
// normal range, an infinity above it
__device__ __forceinline__ double special(double r, int ef) {
  if (ef >= BAD_EXP) return __longlong_as_double(0x7FF8000000000000ll);
  return ef < 2046 ? 0.0 : copysign(__longlong_as_double(0x7FF0000000000000ll), r);
}

// Eight (four) 32-bit columns of each of eight levels (`stride` columns apart) of this
// thread's lane.
__device__ __forceinline__ void load_levels(uint32_t taddr, uint32_t stride, float (&v)[8][8]) {
  uint32_t r[8][8];
#pragma unroll
  for (int l = 0; l < 8; ++l)
    asm volatile("tcgen05.ld.sync.aligned.32x32b.x8.b32 {%0,%1,%2,%3,%4,%5,%6,%7}, [%8];"
                 : "=r"(r[l][0]), "=r"(r[l][1]), "=r"(r[l][2]), "=r"(r[l][3]), "=r"(r[l][4]), "=r"(r[l][5]),
                   "=r"(r[l][6]), "=r"(r[l][7])
                 : "r"(taddr + (uint32_t)l * stride));
  asm volatile("tcgen05.wait::ld.sync.aligned;" ::: "memory");
#pragma unroll
  for (int l = 0; l < 8; ++l)
#pragma unroll
    for (int j = 0; j < 8; ++j) v[l][j] = __uint_as_float(r[l][j]);
}
__device__ __forceinline__ void load_levels(uint32_t taddr, uint32_t stride, float (&v)[8][4]) {
  uint32_t r[8][4];
#pragma unroll
  for (int l = 0; l < 8; ++l)
    asm volatile("tcgen05.ld.sync.aligned.32x32b.x4.b32 {%0,%1,%2,%3}, [%4];"
                 : "=r"(r[l][0]), "=r"(r[l][1]), "=r"(r[l][2]), "=r"(r[l][3])
                 : "r"(taddr + (uint32_t)l * stride));
  asm volatile("tcgen05.wait::ld.sync.aligned;" ::: "memory");
#pragma unroll
  for (int l = 0; l < 8; ++l)
#pragma unroll
    for (int j = 0; j < 4; ++j) v[l][j] = __uint_as_float(r[l][j]);
}
#endif

}  // namespace dig
}  // namespace iedg
