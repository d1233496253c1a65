// Exact fixed-point operands for complex128 work on the tensor cores.
//
// GB300 issues two FP64 multiply-adds per clock and SM but 8192 FP16 ones on
// the tensor cores, so the complex128 contractions run there on integers:
//   * a value x with |x| <= 2^E is held as the 64-bit integer
//     X = x 2^(62 - E) (its last bit is 2^-62 of the scale; FP64 keeps 2^-53
//     of each value), the scale being shared by one vector (sweeps) or one
//     matrix row (GEMM);
//   * X = sum_i d_i 512^(7 - i), i = 1 .. 7, with balanced digits
//     -256 <= d_i <= 255 (-257 .. 257 for the first), each of them exactly
//     an FP16 number;
//   * the product of two such numbers is sum_s 512^(14 - s) sum_{i+j=s}
//     d_i e_j.  Each sum over i + j = s, over K terms as well, is an integer
//     that the FP32 accumulator of tcgen05.mma holds exactly below 2^24
//     (|d e| <= 2^16, so up to 256 terms).  The 28 products with i + j <= 8
//     are kept: those with i + j = 9 are some 2^-61 of the scale product, and
//     for i + j = 8, where a sum may pass 2^24 and round, one unit is
//     2^-70 of it;
//   * the seven sums are put together in 64-bit integer arithmetic.
#pragma once
#include <cuda_fp16.h>
#include <stdint.h>

#include "fs_tc.cuh"

namespace fs {
namespace fx {

constexpr int kDig = 7;   // digits of a value
constexpr int kSum = 7;   // accumulators: i + j = 2 .. 8
constexpr int kFrac = 62; // fraction bits of the fixed-point values
// 2^63 + sum_k 256 * 512^k, k = 0 .. 5: added before the digits are cut out,
// so that each 9-bit field is its balanced digit plus 256 and the top ten
// bits are the first digit plus 512.
constexpr unsigned long long kBias = (1ull << 63) + 0x20100804020100ull;

// The 9-bit fields (digit + 256) of two biased values, least significant
// first, as the two halves of an FP16 pair: 1024 + field is the FP16 number
// with the field in its low mantissa bits, and subtracting 1280 leaves the
// digit exactly.
__device__ __forceinline__ uint32_t pair_digit(uint32_t a, uint32_t b) {
  const uint32_t t = (__byte_perm(a, b, 0x5410) & 0x01FF01FFu) | 0x64006400u;
  const __half2 h = __hsub2(*reinterpret_cast<const __half2*>(&t),
                            __half2{__ushort_as_half(0x6500), __ushort_as_half(0x6500)});
  return *reinterpret_cast<const uint32_t*>(&h);
}
// w[i - 1] = digit i of (x, y), x in the low half.
__device__ __forceinline__ void digits2(long long x, long long y, uint32_t (&w)[kDig]) {
  const unsigned long long u = (unsigned long long)x + kBias, v = (unsigned long long)y + kBias;
  const uint32_t ul = (uint32_t)u, uh = (uint32_t)(u >> 32);
  const uint32_t vl = (uint32_t)v, vh = (uint32_t)(v >> 32);
  {  // ten bits: 1024 + (digit + 512) - 1536
    const uint32_t t = __byte_perm(uh >> 22, vh >> 22, 0x5410) | 0x64006400u;
    const __half2 h = __hsub2(*reinterpret_cast<const __half2*>(&t),
                              __half2{__ushort_as_half(0x6600), __ushort_as_half(0x6600)});
    w[0] = *reinterpret_cast<const uint32_t*>(&h);
  }
  w[1] = pair_digit(uh >> 13, vh >> 13);
  w[2] = pair_digit(uh >> 4, vh >> 4);
  w[3] = pair_digit(__funnelshift_r(ul, uh, 27), __funnelshift_r(vl, vh, 27));
  w[4] = pair_digit(ul >> 18, vl >> 18);
  w[5] = pair_digit(ul >> 9, vl >> 9);
  w[6] = pair_digit(ul, vl);
}
// sum_s D_s 512^(14 - s) 2^-62: the fixed-point result of seven accumulators
// (f[0] = D_2 .. f[6] = D_8), both operands with 62 fraction bits, the result
// below 2^63.  The floats become integers by adding a power of two and
// reading the bits (conversion instructions run at an eighth of the rate of
// additions here): D_2 .. D_4 directly, since with operand rows of 2-norm at
// most 1 and K <= 40 they stay below 2^22 (the first digit of a row has 2-norm
// at most 257 + sqrt(K) / 2, so sum_k d_1k e_jk <= 4.2e5, any other pair is
// below 2.7e6); the others are parted at a multiple of 512, whose quotient
// joins the next sum.
__device__ __forceinline__ long long join(const float (&f)[kSum]) {
  constexpr float kOne = 12582912.f;        // 1.5 2^23: unit 1
  constexpr float k512 = 6442450944.f;      // 1.5 2^32: unit 512
  constexpr uint32_t kOneB = 0x4B400000u, k512B = 0x4FC00000u;  // their bits
  const float f7 = fmaf(f[6], 1.f / 512.f, f[5]);
  const float t7 = f7 + k512, t6 = f[4] + k512, t5 = f[3] + k512;
  const float l7 = f7 - (t7 - k512), l6 = f[4] - (t6 - k512), l5 = f[3] - (t5 - k512);
  const int i7 = (int)(__float_as_uint(fmaf(l7, 2.f, kOne)) - kOneB);
  const int i6 = (int)(__float_as_uint(l6 + kOne) + __float_as_uint(t7) - (kOneB + k512B));
  const int i5 = (int)(__float_as_uint(l5 + kOne) + __float_as_uint(t6) - (kOneB + k512B));
  const int i4 = (int)(__float_as_uint(f[2] + kOne) + __float_as_uint(t5) - (kOneB + k512B));
  const int i3 = (int)(__float_as_uint(f[1] + kOne) - kOneB);
  const int i2 = (int)(__float_as_uint(f[0] + kOne) - kOneB);
  long long a = i6 * 1024 + i7;
  a += (long long)i5 * (1 << 19);
  a += (long long)i4 * (1 << 28);
  a += (long long)((unsigned long long)(long long)(i2 * 512 + i3) << 37);
  return a;
}
// (a * b) 2^-62, both with 62 fraction bits, rounded to nearest.
__device__ __forceinline__ long long mul(long long a, long long b) {
  const long long hi = __mul64hi(a, b);
  const unsigned long long lo = (unsigned long long)a * (unsigned long long)b;
  return (long long)(((unsigned long long)hi << 2) | (lo >> 62)) + (long long)((lo >> 61) & 1ull);
}

// Biased exponent of a double (0 for zero and subnormals).
__device__ __forceinline__ int exp_field(double x) {
  return (__double2hiint(x) >> 20) & 0x7FF;
}
// x 2^(62 - E), rounded to nearest, for |x| < 2^E (eb = E + 1023).
__device__ __forceinline__ long long from_double(double x, int eb) {
  const int f = exp_field(x);
  unsigned long long m = (unsigned long long)__double_as_longlong(x) & 0x000FFFFFFFFFFFFFull;
  if (f != 0) m |= 0x0010000000000000ull;
  m <<= 10;                        // |x| 2^(62 - e), e = max(f, 1) - 1023
  const int r = eb - (f ? f : 1);     // >= 1
  unsigned long long q = r < 63 ? (m + (1ull << (r - 1))) >> r : 0ull;
  return x < 0 ? -(long long)q : (long long)q;
}
// X 2^(E - 62), eb = E + 1023, rounded to 53 bits.  Built from integers (the
// 64-bit conversion instruction runs on the FP64 units).
__device__ __forceinline__ double to_double(long long X, int eb) {
  const unsigned long long mag = (unsigned long long)(X < 0 ? -X : X);
  const int lz = __clzll((long long)mag);
  const int field = eb + 1 - lz;  // exponent field of the result
  if (field >= 1 && field < 2046 && mag) {
    const unsigned long long m = mag << lz;
    const unsigned long long q = (m >> 11) + ((m >> 10) & 1ull);
    const unsigned long long v = ((unsigned long long)(field - 1) << 52) + q;
    return __longlong_as_double((long long)(v | ((unsigned long long)X & (1ull << 63))));
  }
  return scalbn(__ll2double_rn(X), eb - 1023 - kFrac);  // zeros, out of range
}

}  // namespace fx
}  // namespace fs
