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

#include "fs_internal.h"
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
  unsigned long long q = r >= 1 && r < 63 ? (m + (1ull << (r - 1))) >> r : 0ull;
  return x < 0 ? -(long long)q : (long long)q;
}
// About |x| 2^(1023 - f) in FP32 (0 when far below): x relative to the
// exponent field f of the largest of its fellows.
__device__ __forceinline__ float rel_abs(double x, int f) {
  const int q = exp_field(x) - f + 127;
  return q > 1 ? __int_as_float((q << 23) | ((__double2hiint(x) & 0xFFFFF) << 3)) : 0.f;
}
// Biased exponent eb = E + 1023 with 2-norm < 2^E, from the largest exponent
// field f and the sum s of the squares of rel_abs.
__device__ __forceinline__ int norm_exponent(int f, float s) {
  const float r = fmaxf(sqrtf(s) * 1.001f, 1.0f);
  return f + ((__float_as_int(r) >> 23) & 0xFF) - 126;  // r < 2^(eb - f)
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

// ------------------------------------------------- phases in fixed point
// Products of phases on the integer units: two of them cost less than the
// four FP64 multiply-adds of one on GB300 (two issue slots a clock and SM).
// a b up to 2^-60, both with 62 fraction bits and |a b| <= 1.
__device__ __forceinline__ long long mul60(long long a, long long b) {
  return (long long)((unsigned long long)__mul64hi(a, b) << 2);
}
__device__ __forceinline__ longlong2 phase_mul(longlong2 x, longlong2 y) {
  return make_longlong2(mul60(x.x, y.x) - mul60(x.y, y.y), mul60(x.x, y.y) + mul60(x.y, y.x));
}
// (x.x + i x.y) times a phase, rounded at the last bit.
__device__ __forceinline__ longlong2 cmul_fx(longlong2 x, longlong2 y) {
  return make_longlong2(mul(x.x, y.x) - mul(x.y, y.y), mul(x.x, y.y) + mul(x.y, y.x));
}
__device__ __forceinline__ bool not_finite(double2 z) {
  return exp_field(z.x) == 0x7FF || exp_field(z.y) == 0x7FF;
}
__device__ __forceinline__ double2 nan2() {
  return make_double2(__longlong_as_double(0x7FF8000000000000ll),
                      __longlong_as_double(0x7FF8000000000000ll));
}
__device__ __forceinline__ longlong2 phase_from(double2 z) {  // |z| <= 1 + rounding
  return make_longlong2(from_double(z.x, 1024) << 1, from_double(z.y, 1024) << 1);
}
__device__ __forceinline__ double2 phase_to(longlong2 z) {
  return make_double2(to_double(z.x, 1023), to_double(z.y, 1023));
}
// Cross-phase tables of the vectors v0 .. v0 + nv - 1 of the other spin (the
// complex128 form of build_cross_tables): tab[kv][c][v] = exp(i sum over the
// bits b of v of w(8 c + b)), w(x) = sum_{y in I} X[y][x] (this = beta) or
// X[x][y].  One sincos per vector and orbital, then products: pairs of half
// bytes, which are products of single orbitals.  work: nv (32 + 32 nchunk)
// entries; bad: per vector, the orbitals whose angle is not finite (a string
// that holds one has no phase).  Ends with a barrier (`sync`).
template <typename Sync>
__device__ void cross_tables(const uint32_t* masks_other, int dir, int norb, int nchunk,
                             const Mat& X, int v0, int nv, longlong2* tab, longlong2* work,
                             uint32_t* bad, int tid, int nthr, Sync&& sync) {
  longlong2* one = work;                  // [nv][32] exp(i w(x))
  longlong2* half = work + nv * 32;       // [nv][nchunk][2][16]
  for (int i = tid; i < nv; i += nthr) bad[i] = 0;
  sync();
  for (int i = tid; i < nv * 32; i += nthr) {
    const int kv = i >> 5, x = i & 31;
    double s = 0, c = 1, sn = 0;
    if (x < norb) {
      for (uint32_t m = masks_other[v0 + kv]; m; m &= m - 1) {
        const int y = __ffs(m) - 1;
        s += dir == 1 ? X.v[y * norb + x] : X.v[x * norb + y];
      }
      if (exp_field(s) == 0x7FF) atomicOr(bad + kv, 1u << x);
      sincos(s - 6.283185307179586 * rint(s * 0.15915494309189535), &sn, &c);
    }
    one[i] = phase_from(make_double2(c, sn));
  }
  sync();
  for (int i = tid; i < nv * nchunk * 32; i += nthr) {
    const int kv = i / (nchunk * 32), r = i - kv * nchunk * 32;  // r = (c, h, v)
    const longlong2* e = one + kv * 32 + (r >> 4) * 4;
    longlong2 z = make_longlong2(1ll << 62, 0);
    for (int b = 0; b < 4; ++b)
      if ((r >> b) & 1) z = phase_mul(z, e[b]);
    half[i] = z;
  }
  sync();
  for (int i = tid; i < nv * nchunk * 256; i += nthr) {
    const int v = i & 255;
    const longlong2* h = half + (i >> 8) * 32;
    tab[i] = phase_mul(h[16 + (v >> 4)], h[v & 15]);
  }
  sync();
}

}  // namespace fx
}  // namespace fs
