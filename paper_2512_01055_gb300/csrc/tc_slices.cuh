// A double as S BF16 numbers x_0 + x_1 + ..., x_p the BF16 nearest to what the
// ones before leave (Henry, Tang, Heinecke, ARITH 2019), in FP32 arithmetic and
// bit for bit as FP64 residuals give it.  Plain C++ on the host as well, where a
// test compares it with them.
//
// x = h + l + m exactly, h the nearest float, l the leading 24 bits of the rest
// and m its last 5 at most: three FP64 operations (two conversions and a
// difference; m comes from the bits), GB300's FP64 pipe being 1/64 of its FP32
// pipe, where taking every slice and residual in FP64 costs three each.
// A slice is the BF16 nearest to h + l + m: of the FP32 sum s = fl(h + l), or
// where s lies midway between two, of the side on which the rest er + m lies, er
// the sum's rounding error (TwoSum).  (Midways are multiples of ulp(s), and
// |er + m| < ulp(s): m is below the last bit of l, and the sum is exact where s is
// so small that this could matter.)  s less the slice, exact, and er are the next
// h and l.  After the second slice er reaches down from 2^-32 of x, so er + m fits
// 24 bits and takes m in.
//
// Below about 2^-97, bits of x under 2^-149 are lost: BF16 ends at 2^-133.
#pragma once
#include <cstdint>
#include <cstring>

#ifdef __CUDACC__
#include <cuda_bf16.h>
#define TC_HD __host__ __device__ __forceinline__
#else
#define TC_HD inline
#endif

namespace tc {

TC_HD uint32_t float_bits(float x) { uint32_t b; std::memcpy(&b, &x, 4); return b; }
TC_HD float bits_float(uint32_t b) { float x; std::memcpy(&x, &b, 4); return x; }
// The leading 24 of x's 53 bits, add = 0x10000000: rounded to nearest, 0: cut off.
TC_HD double leading24(double x, uint64_t add) {
  uint64_t b;
  std::memcpy(&b, &x, 8);
  b = (b + add) & ~(uint64_t)0x1FFFFFFF;
  std::memcpy(&x, &b, 8);
  return x;
}
TC_HD uint32_t bf16_bits(float x) {                       // round to nearest even
#ifdef __CUDA_ARCH__
  return __bfloat16_as_ushort(__float2bfloat16_rn(x));
#else
  const uint32_t b = float_bits(x);
  if ((b & 0x7FFFFFFF) > 0x7F800000) return 0x7FFF;
  return (b + 0x7FFF + ((b >> 16) & 1)) >> 16;
#endif
}

struct Slicer {
  float h, l, m;
};
TC_HD Slicer slicer(double x) {
  const double a = leading24(x, 0x10000000), r = x - a;
  uint64_t b;
  std::memcpy(&b, &r, 8);
  // the low 29 bits of r's significand: all but the first five are zero, of weight 2^(e - 28)
  const uint32_t hi = (uint32_t)(b >> 32), low = (uint32_t)b >> 24 & 31u;
  const int e = (int)(hi >> 20 & 0x7FF) - 1023 - 28 + 127;
  // e < 255 while x is within the float range
  const float unit = bits_float((e > 0 ? (uint32_t)e << 23 : 0u) | (hi & 0x80000000u));
  return Slicer{(float)a, (float)leading24(r, 0), (float)(int)low * unit};
}
// The bits of slice p; p = 0, 1, 2, ... in order.
TC_HD uint32_t next_slice(Slicer &x, int p) {
  const float s = x.h + x.l, t = s - x.h, er = (x.h - (s - t)) + (x.l - t), rest = er + x.m;
  const uint32_t bits = float_bits(s);
  uint32_t b = bf16_bits(s);
  if ((bits & 0xFFFF) == 0x8000 && rest != 0.f) b = (bits >> 16) + (((float_bits(rest) ^ bits) >> 31) ^ 1u);
  x.h = s - bits_float(b << 16);
  x.l = p == 0 ? er : rest;
  if (p > 0) x.m = 0.f;
  return b;
}

}  // namespace tc
