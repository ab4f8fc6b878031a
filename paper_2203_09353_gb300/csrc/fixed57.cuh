// 57-bit fixed-point arithmetic on the integer pipe, for steps that FP64
// arithmetic bounds. GB300 issues 2 DFMA per clock per SM but 30 multiply-adds
// of 32 x 32 + 64 bits (both measured), so a product of two fixed-point values
// of up to 57 bits, three of them, runs at five times the DFMA rate.
//
// A value x, |x| <= 2^57 units of some power of two, is held as two signed
// limbs, x = h 2^27 + l with -2^26 <= l < 2^26 (|h| <= 2^30). The product of
// two values is h h' 2^54 + (h l' + l h') 2^27 + l l'; the last term, below
// 2^-61 of the largest product, is dropped. Sums keep the first two parts in
// 64-bit accumulators of their own, so that a multiply-add needs no carry
// handling, and fx_val joins them in units of 2^54 products. Signed 64-bit
// sums wrap without harm as long as the final value is in range.
#pragma once

#include <cuda_runtime.h>
#include <stdint.h>

namespace bg {
namespace fx {

constexpr int kLow = 27;  // bits of the low limb

struct Limb {
  int h, l;
};

__device__ __forceinline__ Limb split(long long x) {
  const int l = ((int)x << (32 - kLow)) >> (32 - kLow);  // low bits, sign-extended
  return {(int)((x - l) >> kLow), l};
}
__device__ __forceinline__ long long join(int h, int l) { return ((long long)h << kLow) + l; }

__device__ __forceinline__ void mac(long long& acc, int a, int b) { acc += (long long)a * b; }

// hi + cross 2^-27, rounded to nearest: the sum of products in units of 2^54.
__device__ __forceinline__ long long val(long long hi, long long cross) {
  return hi + ((cross + (1ll << (kLow - 1))) >> kLow);
}

// x 2^-s, s >= 1, rounded to nearest, ties to even. Values here are often one
// to three bits above the unit they are rounded to, so that ties are common;
// rounding them up would add the same sign everywhere, which sums to a rank-one
// error that grows with the order of a matrix (measured: 16 times the whole
// reduction's error at n = 1024).
__device__ __forceinline__ long long rne(long long x, int s) {
  return (x + ((1ll << (s - 1)) - 1) + ((x >> s) & 1)) >> s;
}

// x 2^z, rounded to nearest for z < 0.
__device__ __forceinline__ long long shift(long long x, int z) {
  return z >= 0 ? x << min(z, 63) : rne(x, min(-z, 62));
}

// Complex values: int4 {re.h, re.l, im.h, im.l}; sums of complex products.
struct Sum {
  long long rh = 0, rx = 0, ih = 0, ix = 0;
  __device__ __forceinline__ long long re() const { return val(rh, rx); }
  __device__ __forceinline__ long long im() const { return val(ih, ix); }
};

__device__ __forceinline__ int4 pack(long long re, long long im) {
  const Limb a = split(re), b = split(im);
  return make_int4(a.h, a.l, b.h, b.l);
}

// s += a b
__device__ __forceinline__ void cmac(Sum& s, const int4& a, const int4& b) {
  const int nh = -b.z, nl = -b.w;
  mac(s.rh, a.x, b.x);
  mac(s.rx, a.x, b.y);
  mac(s.ih, a.x, b.z);
  mac(s.ix, a.x, b.w);
  mac(s.rx, a.y, b.x);
  mac(s.ix, a.y, b.z);
  mac(s.rh, a.z, nh);
  mac(s.rx, a.z, nl);
  mac(s.ih, a.z, b.x);
  mac(s.ix, a.z, b.y);
  mac(s.rx, a.w, nh);
  mac(s.ix, a.w, b.x);
}

// s += a conj(b)
__device__ __forceinline__ void cmac_conj(Sum& s, const int4& a, const int4& b) {
  cmac(s, a, make_int4(b.x, b.y, -b.z, -b.w));
}

// A double x times 2^sh as a 64-bit integer, rounded to nearest (ties away
// from zero); |x| 2^sh must be below 2^62. Zero and subnormal x give what
// their bits say; a non-finite x gives a meaningless finite value.
__device__ __forceinline__ long long from_double(double x, int sh) {
  const uint32_t xh = (uint32_t)__double2hiint(x), xl = (uint32_t)__double2loint(x);
  const int eb = (int)(xh >> 20) & 0x7FF;
  const unsigned long long M =
      (unsigned long long)((xh & 0xFFFFFu) | (eb != 0 ? 0x100000u : 0u)) << 32 | xl;
  const int s = sh + (eb > 1 ? eb : 1) - 1075;  // x = M 2^(s - sh)
  unsigned long long N;
  if (s >= 0) N = M << min(s, 62);
  else N = s >= -54 ? ((M >> (-s - 1)) + 1) >> 1 : 0ull;
  return (xh >> 31) ? -(long long)N : (long long)N;
}

__device__ __forceinline__ long long shfl_xor(long long v, int o) {
  return __shfl_xor_sync(0xFFFFFFFFu, v, o);
}
__device__ __forceinline__ long long warp_sum(long long v) {
#pragma unroll
  for (int o = 16; o > 0; o >>= 1) v += shfl_xor(v, o);
  return v;
}

}  // namespace fx
}  // namespace bg
