// 60-bit fixed-point arithmetic on the integer pipe, for steps that FP64
// arithmetic bounds. GB300 issues 2 DFMA per clock per SM but 30 multiply-adds
// of 32 x 32 + 64 bits (both measured), so a product of two fixed-point values
// of up to 60 bits, three of them, runs at five times the DFMA rate.
//
// A value x, of up to 1.4 x 2^60 units of some power of two in magnitude, is
// held as two signed limbs, x = h 2^30 + l with -2^29 <= l < 2^29. The product
// of two values is h h' 2^60 + (h l' + l h') 2^30 + l l'; the last term, below
// 2^-62 of the largest product, is dropped. Sums keep the first two parts in
// 64-bit accumulators of their own, so that a multiply-add needs no carry
// handling; the upper bits of the cross part move to the high part (flush)
// before it can overflow, at intervals that each sum's bounds allow. A high
// part may wrap as long as its final value is in range.
#pragma once

#include <cuda_runtime.h>
#include <stdint.h>

namespace bg {
namespace fx {

constexpr int kLow = 30;   // bits of the low limb
constexpr int kFull = 60;  // full scale: values up to 1.4 x 2^kFull

struct Limb {
  int h, l;
};

__device__ __forceinline__ Limb split(long long x) {
  const unsigned long long v = (unsigned long long)x + (1u << (kLow - 1));
  return {(int)(uint32_t)(v >> kLow),
          (int)((uint32_t)v & ((1u << kLow) - 1)) - (1 << (kLow - 1))};
}
__device__ __forceinline__ long long join(int h, int l) { return ((long long)h << kLow) + l; }

__device__ __forceinline__ void mac(long long& acc, int a, int b) { acc += (long long)a * b; }

// (hi + cross 2^-30) 2^UP, rounded to nearest: the sum of products in units of 2^(60 - UP).
template <int UP = 0>
__device__ __forceinline__ long long val(long long hi, long long cross) {
  return (long long)((unsigned long long)hi << UP) +
         ((cross + (1ll << (kLow - 1 - UP))) >> (kLow - UP));
}
__device__ __forceinline__ void flush(long long& hi, long long& cross) {
  hi += cross >> kLow;
  cross &= (1ll << kLow) - 1;
}

// x 2^-s, s >= 1, rounded to nearest, ties to even. Where a value is one to
// three bits above the unit it is rounded to, ties are common; rounding them
// up would add the same sign everywhere, which sums to a rank-one error that
// grows with the order of a matrix (measured: 16 times the whole reduction's
// error at n = 1024).
__device__ __forceinline__ long long rne(long long x, int s) {
  return (x + ((1ll << (s - 1)) - 1) + ((x >> s) & 1)) >> s;
}

// x 2^z, rounded to nearest for z < 0.
__device__ __forceinline__ long long shift(long long x, int z) {
  return z >= 0 ? x << min(z, 63) : rne(x, min(-z, 62));
}

__device__ __forceinline__ int4 pack(long long re, long long im) {
  const Limb a = split(re), b = split(im);
  return make_int4(a.h, a.l, b.h, b.l);
}

__device__ __forceinline__ int4 conj(const int4& a) { return make_int4(a.x, a.y, -a.z, -a.w); }

// Sums of products of complex values, int4 {re.h, re.l, im.h, im.l}.
struct Sum {
  long long rh = 0, rx = 0, ih = 0, ix = 0;
  __device__ __forceinline__ void add(const int4& a, const int4& b) {  // += a b
    const int2 nb = make_int2(-b.z, -b.w);
    mac(rh, a.x, b.x);
    mac(rx, a.x, b.y);
    mac(ih, a.x, b.z);
    mac(ix, a.x, b.w);
    mac(rx, a.y, b.x);
    mac(ix, a.y, b.z);
    mac(rh, a.z, nb.x);
    mac(rx, a.z, nb.y);
    mac(ih, a.z, b.x);
    mac(ix, a.z, b.y);
    mac(rx, a.w, nb.x);
    mac(ix, a.w, b.x);
  }
  __device__ __forceinline__ void add_conj(const int4& a, const int4& b) { add(a, conj(b)); }
  // (the sum in units of 2^(60 - UP), rounded)
  template <int UP = 0>
  __device__ __forceinline__ long long re() const {
    return val<UP>(rh, rx);
  }
  template <int UP = 0>
  __device__ __forceinline__ long long im() const {
    return val<UP>(ih, ix);
  }
  __device__ __forceinline__ void flush() {
    fx::flush(rh, rx);
    fx::flush(ih, ix);
  }
};

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

__device__ __forceinline__ long long warp_sum(long long v) {
#pragma unroll
  for (int o = 16; o > 0; o >>= 1) v += __shfl_xor_sync(0xFFFFFFFFu, v, o);
  return v;
}

// Unsigned 128-bit sums of squares (a difference below zero wraps).
struct U128 {
  unsigned long long hi = 0, lo = 0;
  __device__ __forceinline__ void add(unsigned long long h, unsigned long long l) {
    asm("add.cc.u64 %0, %0, %2;\n\taddc.u64 %1, %1, %3;" : "+l"(lo), "+l"(hi) : "l"(l), "l"(h));
  }
  __device__ __forceinline__ void add_square(long long x) {
    const unsigned long long u = x < 0 ? 0ull - (unsigned long long)x : (unsigned long long)x;
    add(__umul64hi(u, u), u * u);
  }
  __device__ __forceinline__ void subtract(const U128& v) {
    asm("sub.cc.u64 %0, %0, %2;\n\tsubc.u64 %1, %1, %3;"
        : "+l"(lo), "+l"(hi)
        : "l"(v.lo), "l"(v.hi));
  }
  __device__ __forceinline__ U128 shifted_right(int s) const {  // 0 < s < 64
    return {hi >> s, lo >> s | hi << (64 - s)};
  }
  __device__ __forceinline__ U128 shifted_left(int s) const {  // 0 <= s < 64
    return {hi << s | (lo >> 1) >> (63 - s), lo << s};
  }
};
__device__ __forceinline__ U128 warp_sum(U128 v) {
#pragma unroll
  for (int o = 16; o > 0; o >>= 1)
    v.add(__shfl_xor_sync(0xFFFFFFFFu, v.hi, o), __shfl_xor_sync(0xFFFFFFFFu, v.lo, o));
  return v;
}

// ---- scalars of full precision without the FP64 pipe, whose instructions
// follow one another at 70 clocks (a square root or a division takes 580).
// Each starts from the 22 bits of the approximate FP32 instruction and takes
// two Newton steps, x <- x + r / f'(x) with the exact integer residual r.

__device__ __forceinline__ float rsqrt_approx(float x) {
  float r;
  asm("rsqrt.approx.ftz.f32 %0, %1;" : "=f"(r) : "f"(x));
  return r;
}
__device__ __forceinline__ float rcp_approx(float x) {
  float r;
  asm("rcp.approx.ftz.f32 %0, %1;" : "=f"(r) : "f"(x));
  return r;
}

// sqrt(v) 2^z, to the nearest few units, in [2^58, 2^59); 0 < v < 2^122.
__device__ __forceinline__ long long sqrt_scaled(const U128& v, int* z) {
  const int lz = v.hi ? __clzll((long long)v.hi) : 64 + __clzll((long long)v.lo);
  const int sh = (lz & ~1) - 2;  // t = v 2^sh in [2^124, 2^126)
  unsigned long long th, tl;
  if (sh >= 64) {
    th = v.lo << (sh - 64);
    tl = 0;
  } else {
    th = v.hi << sh | v.lo >> (64 - sh);
    tl = v.lo << sh;
  }
  const float f = (float)(uint32_t)(th >> 38), r = rsqrt_approx(f);
  const uint32_t g = __float2uint_rn(f * r * 0x1p19f);  // sqrt(t) 2^-32, in [2^30, 2^31]
  const long long rho = (long long)(th - (unsigned long long)g * g);
  // (|rho| < 2^43: the start is within 2^-21)
  const float d = (float)(int)(rho >> 13) * r * 0x1p13f;  // rho / (2 g) 2^20
  unsigned long long s = ((unsigned long long)g << 32) + ((long long)__float2int_rn(d) << 12);
  const unsigned long long pl = s * s, ph = __umul64hi(s, s);
  const unsigned long long dl = tl - pl, dh = th - ph - (tl < pl ? 1ull : 0ull);
  const int e = (int)(uint32_t)(dh << 7 | dl >> 57);  // (t - s^2) 2^-57
  s += (long long)__float2int_rn((float)e * r * 0x1p5f);  // e 2^57 / (2 s)
  *z = sh / 2 - 4;
  return (long long)((s + 8) >> 4);
}

// 2^126 / q for q in [2^63, 2^64), to the nearest few units: in (2^62, 2^63].
__device__ __forceinline__ unsigned long long recip126(unsigned long long q) {
  const float r = rcp_approx((float)(uint32_t)(q >> 40));
  const uint32_t g = __float2uint_rn(r * 0x1p54f);  // 2^94 / q
  unsigned long long pl = q * g, ph = __umul64hi(q, g);
  unsigned long long dl = 0 - pl, dh = (1ull << 30) - ph - (pl ? 1ull : 0ull);
  const int e = (int)(uint32_t)(dh << 19 | dl >> 45);  // (2^94 - q g) 2^-45
  unsigned long long x =
      ((unsigned long long)g << 32) + ((long long)__float2int_rn((float)e * r * 0x1p25f) << 12);
  pl = q * x;
  ph = __umul64hi(q, x);
  dl = 0 - pl;
  dh = (1ull << 62) - ph - (pl ? 1ull : 0ull);
  const int e2 = (int)(uint32_t)(dh << 7 | dl >> 57);  // (2^126 - q x) 2^-57
  x += (long long)__float2int_rn((float)e2 * r * 0x1p17f);
  return x;
}

// x 2^e as a double.
__device__ __forceinline__ double to_double(long long x, int e) {
  const double d = __ll2double_rn(x);
  if (x != 0 && e > -900 && e < 900)
    return __hiloint2double(__double2hiint(d) + (e << 20), __double2loint(d));
  return scalbn(d, e);
}

}  // namespace fx
}  // namespace bg
