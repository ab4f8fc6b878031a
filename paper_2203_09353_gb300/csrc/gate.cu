// Local two-spin gate of the annealing step (Sec. 2 and Alg. 1, "Apply Local
// Gate"): a 4 x 4 unitary U_w on spins (j, j+1) of each walker's state vector
// psi_w of 2^S complex amplitudes, in place:
//
//   psi_w'[x] = sum_{c=0..3} U_w[a(x), c] psi_w[x - a(x) 2^j + c 2^j],
//   a(x) = b_j(x) + 2 b_{j+1}(x),  b_i(x) = bit i of x (spin i).
//
// The 2^S amplitudes fall into 2^(S-2) independent groups of four (the basis
// states that differ only in spins j and j+1). One thread owns one group:
// it reads the four amplitudes, multiplies by U_w held in registers, and
// writes the four results back, so every amplitude is read and written once
// and no two threads touch the same one. Group g starts at x0 = g with two
// zero bits inserted at bit j; consecutive threads take consecutive g, which
// for j >= 5 makes each of the four loads 32 neighbouring amplitudes.
//
// Bound: HBM, with the integer pipe close behind. An amplitude costs 16 real
// multiply-adds against 32 bytes moved. At 2 DFMA per clock per SM the FP64
// pipe took 8 clocks for that: 3.67 ms for 1024 states of 17 spins, 17% of the
// copy bandwidth. In fixed point (fixed60.cuh), with three real products per
// complex one (Gauss's form), it is 36 integer multiply-adds, 1.1 clocks,
// where the copy bandwidth allows 1.4; with the conversions around them it
// measured 0.97 ms, 65% of the copy bandwidth (four real products: 1.04 ms).
// A group's four amplitudes get one exponent, 59 bits below the largest
// component (2^E above it), the gate's entries another (2^EU); the sums are in
// units of 2^(E + EU - 58), rounded to nearest and then once more to FP64.
//
// The error before that last rounding comes from the cut of the operands to 59
// bits, the dropped products of two low limbs and the rounding of the cross
// sums: 0.4 units rms (0.5 for one large amplitude), 13 at most. With the last
// rounding, Haar gates on random amplitudes are off by 31 x 2^-60 of the
// group's largest component rms, the FP64 chain by 65; one large amplitude in
// a group: 22 against 59. The chain's error goes with the sum of |U| |psi| over
// a row, the fixed form's with the largest of each: an output that only small
// entries of U meet can be the less exact one (4% of them with one large
// amplitude), by a few units. A gate with an entry below 2^-6 of its largest (a
// permutation, a controlled gate, 1% of random ones) keeps the FP64 chain for
// its walker, exact where its entries are. So do groups with an infinity, a NaN
// or magnitudes within a factor 2^300 of the ends of the range.
#include <algorithm>

#include "bgemm_internal.h"
#include "fixed60.cuh"

namespace bg {

namespace {

constexpr int kGateThreads = 256;

// Same protocol as the other kernels' error word: the first code wins, the
// count keeps growing.
__device__ __forceinline__ void gate_error(int* err, int walker) {
  if (atomicCAS(err, 0, (int)BG_ERR_INVALID_ARG) == 0) {
    err[1] = ERRLOC_GATE_SITE;
    err[2] = walker;
  }
  atomicAdd(err + 3, 1);
}

constexpr int kGateSmall = 6;                   // log2 of the largest ratio of U's entries
constexpr int kGateLowExp = 300, kGateHighExp = 1700;  // biased exponents of the fixed form

__device__ __forceinline__ uint32_t magnitude_hi(double x) {
  return (uint32_t)__double2hiint(x) & 0x7FFFFFFFu;
}

// |x| 2^(59 - E) cut to an integer and put into limbs, with x's sign, for
// biased exponent top = E + 1022 of a normal magnitude no smaller than x's
// (zero and subnormal x give 0).
__device__ __forceinline__ fx::Limb to_fixed59(double x, int top) {
  const uint32_t xh = (uint32_t)__double2hiint(x), xl = (uint32_t)__double2loint(x);
  const uint32_t r = (uint32_t)(top - (int)((xh >> 20) & 0x7FF));  // places to the right
  const uint32_t mh = (xh & 0xFFFFFu) | 0x100000u;
  // the significand at the top of 59 bits, then r places to the right
  uint32_t H = __funnelshift_l(xl, mh, 6), L = xl << 6;
  L = r < 32 ? __funnelshift_r(L, H, r) : __funnelshift_rc(H, 0u, r - 32);
  H = __funnelshift_rc(H, 0u, r);
  // balanced limbs: add 2^29, cut at bit 30, subtract 2^29 from the low one
  const unsigned long long V = ((unsigned long long)H << 32 | L) + (1u << 29);
  const int s = (int)xh >> 31;
  const int h = (int)(uint32_t)(V >> 30), l = (int)((uint32_t)V & 0x3FFFFFFFu) - (1 << 29);
  return {(h ^ s) - s, (l ^ s) - s};
}

// X 2^k as a double, rounded to nearest even; the result is zero or normal.
__device__ __forceinline__ double scaled_double(long long X, int k) {
  const double d = __ll2double_rn(X);
  const int hi = __double2hiint(d);
  return __hiloint2double(X != 0 ? hi + (k << 20) : hi, __double2loint(d));
}

__device__ __forceinline__ void gate_fp64(const double2* g, const double2 (&v)[4],
                                          double2 (&o)[4]) {
#pragma unroll
  for (int a = 0; a < 4; ++a) {
    double re = 0.0, im = 0.0;
#pragma unroll
    for (int c = 0; c < 4; ++c) {
      const double2 uc = __ldg(g + a + 4 * c);
      re = fma(uc.x, v[c].x, fma(-uc.y, v[c].y, re));
      im = fma(uc.x, v[c].y, fma(uc.y, v[c].x, im));
    }
    o[a] = make_double2(re, im);
  }
}

// src and dst may be the same array (in place). A walker with a bad site is
// left as it is: copied when dst is another array.
__global__ void __launch_bounds__(kGateThreads, 3)
    local_gate_kernel(int64_t walkers, int spins, const int32_t* sites, const double2* gates,
                      const double2* src, int64_t src_stride, double2* dst, int64_t dst_stride,
                      int* err) {
  const int64_t w = blockIdx.y + (int64_t)blockIdx.z * gridDim.y;
  if (w >= walkers) return;
  const int j = __ldg(sites + w);
  const double2* psi = src + w * src_stride;
  double2* out = dst + w * dst_stride;
  const int64_t first = blockIdx.x * (int64_t)blockDim.x + threadIdx.x;
  const int64_t stride = (int64_t)gridDim.x * blockDim.x;
  if (j < 0 || j > spins - 2) {
    if (blockIdx.x == 0 && threadIdx.x == 0) gate_error(err, (int)w);
    if (psi != out)
      for (int64_t x = first; x < (int64_t)1 << spins; x += stride) out[x] = psi[x];
    return;
  }
  const double2* g = gates + 16 * w;  // U_w column-major: g[a + 4 c] = U[a, c]
  // U in limbs, 59 bits below its largest entry, with Re + Im beside it, and
  // whether its entries lie close enough together
  __shared__ int4 u[16];
  __shared__ int2 us[16];
  __shared__ int s_utop, s_fixed;
  if (threadIdx.x < 32) {
    const int e = threadIdx.x & 15;
    const double2 z = __ldg(g + e);
    uint32_t umax = max(magnitude_hi(z.x), magnitude_hi(z.y)), umin = umax;
#pragma unroll
    for (int o = 8; o > 0; o >>= 1) {
      umax = max(umax, __shfl_xor_sync(0xFFFFFFFFu, umax, o));
      umin = min(umin, __shfl_xor_sync(0xFFFFFFFFu, umin, o));
    }
    const int top = (int)(umax >> 20);
    const long long re = fx::from_double(z.x, 59 - (top - 1022));
    const long long im = fx::from_double(z.y, 59 - (top - 1022));
    const fx::Limb sum = fx::split(re + im);
    if (threadIdx.x < 16) {
      u[e] = fx::pack(re, im);
      us[e] = make_int2(sum.h, sum.l);
    }
    if (threadIdx.x == 0) {
      s_utop = top;
      s_fixed = (umin >> 20) + kGateSmall >= (umax >> 20) && top > 895 && top < 1151;
    }
  }
  __syncthreads();
  const int utop = s_utop;
  const bool fixed = s_fixed != 0;
  const int64_t groups = (int64_t)1 << (spins - 2);
  const int64_t low = ((int64_t)1 << j) - 1;
  const int64_t step = (int64_t)1 << j;
  auto base = [&](int64_t q) { return ((q & ~low) << 2) | (q & low); };
  if (!fixed) {
    for (int64_t q = first; q < groups; q += stride) {
      const int64_t x0 = base(q);
      double2 v[4], o[4];
#pragma unroll
      for (int c = 0; c < 4; ++c) v[c] = psi[x0 + c * step];
      gate_fp64(g, v, o);
#pragma unroll
      for (int a = 0; a < 4; ++a) out[x0 + a * step] = o[a];
    }
    return;
  }
  for (int64_t q = first; q < groups; q += stride) {
    const int64_t x0 = base(q);
    double2 v[4];
#pragma unroll
    for (int c = 0; c < 4; ++c) v[c] = psi[x0 + c * step];
    uint32_t m = 0;
#pragma unroll
    for (int c = 0; c < 4; ++c) m = max(m, max(magnitude_hi(v[c].x), magnitude_hi(v[c].y)));
    const int top = (int)(m >> 20);
    double2 o[4];
    if (top > kGateLowExp && top < kGateHighExp) {
      int4 f[4];
      int2 fs[4];  // Re + Im
#pragma unroll
      for (int c = 0; c < 4; ++c) {
        const fx::Limb re = to_fixed59(v[c].x, top), im = to_fixed59(v[c].y, top);
        f[c] = make_int4(re.h, re.l, im.h, im.l);
        fs[c] = make_int2(re.h + im.h, re.l + im.l);
      }
      // psi = f 2^(E - 59), U = u 2^(EU - 59): the sums are in 2^(E + EU - 58).
      // The cross sums stay below 2^61 (x1, x2) and 4 (2^30 2^30 + 2^30 2^29) < 2^63 (x3).
      // They are rounded to nearest (cut, every result was half a unit low on average).
      const int k = (top - 1022) + (utop - 1022) - 58;
#pragma unroll
      for (int a = 0; a < 4; ++a) {
        long long h1 = 0, x1 = 0, h2 = 0, x2 = 0, h3 = 0, x3 = 0;
#pragma unroll
        for (int c = 0; c < 4; ++c) {
          const int4 uc = u[a + 4 * c];
          const int2 sc = us[a + 4 * c];
          fx::mac(h1, uc.x, f[c].x);
          fx::mac(x1, uc.x, f[c].y);
          fx::mac(x1, uc.y, f[c].x);
          fx::mac(h2, uc.z, f[c].z);
          fx::mac(x2, uc.z, f[c].w);
          fx::mac(x2, uc.w, f[c].z);
          fx::mac(h3, sc.x, fs[c].x);
          fx::mac(x3, sc.x, fs[c].y);
          fx::mac(x3, sc.y, fs[c].x);
        }
        o[a] = make_double2(
            scaled_double(h1 - h2 + ((x1 - x2 + (1 << (fx::kLow - 1))) >> fx::kLow), k),
            scaled_double(h3 - h1 - h2 + (((x3 >> 1) - ((x1 + x2) >> 1) + (1 << (fx::kLow - 2))) >>
                                          (fx::kLow - 1)),
                          k));
      }
    } else if (m == 0) {  // (the FP64 chain gives +0 as well)
#pragma unroll
      for (int a = 0; a < 4; ++a) o[a] = make_double2(0.0, 0.0);
    } else {
      gate_fp64(g, v, o);
    }
#pragma unroll
    for (int a = 0; a < 4; ++a) out[x0 + a * step] = o[a];
  }
}

}  // namespace

cudaError_t launch_local_gate(int64_t walkers, int spins, const int32_t* sites, const void* gates,
                              const void* src, int64_t src_stride, void* dst, int64_t dst_stride,
                              int* d_err, int sms, cudaStream_t st) {
  if (walkers <= 0) return cudaSuccess;
  const int64_t groups = (int64_t)1 << (spins - 2);
  // CTAs per walker: the fewest groups per SM slot, counting whole waves of
  // three CTAs per SM, whole rounds of 256 groups per CTA and one round for a
  // CTA's start (site, gate and its limbs)
  const int64_t slots = (int64_t)sms * 3;
  const int64_t rounds = (groups + kGateThreads - 1) / kGateThreads;
  int64_t gx = 1, best = INT64_MAX;
  for (int64_t x = 1; x <= std::min<int64_t>(rounds, 64); ++x) {
    const int64_t waves = (walkers * x + slots - 1) / slots;
    const int64_t cost = waves * ((rounds + x - 1) / x + 1);
    if (cost < best) {
      best = cost;
      gx = x;
    }
  }
  if (rounds > 64 && walkers < slots / 64)  // few large states: fill the GPU
    gx = std::min<int64_t>(rounds, slots / std::max<int64_t>(1, walkers));
  const int64_t gy = std::min<int64_t>(walkers, 65535);
  const int64_t gz = (walkers + gy - 1) / gy;
  if (gz > 65535) return cudaErrorInvalidConfiguration;
  local_gate_kernel<<<dim3((unsigned)gx, (unsigned)gy, (unsigned)gz), kGateThreads, 0, st>>>(
      walkers, spins, sites, static_cast<const double2*>(gates),
      static_cast<const double2*>(src), src_stride, static_cast<double2*>(dst), dst_stride,
      d_err);
  count_launch();
  return cudaGetLastError();
}

}  // namespace bg
