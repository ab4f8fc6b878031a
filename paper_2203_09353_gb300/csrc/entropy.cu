// Entanglement entropy of a batch of states (Alg. 1, "Calculate Entropy";
// Sec. 3): for each walker, the K x K Gram matrix G = X X^H of the state seen
// as the column-major K x M matrix X (K = 2^split rows: the lower spins), whose
// nonzero eigenvalues are those of rho = Psi Psi^H; then p_i = lambda_i /
// sum(lambda) and S = -sum p_i ln p_i.
//
// G comes from the library's Hermitian rank-k update (a grouped plan with
// BG_PLAN_HERK, FP64 or split precision), lower triangle; tridiag.cu reduces
// it to a real symmetric tridiagonal matrix (d, e). Here, bisect_kernel takes
// every eigenvalue of the tridiagonal matrix by bisection on the Sturm count
// (the number of eigenvalues below x), spread over the GPU, and
// entropy_sum_kernel the entropies. An FP64 count is bound by the FP64 pipe
// (3 instructions a step at 2 per clock per SM), so most of the bisection
// runs in FP32 and in pairs of floats; few eigenvalues per SM are bound by
// the counts' latency and get several lanes each. Measured: 128 matrices of
// order 256 3.05 -> 1.3 ms, 16 of order 1024 47.8 -> 3.7 ms.
#include <cuda_runtime.h>

#include <algorithm>
#include <cfloat>
#include <cmath>

#include "bgemm_internal.h"

namespace bg {
namespace {

constexpr int kEntThreads = 256;  // the entropy sums

// Sum of v over the block (all threads call it; the result reaches every thread).
// red: one double per warp.
__device__ double block_sum(double v, double* red) {
  for (int o = 16; o > 0; o >>= 1) v += __shfl_xor_sync(0xFFFFFFFFu, v, o);
  const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31, nw = blockDim.x >> 5;
  __syncthreads();  // red[] may still be read by a previous call
  if (lane == 0) red[warp] = v;
  __syncthreads();
  double s = 0.0;
  for (int i = 0; i < nw; ++i) s += red[i];  // fixed order: same value in every thread
  return s;
}

__device__ double block_max(double v, double* red) {
  for (int o = 16; o > 0; o >>= 1) v = fmax(v, __shfl_xor_sync(0xFFFFFFFFu, v, o));
  const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31, nw = blockDim.x >> 5;
  __syncthreads();
  if (lane == 0) red[warp] = v;
  __syncthreads();
  double s = red[0];
  for (int i = 1; i < nw; ++i) s = fmax(s, red[i]);
  return s;
}

// Number of eigenvalues of the symmetric tridiagonal (d, e2 = e^2) below x, by
// the three-term recurrence of the leading principal minors, p_0 = 1, p_1 = d_0 - x, p_i = (d_{i-1} - x) p_{i-1} - e_{i-2}^2
// p_{i-2}: the number of sign changes along p_0 .. p_n is the number of
// negative pivots q_i = p_i / p_{i-1}, that is, of eigenvalues below x. No
// division: a DADD, a DMUL and a DFMA a step, with the sign and zero tests
// on the bit pattern. For the matrix scaled into [-1, 1] (|d - x| <= 3,
// e^2 <= 1) a step changes |p| by a factor of at most 4 upwards, and a
// cancellation leaves at least an ulp of its terms. A zero p_i is replaced
// by -2^-60 p_{i-1} (the pivot -2^-60, below an ulp of the scaled entries:
// the pivot form's rule for a zero pivot), an exact change of the sign and
// exponent. Every 8 steps p and p_{i-1} are rescaled together by 2^-500 or
// 2^500 when p's binary exponent has left [-500, 500]: in between, no p
// leaves the normal range, and no sign changes. Each step is exact for
// d - x and e^2 perturbed by a few ulps (the rounding factors of the p's
// cancel in the ratios), so the count is exact for a matrix within a few
// ulps of the scaled one.
__device__ __forceinline__ void sturm3_step(double dx, double e2, double& p, double& pm,
                                            long long& pb, int& neg, int& cnt) {
  const double pn = fma(-e2, pm, dx * p);
  long long nb = __double_as_longlong(pn);
  if ((nb << 1) == 0) nb = (pb ^ (long long)0x8000000000000000ull) - (60ll << 52);  // -2^-60 p
  const int s = (int)((unsigned long long)nb >> 63);
  cnt += s ^ neg;
  neg = s;
  pm = p;
  pb = nb;
  p = __longlong_as_double(nb);
}

// Also returns det(T - x I) as value 2^(500 shifts).
struct SturmValue {
  int cnt, shifts;
  double value;
};

__device__ __forceinline__ SturmValue sturm_count3(const double* d, const double* e2, int n,
                                                   double x) {
  double pm = 1.0, p = d[0] - x;
  long long pb = __double_as_longlong(p);
  if ((pb << 1) == 0) pb = __double_as_longlong(-0x1p-60);
  p = __longlong_as_double(pb);
  int neg = (int)((unsigned long long)pb >> 63);
  int cnt = neg, shifts = 0;
  int i = 1;
  for (; i + 8 <= n; i += 8) {
#pragma unroll 1
    for (int u = 0; u < 8; ++u) sturm3_step(d[i + u] - x, e2[i + u - 1], p, pm, pb, neg, cnt);
    const int ex = (int)((pb >> 52) & 0x7FF) - 1023;
    if (ex > 500) {
      p *= 0x1p-500;
      pm *= 0x1p-500;
      pb = __double_as_longlong(p);
      ++shifts;
    } else if (ex < -500) {
      p *= 0x1p500;
      pm *= 0x1p500;
      pb = __double_as_longlong(p);
      --shifts;
    }
  }
  for (; i < n; ++i) sturm3_step(d[i] - x, e2[i - 1], p, pm, pb, neg, cnt);
  return {cnt, shifts, p};
}

// The same recurrence in FP32 on the float copy of the scaled matrix, the
// rescaling by 2^-60 / 2^60 checked at every step and a zero p_i replaced
// by -2^-24 p_{i-1}. Its backward error, a few FP32 ulps of the scaled
// entries, stays below the 32 x 2^-24 by which the FP32 brackets are
// widened.
__device__ __forceinline__ int sturm_count3f(const float4* de, int n, float x) {
  float pm = 1.0f, p = de[0].x - x;
  if (p == 0.0f) p = -0x1p-24f;
  bool neg = p < 0.0f;
  int cnt = neg;
  for (int i = 1; i < n; ++i) {
    const float4 v = de[i];  // (d_i, -, e_{i-1}^2, -)
    float pn = fmaf(-v.z, pm, (v.x - x) * p);
    if (pn == 0.0f) pn = -0x1p-24f * p;
    const bool s = pn < 0.0f;
    cnt += s != neg;
    neg = s;
    pm = p;
    p = pn;
    const int ex = (int)((__float_as_uint(p) >> 23) & 0xFF) - 127;
    if (ex > 60) {
      p *= 0x1p-60f;
      pm *= 0x1p-60f;
    } else if (ex < -60) {
      p *= 0x1p60f;
      pm *= 0x1p60f;
    }
  }
  return cnt;
}

// The same recurrence on pairs of floats (the value hi + lo, 48 bits):
// products by Dekker's error-free transformation with FMA, their difference
// by Knuth's two-sum of the high parts and one addition of the low ones. The
// rounding of a step is at most about 10 x 2^-48 of each of its two products
// (the dropped low x low term of the product with d - x is below 2^-48 of p),
// which perturbs d - x (at most 3) and e^2 (at most 1) by that much, so the
// count is exact for a matrix within 2^-42 of the scaled one. A step takes
// about 30 FP32 instructions at 128 per clock per SM, against three FP64 ones
// at 2: six times faster. p is kept within 2^-40 .. 2^40 by powers of 2^60.
__device__ __forceinline__ int sturm_count3ff(const float4* de, int n, float xh, float xl) {
  // de[i] = (d_i hi, d_i lo, e_{i-1}^2 hi, e_{i-1}^2 lo)
  float ph = 1.0f, pl = 0.0f, mh = 0.0f, ml = 0.0f;
  bool neg = false;
  int cnt = 0;
#pragma unroll 4
  for (int i = 0; i < n; ++i) {
    const float4 v = de[i];
    // d - x
    const float th = __fsub_rn(v.x, xh), tb = __fsub_rn(th, v.x);
    const float tl = __fadd_rn(__fsub_rn(__fsub_rn(v.x, __fsub_rn(th, tb)), __fadd_rn(xh, tb)),
                               __fsub_rn(v.y, xl));
    // (d - x) p and e^2 p_{i-2}
    const float ah = __fmul_rn(th, ph);
    const float al = __fmaf_rn(th, pl, __fmaf_rn(tl, ph, __fmaf_rn(th, ph, -ah)));
    const float bh = __fmul_rn(v.z, mh);
    const float bl = __fmaf_rn(v.z, ml, __fmaf_rn(v.w, mh, __fmaf_rn(v.z, mh, -bh)));
    const float sh = __fsub_rn(ah, bh), sb = __fsub_rn(sh, ah);
    const float sl = __fsub_rn(__fsub_rn(ah, __fsub_rn(sh, sb)), __fadd_rn(bh, sb));
    const float lo = __fadd_rn(sl, __fsub_rn(al, bl));
    mh = ph;
    ml = pl;
    ph = __fadd_rn(sh, lo);
    pl = __fsub_rn(lo, __fsub_rn(ph, sh));
    if (ph == 0.0f) {  // a zero minor: the pivot -2^-48
      ph = -0x1p-48f * mh;
      pl = 0.0f;
    }
    const bool s = ph < 0.0f;
    cnt += s != neg;
    neg = s;
    const uint32_t ex = (__float_as_uint(ph) >> 23) & 0xFF;
    if (ex - 87u > 80u) {
      const float f = ex > 127u ? 0x1p-60f : 0x1p60f;
      ph *= f;
      pl *= f;
      mh *= f;
      ml *= f;
    }
  }
  return cnt;
}

// One narrowing of the bracket [a, b] of eigenvalue k by P >= 2 lanes, one
// point each: `below` says whether this lane's point j (at a + w (j + 1) /
// (P + 1)) has at most k eigenvalues below it. Returns how many points, from
// the first on, do.
template <int P>
__device__ __forceinline__ int points_below(bool below) {
  const uint32_t all = __ballot_sync(0xFFFFFFFFu, below);
  const uint32_t mask = P == 32 ? all : (all >> (threadIdx.x & 31 & ~(P - 1))) & ((1u << (P & 31)) - 1u);
  return P == 32 && mask == 0xFFFFFFFFu ? 32 : __ffs(~mask) - 1;
}

// Eigenvalues of each walker's tridiagonal matrix (blockIdx.y) by bisection,
// kBisThreads / P of them per CTA, P lanes to each. The matrix is scaled by a
// power of two into [-1, 1] and counted by the three-term recurrence, in
// three precisions, each narrowing the bracket down to its own error bound:
// in FP32 to 32 x 2^-24, in float pairs to 2^-40, then FP64. A bracket [a, b]
// with count(a) <= k < count(b) in one precision holds lambda_k within
// [a - del, b + del]. In FP64, a bracket that holds one eigenvalue is closed
// around the secant of det(T - x I) over it, two counts either side of that
// point proving the result; otherwise (a cluster, or a secant that missed)
// the bisection goes on. That leaves about 5 FP64 counts per eigenvalue of
// the 35 that bisecting from the FP32 bracket took.
// P: the lanes cut the bracket into P + 1 parts per count, so that fewer counts
// follow one another.
// Dynamic shared memory: d and e^2 (2 n doubles), the same as float pairs
// (n float4).
constexpr int kBisThreads = 128;
template <int P>
__global__ void __launch_bounds__(kBisThreads) bisect_kernel(const double* d, const double* e,
                                                             int n, double* lam) {
  extern __shared__ float4 sde[];
  double* sd = reinterpret_cast<double*>(sde + n);
  double* se2 = sd + n;
  __shared__ double red[kBisThreads / 32];
  __shared__ int cnt[kBisThreads + 1];
  const int t = threadIdx.x;
  constexpr int T = kBisThreads;
  const double* dw = d + (size_t)blockIdx.y * n;
  const double* ew = e + (size_t)blockIdx.y * n;
  double lo = DBL_MAX, hi = -DBL_MAX;
  bool finite = true;
  for (int i = t; i < n; i += T) {
    // Gershgorin interval of row i
    const double di = dw[i];
    const double r = (i + 1 < n ? fabs(ew[i]) : 0.0) + (i > 0 ? fabs(ew[i - 1]) : 0.0);
    lo = fmin(lo, di - r);
    hi = fmax(hi, di + r);
    finite = finite && fabs(di) <= DBL_MAX && r <= DBL_MAX;
  }
  finite = __syncthreads_and(finite);
  lo = -block_max(-lo, red);
  hi = block_max(hi, red);
  const double scale = fmax(fabs(lo), fabs(hi));
  const int kt = blockIdx.x * (T / P) + t / P, k = min(kt, n - 1), j = t % P;
  const bool store = j == 0 && kt < n;
  const size_t at = (size_t)blockIdx.y * n + k;
  if (!finite || scale == 0.0 || scale > DBL_MAX) {  // uniform over the CTA
    const double v = finite && scale == 0.0 ? 0.0 : __longlong_as_double(0x7FF8000000000000ll);
    if (store) lam[at] = v;
    return;
  }
  int ex = 0;
  frexp(scale, &ex);  // scale 2^-ex in [0.5, 1)
  for (int i = t; i < n; i += T) {
    const double di = scalbn(dw[i], -ex);
    const double es = i > 0 ? scalbn(ew[i - 1], -ex) : 0.0;
    const double e2 = es * es;
    sd[i] = di;
    if (i > 0) se2[i - 1] = e2;
    const float dh = (float)di, eh = (float)e2;
    sde[i] = make_float4(dh, (float)(di - (double)dh), eh, (float)(e2 - (double)eh));
  }
  lo = scalbn(lo, -ex);
  hi = scalbn(hi, -ex);
  const double tol = 2.0 * DBL_EPSILON * fmax(fabs(lo), fabs(hi));
  __syncthreads();
  // multisection: one FP32 count per thread on an even grid gives every
  // eigenvalue a bracket T times narrower to start from (the ends widened
  // by twice the FP32 bound, so that the counts there are 0 and n)
  constexpr float del32 = 32.0f * 0x1p-24f;
  const float lo32 = (float)lo - 2.0f * del32, hi32 = (float)hi + 2.0f * del32;
  const float h32 = (hi32 - lo32) / (float)T;
  auto grid32 = [&](int i) { return __fmaf_rn((float)i, h32, lo32); };
  cnt[t + 1] = t + 1 < T ? sturm_count3f(sde, n, grid32(t + 1)) : n;
  if (t == 0) cnt[0] = 0;
  __syncthreads();
  // the k-th smallest eigenvalue: count(a) <= k < count(b)
  int lo_i = 0, hi_i = T;
  while (hi_i - lo_i > 1) {
    const int mid = (lo_i + hi_i) >> 1;
    if (cnt[mid] <= k) lo_i = mid;
    else hi_i = mid;
  }
  constexpr float kPart = 1.0f / (float)(P + 1);
  float a32 = grid32(lo_i), b32 = lo_i + 1 < T ? grid32(lo_i + 1) : hi32;
  for (int it = 0; it < 40 && __any_sync(0xFFFFFFFFu, b32 - a32 > del32); ++it) {
    const float w = (b32 - a32) * kPart;
    const int m = points_below<P>(sturm_count3f(sde, n, __fmaf_rn((float)(j + 1), w, a32)) <= k);
    if (b32 - a32 > del32) {
      const float a0 = a32;
      if (m > 0) a32 = __fmaf_rn((float)m, w, a0);
      if (m < P) b32 = __fmaf_rn((float)(m + 1), w, a0);
    }
  }
  double a = (double)a32 - (double)del32, b = (double)b32 + (double)del32;
  constexpr double delff = 0x1p-40;
  for (int it = 0; it < 60 && __any_sync(0xFFFFFFFFu, b - a > delff); ++it) {
    const double w = (b - a) * (1.0 / (P + 1));
    // (the points are pairs of floats: rounding x to 48 bits moves it by less than the bound)
    const double x = fma((double)(j + 1), w, a);
    const float xh = (float)x, xl = (float)(x - (double)xh);
    const int m = points_below<P>(sturm_count3ff(sde, n, xh, xl) <= k);
    if (b - a > delff) {
      const double a0 = a;
      if (m > 0) a = fma((double)m, w, a0);
      if (m < P) b = fma((double)(m + 1), w, a0);
    }
  }
  a -= delff;
  b += delff;
  // two points at once, by the even and the odd lanes
  auto two = [&](double x0, double x1, SturmValue& v0, SturmValue& v1) {
    const SturmValue v = sturm_count3(sd, se2, n, (j & 1) ? x1 : x0);
    const int l0 = t & 31 & ~(P - 1);
    v0.cnt = __shfl_sync(0xFFFFFFFFu, v.cnt, l0);
    v0.shifts = __shfl_sync(0xFFFFFFFFu, v.shifts, l0);
    v0.value = __shfl_sync(0xFFFFFFFFu, v.value, l0);
    v1.cnt = __shfl_sync(0xFFFFFFFFu, v.cnt, l0 + 1);
    v1.shifts = __shfl_sync(0xFFFFFFFFu, v.shifts, l0 + 1);
    v1.value = __shfl_sync(0xFFFFFFFFu, v.value, l0 + 1);
  };
  SturmValue va, vb;
  two(a, b, va, vb);
  double x0 = a, x1 = b;
  if (va.cnt > k) {  // outside the bracket after all: take the whole interval below
    b = a;
    a = lo - 4.0 * tol;
  } else if (vb.cnt <= k) {
    a = b;
    b = hi + 4.0 * tol;
  } else if (vb.cnt - va.cnt == 1 && va.shifts == vb.shifts) {
    const double fa = fabs(va.value), fb = fabs(vb.value);
    const double x = fma(b - a, fa / (fa + fb), a);
    x0 = fmax(a, x - tol);
    x1 = fmin(b, x + tol);
  }
  // (a lane with no secant asks again for the ends of its bracket, or stays at x0 = x1)
  SturmValue w0, w1;
  two(x0, x1, w0, w1);
  if (x0 >= a && x1 <= b) {
    if (w0.cnt <= k) a = fmax(a, x0);
    else b = fmin(b, x0);
    if (w1.cnt > k) b = fmin(b, x1);
    else a = fmax(a, x1);
  }
  // near zero (the empty part of a low-entropy spectrum) the bisection goes on
  // to 2^-58: there are many such eigenvalues, and -p ln p is steep
  auto open = [&]() { return b - a > (fmax(fabs(a), fabs(b)) < 0x1p-10 ? 0x1p-58 : tol); };
  for (int it = 0; it < 200 && __any_sync(0xFFFFFFFFu, open()); ++it) {
    const double w = (b - a) * (1.0 / (P + 1));
    const int m =
        points_below<P>(sturm_count3(sd, se2, n, fma((double)(j + 1), w, a)).cnt <= k);
    if (open()) {
      const double a0 = a;
      if (m > 0) a = fma((double)m, w, a0);
      if (m < P) b = fma((double)(m + 1), w, a0);
    }
  }
  if (store) lam[at] = scalbn(0.5 * (a + b), ex);
}

// S = -sum p ln p over p = lambda / sum(lambda) > 0, T threads per walker: a CTA,
// or a warp where n <= 32 (16000 walkers of order 2: 254 us with a CTA each); eigs
// (optional) receives the eigenvalues in ascending order: two that lie within
// the bisection's tolerance of each other may come in either order, so each
// takes the largest value up to it.
template <int T>
__global__ void __launch_bounds__(kEntThreads)
    entropy_sum_kernel(const double* lam, int64_t walkers, int n, double* entropy, double* eigs) {
  static_assert(T == 32 || T == kEntThreads, "a warp or the CTA per walker");
  constexpr bool kWarp = T == 32;
  __shared__ double red[kEntThreads / 32];
  __shared__ double top[2][kEntThreads];
  const int t = threadIdx.x % T;
  const int64_t w = blockIdx.x * (int64_t)(kEntThreads / T) + threadIdx.x / T;
  if (w >= walkers) return;
  auto sum = [&](double v) {
    if constexpr (!kWarp) return block_sum(v, red);
    for (int o = 16; o > 0; o >>= 1) v += __shfl_xor_sync(0xFFFFFFFFu, v, o);
    return v;
  };
  const double* l = lam + (size_t)w * n;
  double tot = 0.0;
  for (int k = t; k < n; k += T) tot += l[k];
  tot = sum(tot);
  double s = tot != tot ? tot : 0.0;
  for (int k = t; k < n; k += T) {
    const double p = tot > 0.0 ? l[k] / tot : 0.0;
    if (p > 0.0) s -= p * log(p);
  }
  s = sum(s);
  if (t == 0) entropy[w] = s;
  if (!eigs) return;
  const int per = (n + T - 1) / T, k0 = t * per, k1 = min(n, k0 + per);
  double m = -DBL_MAX;
  for (int k = k0; k < k1; ++k) m = fmax(m, l[k]);
  // running maximum over the threads before this one
  if constexpr (kWarp) {
    for (int o = 1; o < 32; o <<= 1) {
      const double v = __shfl_up_sync(0xFFFFFFFFu, m, o);
      if (t >= o) m = fmax(m, v);
    }
    m = __shfl_up_sync(0xFFFFFFFFu, m, 1);
  } else {
    top[0][t] = m;
    __syncthreads();
    int cur = 0;
    for (int o = 1; o < T; o <<= 1, cur ^= 1) {
      top[cur ^ 1][t] = t >= o ? fmax(top[cur][t], top[cur][t - o]) : top[cur][t];
      __syncthreads();
    }
    m = t > 0 ? top[cur][t - 1] : 0.0;
  }
  if (t == 0) m = -DBL_MAX;
  for (int k = k0; k < k1; ++k) {
    const double v = l[k];
    m = fmax(m, v);
    eigs[(size_t)w * n + k] = v != v ? v : m;
  }
}

template <int P>
cudaError_t bisect_launch(const double* d, const double* e, int64_t walkers, int n, double* lam,
                          cudaStream_t st) {
  // (n <= 1024: at most 32 KB, which needs no raised limit)
  constexpr int per = kBisThreads / P;
  bisect_kernel<P><<<dim3((unsigned)((n + per - 1) / per), (unsigned)walkers), kBisThreads,
                     (size_t)n * 32, st>>>(d, e, n, lam);
  count_launch();
  return cudaGetLastError();
}

}  // namespace

// Lanes per eigenvalue, by the eigenvalues per SM: more lanes shorten the chain
// of dependent counts but add counts, so each line lies where the pipes fill.
// Measured (us, with 1 / 2 / 4 / 8 / 16 / 32 lanes; eigenvalues per SM first):
//   1.7 (4 of order 64)    211   145  113   99   86   82
//   6.7 (1 of 1024)       5200  3280 2450 1900 1720 1990
//   13  (8 of 256)        1310   516  621  351  442  712
//   27  (32 of 128)        403   268  206  256  381  582
//   54  (128 of 64)        210   145  150  217  318  573
//   108 (16 of 1024)      5200  3900 4110 4910 8240
//   216 (128 of 256)      1610  1280 1490 2050 3770
//   1700 (4096 of 64)     2025  1300 2300
// One lane was the fastest nowhere and is not built.
cudaError_t launch_entropy_bisect(const double* d, const double* e, int64_t walkers, int n,
                                  double* lam, double* entropy, double* eigs, int sms,
                                  cudaStream_t st) {
  if (walkers <= 0) return cudaSuccess;
  const int64_t per_sm = (walkers * n + sms - 1) / sms;
  cudaError_t err = per_sm <= 4    ? bisect_launch<32>(d, e, walkers, n, lam, st)
                    : per_sm <= 10 ? bisect_launch<16>(d, e, walkers, n, lam, st)
                    : per_sm <= 20 ? bisect_launch<8>(d, e, walkers, n, lam, st)
                    : per_sm <= 40 ? bisect_launch<4>(d, e, walkers, n, lam, st)
                                   : bisect_launch<2>(d, e, walkers, n, lam, st);
  if (err != cudaSuccess) return err;
  if (n <= 32)
    entropy_sum_kernel<32><<<(unsigned)((walkers + kEntThreads / 32 - 1) / (kEntThreads / 32)),
                             kEntThreads, 0, st>>>(lam, walkers, n, entropy, eigs);
  else
    entropy_sum_kernel<kEntThreads><<<(unsigned)walkers, kEntThreads, 0, st>>>(lam, walkers, n,
                                                                             entropy, eigs);
  count_launch();
  return cudaGetLastError();
}

}  // namespace bg
