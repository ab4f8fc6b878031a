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
// (the number of eigenvalues below x), one thread per eigenvalue, then the
// entropy by a block reduction; it is bound by the FP64 pipe (about 2 DFMA
// per clock per SM on this part), not by memory.
#include <cuda_runtime.h>

#include <algorithm>
#include <cfloat>
#include <cmath>

#include "bgemm_internal.h"

namespace bg {
namespace {

constexpr int kEntThreads = 256;  // bisection
// A kernel's dynamic shared-memory limit is a property of the device: set it
// once per device (at every call for ordinals beyond the table).
constexpr int kAttrDevices = 64;
template <typename Kernel>
cudaError_t smem_limit(Kernel kernel, int bytes, bool (&done)[kAttrDevices]) {
  int dev = 0;
  cudaError_t e = cudaGetDevice(&dev);
  if (e != cudaSuccess) return e;
  const bool tracked = dev >= 0 && dev < kAttrDevices;
  if (tracked && done[dev]) return cudaSuccess;
  e = cudaFuncSetAttribute(kernel, cudaFuncAttributeMaxDynamicSharedMemorySize, bytes);
  if (e == cudaSuccess && tracked) done[dev] = true;
  return e;
}

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

// 1/q for a normal q: the hardware's approximate reciprocal, then two
// Newton-Raphson steps r <- r + r (1 - q r), each of which squares the
// relative error (to well below 2^-80, so r is within an ulp or so of 1/q).
// On this part an FP64 instruction is slow; this takes five of them where
// an IEEE division takes about twice as many.
__device__ __forceinline__ double recip_nr(double q) {
  double r;
  asm("rcp.approx.ftz.f64 %0, %1;" : "=d"(r) : "d"(q));
  double e = fma(-q, r, 1.0);
  r = fma(r, e, r);
  e = fma(-q, r, 1.0);
  return fma(r, e, r);
}

// Number of eigenvalues of the symmetric tridiagonal (d, e2 = e^2) below x:
// the negative pivots of T - x I (a pivot smaller than pivmin in magnitude
// is replaced by -pivmin, as in LAPACK's dstebz). The pivot recurrence
// q_i = (d_i - x) - e2_{i-1} / q_{i-1} is backward stable: the count is exact
// for entries perturbed by a few ulps, which also covers a quotient formed
// with a reciprocal that is not correctly rounded. The sign and the pivmin
// test read the bit pattern (integer compares of |q|'s bits order like the
// magnitudes), so that they stay off the FP64 pipe.
__device__ __forceinline__ int sturm_count(const double* d, const double* e2, int n, double x,
                                           double pivmin) {
  const long long pmin_bits = __double_as_longlong(pivmin);
  const double neg_pmin = -pivmin;
  double q = d[0] - x;
  long long qb = __double_as_longlong(q);
  if ((qb & 0x7FFFFFFFFFFFFFFFll) < pmin_bits) {
    q = neg_pmin;
    qb = __double_as_longlong(q);
  }
  int cnt = (int)((unsigned long long)qb >> 63);
  for (int i = 1; i < n; ++i) {
    q = fma(-e2[i - 1], recip_nr(q), d[i] - x);
    qb = __double_as_longlong(q);
    if ((qb & 0x7FFFFFFFFFFFFFFFll) < pmin_bits) {
      q = neg_pmin;
      qb = __double_as_longlong(q);
    }
    cnt += (int)((unsigned long long)qb >> 63);
  }
  return cnt;
}

// The same count by the three-term recurrence of the leading principal
// minors, p_0 = 1, p_1 = d_0 - x, p_i = (d_{i-1} - x) p_{i-1} - e_{i-2}^2
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

__device__ __forceinline__ int sturm_count3(const double* d, const double* e2, int n, double x) {
  double pm = 1.0, p = d[0] - x;
  long long pb = __double_as_longlong(p);
  if ((pb << 1) == 0) pb = __double_as_longlong(-0x1p-60);
  p = __longlong_as_double(pb);
  int neg = (int)((unsigned long long)pb >> 63);
  int cnt = neg;
  int i = 1;
  for (; i + 8 <= n; i += 8) {
#pragma unroll 1
    for (int u = 0; u < 8; ++u) sturm3_step(d[i + u] - x, e2[i + u - 1], p, pm, pb, neg, cnt);
    const int ex = (int)((pb >> 52) & 0x7FF) - 1023;
    if (ex > 500) {
      p *= 0x1p-500;
      pm *= 0x1p-500;
      pb = __double_as_longlong(p);
    } else if (ex < -500) {
      p *= 0x1p500;
      pm *= 0x1p500;
      pb = __double_as_longlong(p);
    }
  }
  for (; i < n; ++i) sturm3_step(d[i] - x, e2[i - 1], p, pm, pb, neg, cnt);
  return cnt;
}

// The same recurrence in FP32 on the float copy of the scaled matrix, the
// rescaling by 2^-60 / 2^60 checked at every step and a zero p_i replaced
// by -2^-24 p_{i-1}. Its backward error, a few FP32 ulps of the scaled
// entries, stays below the 32 x 2^-24 by which the FP32 brackets are
// widened.
__device__ __forceinline__ int sturm_count3f(const float* d, const float* e2, int n, float x) {
  float pm = 1.0f, p = d[0] - x;
  if (p == 0.0f) p = -0x1p-24f;
  bool neg = p < 0.0f;
  int cnt = neg;
  for (int i = 1; i < n; ++i) {
    float pn = fmaf(-e2[i - 1], pm, (d[i] - x) * p);
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

// Eigenvalues of each walker's tridiagonal matrix by bisection, then
// S = -sum p ln p with p = lambda / sum(lambda) over p > 0. The matrix is
// scaled by a power of two into [-1, 1] and counted by the three-term
// recurrence; the brackets are first narrowed in FP32: from there a bracket
// [a, b] with count32(a) <= k < count32(b) holds lambda_k within
// [a - del, b + del] (del = 32 x 2^-24, above the FP32 count's error
// bound), and FP64 bisection takes it on to the tolerance. That saves about
// 10 of the 45 FP64 Sturm counts per eigenvalue, and the recurrence halves
// the FP64 instructions of a count. Matrices whose scale lies outside
// [2^-1000, 2^1000] take the pivot form unscaled, in FP64 only. Dynamic
// shared memory: d, e^2 and the eigenvalues (3 n doubles), T + 1 int
// counts, then d and e^2 as scaled floats (2 n).
__global__ void __launch_bounds__(kEntThreads) bisect_kernel(const double* d, const double* e,
                                                             int n, double* entropy,
                                                             double* eigs) {
  extern __shared__ double sb[];
  double* sd = sb;
  double* se2 = sb + n;
  double* lam = sb + 2 * n;
  __shared__ double red[kEntThreads / 32];
  const int t = threadIdx.x, T = blockDim.x;
  const double* dw = d + (size_t)blockIdx.x * n;
  const double* ew = e + (size_t)blockIdx.x * n;
  double lo = DBL_MAX, hi = -DBL_MAX, e2max = 0.0;
  for (int i = t; i < n; i += T) {
    sd[i] = dw[i];
    const double ei = i + 1 < n ? ew[i] : 0.0;
    se2[i] = ei * ei;
    e2max = fmax(e2max, ei * ei);
    // Gershgorin interval of row i
    const double r = fabs(ei) + (i > 0 ? fabs(ew[i - 1]) : 0.0);
    lo = fmin(lo, dw[i] - r);
    hi = fmax(hi, dw[i] + r);
  }
  lo = -block_max(-lo, red);
  hi = block_max(hi, red);
  e2max = block_max(e2max, red);
  const double pivmin = DBL_MIN * fmax(1.0, e2max);
  const double scale = fmax(fabs(lo), fabs(hi));
  const double tol = 2.0 * DBL_EPSILON * scale + 2.0 * pivmin;
  lo -= tol;
  hi += tol;
  int* cnt = reinterpret_cast<int*>(lam + n);  // T + 1 counts
  float* d32 = reinterpret_cast<float*>(cnt + T + 1);
  float* e32 = d32 + n;
  int ex = 0;
  frexp(scale, &ex);
  const bool use32 = scale > 0x1p-1000 && scale < 0x1p1000;
  const double sc = ldexp(1.0, -ex);  // scale x sc in [0.5, 1)
  if (use32) {  // the scaled matrix, in place of d and e^2, and as floats
    for (int i = t; i < n; i += T) {
      sd[i] *= sc;
      const double es = (i + 1 < n ? ew[i] : 0.0) * sc;
      se2[i] = es * es;
      d32[i] = (float)sd[i];
      e32[i] = (float)se2[i];
    }
  }
  __syncthreads();
  // multisection: one Sturm count per thread on an even grid gives every
  // eigenvalue a bracket T times narrower to start from (the ends widened
  // by twice the FP32 bound, so that the counts there are 0 and n)
  const float del32 = 32.0f * 0x1p-24f;
  const float lo32 = (float)(lo * sc) - 2.0f * del32, hi32 = (float)(hi * sc) + 2.0f * del32;
  const float h32 = (hi32 - lo32) / (float)T;
  const double hstep = (hi - lo) / T;
  auto grid32 = [&](int j) { return __fmaf_rn((float)j, h32, lo32); };
  auto grid64 = [&](int j) { return fma((double)j, hstep, lo); };
  if (use32) cnt[t + 1] = t + 1 < T ? sturm_count3f(d32, e32, n, grid32(t + 1)) : n;
  else cnt[t + 1] = t + 1 < T ? sturm_count(sd, se2, n, grid64(t + 1), pivmin) : n;
  if (t == 0) cnt[0] = 0;
  __syncthreads();
  for (int k = t; k < n; k += T) {
    // the k-th smallest eigenvalue: count(a) <= k < count(b)
    int g = 0;  // a grid cell with cnt[g] <= k < cnt[g + 1]
    int lo_i = 0, hi_i = T;
    while (hi_i - lo_i > 1) {
      const int mid = (lo_i + hi_i) >> 1;
      if (cnt[mid] <= k) lo_i = mid;
      else hi_i = mid;
    }
    g = lo_i;
    double a, b;
    if (use32) {
      float a32 = grid32(g), b32 = g + 1 < T ? grid32(g + 1) : hi32;
      for (int it = 0; it < 40 && b32 - a32 > del32; ++it) {
        const float mid = 0.5f * (a32 + b32);
        if (sturm_count3f(d32, e32, n, mid) <= k) a32 = mid;
        else b32 = mid;
      }
      // in scaled units from here
      a = (double)a32 - (double)del32;
      b = (double)b32 + (double)del32;
      const double tol_s = tol * sc;
      for (int it = 0; it < 200 && b - a > tol_s; ++it) {
        const double mid = 0.5 * (a + b);
        if (sturm_count3(sd, se2, n, mid) <= k) a = mid;
        else b = mid;
      }
      lam[k] = 0.5 * (a + b) / sc;  // dividing by a power of two: exact
    } else {
      a = grid64(g);
      b = g + 1 < T ? grid64(g + 1) : hi;
      for (int it = 0; it < 200 && b - a > tol; ++it) {
        const double mid = 0.5 * (a + b);
        if (sturm_count(sd, se2, n, mid, pivmin) <= k) a = mid;
        else b = mid;
      }
      lam[k] = 0.5 * (a + b);
    }
  }
  __syncthreads();
  double tot = 0.0;
  for (int k = t; k < n; k += T) tot += lam[k];
  tot = block_sum(tot, red);
  double s = 0.0;
  for (int k = t; k < n; k += T) {
    if (eigs) eigs[(size_t)blockIdx.x * n + k] = lam[k];
    const double p = tot > 0.0 ? lam[k] / tot : 0.0;
    if (p > 0.0) s -= p * log(p);
  }
  s = block_sum(s, red);
  if (t == 0) entropy[blockIdx.x] = s;
}

}  // namespace

cudaError_t launch_entropy_bisect(const double* d, const double* e, int64_t walkers, int n,
                                  double* entropy, double* eigs, cudaStream_t st) {
  if (walkers <= 0) return cudaSuccess;
  static bool attr[kAttrDevices] = {};
  const cudaError_t err = smem_limit(bisect_kernel, 96 * 1024, attr);
  if (err != cudaSuccess) return err;
  const size_t sm2 = 3 * (size_t)n * sizeof(double) + (kEntThreads + 1) * sizeof(int) +
                     2 * (size_t)n * sizeof(float);
  bisect_kernel<<<(unsigned)walkers, kEntThreads, sm2, st>>>(d, e, n, entropy, eigs);
  count_launch();
  return cudaGetLastError();
}

}  // namespace bg
