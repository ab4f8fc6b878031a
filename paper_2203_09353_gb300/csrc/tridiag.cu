// Householder reduction of each walker's Hermitian positive semidefinite
// n x n Gram matrix to a real tridiagonal matrix (d, e), for the entanglement
// entropy (Alg. 1, "Calculate Entropy"): the steps of LAPACK's zlatrd/zhetrd
// for the lower triangle, in 60-bit fixed point (fixed60.cuh) on the integer
// pipe, one kernel for the whole reduction.
//
// Why fixed point. The reduction is (16/3) n^3 FP64 flops, half of them in
// products A v that read the whole trailing matrix for each column. The FP64
// pipe (2 DFMA per clock per SM) bounded it; three 32 x 32 + 64 bit integer
// multiply-adds per real product are five times faster than a DFMA. Every
// quantity of the reduction is bounded by the matrix norm, so a single power of
// two B scales it: entries, W and y carry an absolute resolution of 2^-60 B ..
// 2^-58 B, below the FP64 reduction's own normwise backward error.
//
// Per panel of kNb columns (c = column, u = reflector vector, H = I - tau u u^H):
//   1. column c minus the panel's earlier rank-2 updates; d[c], and the exact
//      integer sum of squares below the diagonal;
//   2. norm N, e[c] = beta = -+N, u = (alpha - beta, x...): the column itself,
//      shifted to full scale, not divided by alpha - beta, so that only the
//      square root is on the critical path; tau = -u0 / (beta |u0|^2) is formed
//      while the product runs;
//   3. y = A u over the full (mirrored) trailing matrix, and W^H u, V^H u;
//   4. y -= V (W^H u) + W (V^H u), p = tau y, rho = u^H y;
//   5. w = p - (|tau|^2 rho / 2) u. (u, w) are column i of the panel's [V W].
// After a panel, A -= V W^H + W V^H on the lower triangle, mirrored.
//
// A walker runs on one CTA, or on a cluster of up to 8 when there are fewer
// walkers than SMs: rows are dealt to the CTAs in groups of 32 (group g to
// rank g mod CL), every CTA holds u, and partial sums and the u rows go
// through distributed shared memory, four cluster barriers a column. The
// last kTail columns (or a whole matrix up to that order) are reduced by one
// CTA with the matrix in shared memory.
//
// Bounds used by the formats (B = 2^60 units "uA" of the entries), with
// |u|^2 in [0.5, 4) after scaling (unit 2^-59) and lambda = ||A|| <= B (the
// limbs leave room for lambda <= kScaleRoom B):
//   |y| <= 2 B (2 uA), |W^H u| <= 4 B (4 uA), |V^H u| <= 4 (2^-58),
//   |tau| <= 4 (2^-58), rho <= 4 B (4 uA), |w| <= 1.25 lambda / |u| < 1.8 B (2 uA).
// Row and column norms of A are at most lambda, so sums of products stay in
// 64 bits by the Cauchy-Schwarz inequality; a cross sum is flushed every 16
// columns of A u (2^62.8 at most), 8 rows of V^H u, 2 columns of V and W.
#include <cuda_runtime.h>

#include <algorithm>
#include <cmath>
#include <mutex>

#include "bgemm_internal.h"
#include "fixed60.cuh"

namespace bg {
namespace {

using fx::Sum;

constexpr int kThreads = 512;
constexpr int kWarps = kThreads / 32;
constexpr int kNb = 16;       // panel width
constexpr int kTail = 96;     // columns reduced with the matrix in shared memory
// Orders up to kPacked of more walkers than SMs: several CTAs of fewer warps per
// SM. With the shared memory and threads of order 96 an SM held one walker at a
// time, whatever its order: 16000 matrices of order 2 took 0.90 ms where the FP64
// kernel before it took 0.45. Whole calls, with one CTA and with five per SM:
// 16000 of order 2 2290 -> 1340 us (FP64 kernel: 1730), of 8 4400 -> 2160 us, of 32
// 17.5 -> 10.1 ms, 153 of order 32 350 -> 256 us. Up to one walker per SM the 16
// warps are no slower and are kept.
constexpr int kPacked = 32, kPackedWarps = 4, kPackedCtas = 5;
constexpr int kStrip = 4;     // columns per update work item
constexpr int kMaxCl = 8;
constexpr float kScaleRoom = 1.4f;
constexpr size_t kSmemMax = 227 * 1024;
constexpr int kAttrDevices = 64;

struct TriArgs {
  double2* G;   // walkers x n x n, lower triangle; overwritten
  int4* P;      // walkers x 2 kNb x n: the panel's [V W] (clusters, or when it exceeds shared memory)
  double* d;
  double* e;
  int n;
  int own;      // rows a CTA owns at most (a multiple of 32)
};

struct ColumnScalars {  // a column's scalars, written by one thread
  int z;           // u = column 2^z
  int skip;
  long long u0r, u0i, nint;
  longlong2 sum;   // squares below the diagonal (uA^2; hi, lo)
};

struct Shared {
  longlong2 alpha[2];
  long long diag[2];                   // the column's diagonal entry
  long long trace;                     // of the rows not reduced yet (2^kTraceUnit uA)
  longlong2 fro;                       // their squared Frobenius norm (2^kFroUnit uA^2; hi, lo)
  int tail_z[2], unit[2];              // the tail's shift after a column, the column's unit
  longlong2 norm[2][kMaxCl * kWarps];  // sums of squares (hi, lo) of every warp
  longlong2 spart[2 * kNb][kMaxCl];    // V^H u and W^H u, a partial per CTA
  long long rho[kMaxCl * kWarps];
  longlong2 pnext;                     // p of row c + 1
  int4 rowV[kNb], rowW[kNb];           // row c + 1 of V and W
  int4 scoef[kWarps][2 * kNb];
  int4 tau;                            // limbs, unit 2^-58
  int2 t2;                             // |tau|^2 / 2, unit 2^-57
  ColumnScalars sc;
  double dred[kWarps];
  float2 fsum[kMaxCl * kWarps];        // (sum of squares, trace) of every warp
};

__device__ __forceinline__ uint32_t smem_addr(const void* p) {
  return static_cast<uint32_t>(__cvta_generic_to_shared(p));
}
__device__ __forceinline__ uint32_t mapa(uint32_t addr, int rank) {
  uint32_t r;
  asm("mapa.shared::cluster.u32 %0, %1, %2;" : "=r"(r) : "r"(addr), "r"(rank));
  return r;
}

// Writes v to the same shared-memory variable of every CTA of the cluster.
template <bool MULTI>
__device__ __forceinline__ void publish(int4* dst, const int4& v, int cl) {
  if constexpr (!MULTI) {
    *dst = v;
  } else {
    const uint32_t a = smem_addr(dst);
    for (int r = 0; r < cl; ++r)
      asm volatile("st.shared::cluster.v4.b32 [%0], {%1, %2, %3, %4};" ::"r"(mapa(a, r)), "r"(v.x),
                   "r"(v.y), "r"(v.z), "r"(v.w)
                   : "memory");
  }
}
template <bool MULTI>
__device__ __forceinline__ void publish(longlong2* dst, long long x, long long y, int cl) {
  if constexpr (!MULTI) {
    *dst = make_longlong2(x, y);
  } else {
    const uint32_t a = smem_addr(dst);
    for (int r = 0; r < cl; ++r)
      asm volatile("st.shared::cluster.v2.b64 [%0], {%1, %2};" ::"r"(mapa(a, r)), "l"(x), "l"(y)
                   : "memory");
  }
}
template <bool MULTI>
__device__ __forceinline__ void publish(long long* dst, long long x, int cl) {
  if constexpr (!MULTI) {
    *dst = x;
  } else {
    const uint32_t a = smem_addr(dst);
    for (int r = 0; r < cl; ++r)
      asm volatile("st.shared::cluster.b64 [%0], %1;" ::"r"(mapa(a, r)), "l"(x) : "memory");
  }
}

// Barrier over the walker's threads: the CTA, or the cluster (release / acquire).
template <bool MULTI>
__device__ __forceinline__ void walker_sync() {
  if constexpr (MULTI) {
    __syncwarp();
    asm volatile("barrier.cluster.arrive.release.aligned;" ::: "memory");
    asm volatile("barrier.cluster.wait.acquire.aligned;" ::: "memory");
  } else {
    __syncthreads();
  }
}

// How far the trailing matrix may be scaled up once it has become small: a
// low-entropy state leaves most of its weight in the first columns, and the rest
// then keeps its precision. At most kMaxShift bits in all, so that the rounding
// noise of the first columns stays far below full scale.
// Two bounds on its norm, both followed exactly from column to column, the
// smaller shift taken. The trace bounds the norm of a positive semidefinite
// matrix and resolves it to the last bit. A Gram matrix of few digit planes is not
// one: its truncation error, 2^-14 of the norm with 2 slices, can leave a
// trailing trace near zero or below under a matrix that is not (with the trace
// alone, 2 slices and K = 64, the entries for Schmidt weights 2^-i left the
// 60-bit range and its eigenvalues were off by 1e-5 of the largest). The
// Frobenius norm bounds any Hermitian matrix. A reflector does not change it, so
// each column takes d^2 + 2 |e|^2 from its square, which resolves the norm to
// about 2^-27: below the noise that kMaxShift allows for.
// Units: n full-scale entries fit the trace, n of their squares the other.
constexpr int kMaxShift = 24;
constexpr int kTraceUnit = 10;
constexpr int kFroUnit = 12;
__device__ __forceinline__ int rescale(long long trace, const fx::U128& fro, int shifted) {
  // trace 2^z < 2^60 uA, and the same for the square root of fro
  const int zt = trace > 0 ? __clzll(trace) - (64 - fx::kFull) - kTraceUnit : kMaxShift;
  const int lz = fro.hi ? __clzll((long long)fro.hi) : 64 + __clzll((long long)fro.lo);
  const int zf = lz > 0 ? (2 * fx::kFull - kFroUnit - 128 + lz) >> 1 : kMaxShift;  // (0: negative)
  return max(0, min(min(zt, zf), kMaxShift - shifted));
}

__device__ __forceinline__ fx::U128 unpack(const longlong2& v) {
  return {(unsigned long long)v.x, (unsigned long long)v.y};
}
__device__ __forceinline__ longlong2 pack(const fx::U128& v) {
  return make_longlong2((long long)v.hi, (long long)v.lo);
}

// |x|^2 of the lower triangle's entry x, twice off the diagonal, and what a column with
// diagonal d and the squares `below` under it takes from the trailing matrix.
__device__ __forceinline__ fx::U128 fro_entry(long long re, long long im, bool diagonal) {
  fx::U128 v;
  v.add_square(re);
  v.add_square(im);
  return v.shifted_right(diagonal ? kFroUnit : kFroUnit - 1);
}
__device__ __forceinline__ fx::U128 fro_column(long long d, const longlong2& below) {
  fx::U128 v;
  v.add_square(d);
  v.add((unsigned long long)below.x, (unsigned long long)below.y);
  v.add((unsigned long long)below.x, (unsigned long long)below.y);
  return v.shifted_right(kFroUnit);
}

// The reflector of a column (alpha, x...) with |x|^2 = sum: beta = -+N, N the
// column's norm, and u = (alpha - beta, x...) 2^z with nint = N 2^z in
// [2^58, 2^59).
__device__ __forceinline__ ColumnScalars reflector(const fx::U128& sum, long long alr,
                                                   long long ali) {
  fx::U128 all = sum;
  all.add_square(alr);
  all.add_square(ali);
  ColumnScalars sc{0, 0, 0, 0, 0, pack(all)};
  if (sum.hi == 0 && sum.lo == 0 && ali == 0) {
    sc.skip = 1;  // already reduced: H = I
    return sc;
  }
  sc.nint = fx::sqrt_scaled(all, &sc.z);
  const long long xr = fx::shift(alr, sc.z);
  sc.u0r = alr < 0 ? xr - sc.nint : xr + sc.nint;
  sc.u0i = fx::shift(ali, sc.z);
  return sc;
}

// The sub-diagonal entry beta of a column with first entry alr.
__device__ __forceinline__ double column_beta(const ColumnScalars& sc, long long alr, int eunit) {
  return sc.skip ? fx::to_double(alr, eunit)
                 : fx::to_double(alr < 0 ? sc.nint : -sc.nint, eunit - sc.z);
}

// tau = -u0 / (beta |u0|^2) in limbs of unit 2^-58, and |tau|^2 / 2 in limbs of
// unit 2^-57. With N = nint 2^-59 in [0.5, 1) and |u0|^2 in [0.25, 4), tau is
// +-u0 times 1 / (N |u0|^2).
__device__ __forceinline__ void reflector_tau(const ColumnScalars& sc, int4* tau, int2* t2) {
  fx::U128 M;
  M.add_square(sc.u0r);
  M.add_square(sc.u0i);
  const unsigned long long a = (unsigned long long)sc.nint << 4, b = M.hi << 7 | M.lo >> 57;
  const unsigned long long hi = __umul64hi(a, b), lo = a * b;
  const int lz = __clzll((long long)hi);  // 2 .. 6
  const unsigned long long R = fx::recip126(hi << lz | lo >> (64 - lz));
  const long long r = (long long)(R >> 1), sr = sc.u0r < 0 ? -r : r;  // beta's sign is -u0r's
  // u0 R 2^(lz - 67)
  const long long tr = fx::shift(__mul64hi(sc.u0r << 2, sr), lz - 4);
  const long long ti = fx::shift(__mul64hi(sc.u0i << 2, sr), lz - 4);
  *tau = fx::pack(tr, ti);
  fx::U128 T;
  T.add_square(tr);
  T.add_square(ti);
  const fx::Limb l = fx::split((long long)(T.hi << 4 | T.lo >> 60));
  *t2 = make_int2(l.h, l.l);
}

// u^H y of one row (real part), unit 4 uA.
__device__ __forceinline__ long long real_dot(const int4& u, const int4& y) {
  long long h = 0, x = 0;
  fx::mac(h, u.x, y.x);
  fx::mac(h, u.z, y.z);
  fx::mac(x, u.x, y.y);
  fx::mac(x, u.y, y.x);
  fx::mac(x, u.z, y.w);
  fx::mac(x, u.w, y.z);
  return fx::val(h, x);
}

// c = |tau|^2 rho / 2, unit 4 uA.
__device__ __forceinline__ fx::Limb w_coef(const int2& t2, long long rho) {
  const fx::Limb rq = fx::split(rho);
  long long h = 0, x = 0;
  fx::mac(h, t2.x, rq.h);
  fx::mac(x, t2.x, rq.l);
  fx::mac(x, t2.y, rq.h);
  return fx::split(fx::val<3>(h, x));
}

// w = p - c u for one row: p in uA, w in 2 uA.
__device__ __forceinline__ int4 make_w(long long pr, long long pi, const fx::Limb& c,
                                       const int4& u) {
  long long rh = 0, rx = 0, ih = 0, ix = 0;
  fx::mac(rh, c.h, u.x);
  fx::mac(rx, c.h, u.y);
  fx::mac(rx, c.l, u.x);
  fx::mac(ih, c.h, u.z);
  fx::mac(ix, c.h, u.w);
  fx::mac(ix, c.l, u.z);
  return fx::pack(fx::rne(pr - fx::val<3>(rh, rx), 1), fx::rne(pi - fx::val<3>(ih, ix), 1));
}

// One walker's (or its tail's) reduction state.
struct Red {
  int4* A;       // full matrix (both triangles), column-major
  int ld, n;     // leading dimension, order
  int4* P;       // [V W] in global memory, column q at P + q n (or null)
  int4* vw;      // [V W] of the own rows in shared memory, column q at vw + q own
  int own;
  int4* us;      // u
  longlong2* part;  // partial products; also x and p of the own rows
  int4* stage;   // per-warp copies of [V W] rows for the update
  double* d;
  double* e;
  int eunit;     // uA = 2^eunit
  int shifted;   // bits the matrix has been scaled up since the start
  int rank, cl;
  Shared* S;
};

// Reduces columns 0 .. cend - 1 (cend <= n - 1). MULTI: a cluster shares the
// walker. VWS: the panel's own rows of V and W are in shared memory.
template <bool MULTI, bool VWS>
__device__ __forceinline__ void reduce(Red& R, int cend) {
  const int t = threadIdx.x, warp = t >> 5, lane = t & 31;
  const int n = R.n, ld = R.ld, own = R.own;
  const int cl = MULTI ? R.cl : 1, rank = MULTI ? R.rank : 0;
  const int ngroups = (n + 31) >> 5;
  const int kmax = (ngroups - rank + cl - 1) / cl;  // own groups
  Shared& S = *R.S;
  longlong2* xs = R.part;  // x of the own rows (between steps 1 and 2)
  int eunit = R.eunit;
  auto vptr = [&](int q, int lr, int r) -> int4* {
    return VWS ? R.vw + q * own + lr : R.P + (size_t)q * n + r;
  };
  auto vload = [&](int q, int lr, int r) -> int4 {
    return VWS ? *vptr(q, lr, r) : __ldcg(vptr(q, lr, r));
  };
  for (int p0 = 0; p0 < cend; p0 += kNb) {
    const int nbp = min(kNb, cend - p0);
    for (int i = 0; i < nbp; ++i) {
      const int c = p0 + i, par = c & 1;
      // ---- 1. column c with the panel's earlier updates; sums of squares
      fx::U128 sq;
      for (int k = warp; k < kmax; k += kWarps) {
        const int r = 32 * (rank + cl * k) + lane, lr = 32 * k + lane;
        if (32 * (rank + cl * k) + 31 < c) continue;
        long long xr = 0, xi = 0;
        if (r >= c && r < n) {
          const int4 a = __ldcg(R.A + r + (size_t)c * ld);
          Sum s;
          for (int q = 0; q < i; ++q) {
            s.add_conj(vload(q, lr, r), S.rowW[q]);
            s.add_conj(vload(kNb + q, lr, r), S.rowV[q]);
            if (q & 1) s.flush();
          }
          xr = fx::join(a.x, a.y) - s.re<2>();
          xi = fx::join(a.z, a.w) - s.im<2>();
          if (r == c) publish<MULTI>(&S.diag[par], xr, cl);
          if (r == c + 1) publish<MULTI>(&S.alpha[par], xr, xi, cl);
          if (r >= c + 2) {
            sq.add_square(xr);
            sq.add_square(xi);
          }
        }
        xs[lr] = make_longlong2(xr, xi);
      }
      sq = fx::warp_sum(sq);
      if (lane == 0)
        publish<MULTI>(&S.norm[par][rank * kWarps + warp], (long long)sq.hi, (long long)sq.lo, cl);
      walker_sync<MULTI>();
      // ---- 2. norm, beta, u0: one warp of every CTA, from the same numbers
      if (warp == 0) {
        fx::U128 sum;
        for (int x = lane; x < cl * kWarps; x += 32) {
          const longlong2 v = S.norm[par][x];
          sum.add((unsigned long long)v.x, (unsigned long long)v.y);
        }
        sum = fx::warp_sum(sum);
        if (lane == 0) {
          const longlong2 al = S.alpha[par];
          S.sc = reflector(sum, al.x, al.y);
          S.trace -= S.diag[par] >> kTraceUnit;
        }
      }
      __syncthreads();
      const ColumnScalars sc = S.sc;
      // the column's results, beside step 4 (by a warp with few rows there or none)
      auto finish_column = [&]() {
        if (t != kThreads - 32) return;
        fx::U128 fro = unpack(S.fro);
        fro.subtract(fro_column(S.diag[par], S.sc.sum));
        S.fro = pack(fro);
        if (rank == 0) {
          R.d[c] = fx::to_double(S.diag[par], eunit);
          R.e[c] = column_beta(S.sc, S.alpha[par].x, eunit);
        }
      };
      // u to every CTA; V's column i
      for (int k = warp; k < kmax; k += kWarps) {
        const int r = 32 * (rank + cl * k) + lane, lr = 32 * k + lane;
        if (32 * (rank + cl * k) + 31 <= c) continue;
        if (r > c && r < n) {
          int4 u = make_int4(0, 0, 0, 0);
          if (!sc.skip) {
            const longlong2 x = xs[lr];
            u = r == c + 1 ? fx::pack(sc.u0r, sc.u0i)
                           : fx::pack(fx::shift(x.x, sc.z), fx::shift(x.y, sc.z));
            publish<MULTI>(R.us + r, u, cl);
          }
          if constexpr (VWS) *vptr(i, lr, r) = u;
          if (MULTI || !VWS) R.P[(size_t)i * n + r] = u;
          if (sc.skip) {
            if constexpr (VWS) *vptr(kNb + i, lr, r) = u;
            if (MULTI || !VWS) R.P[(size_t)(kNb + i) * n + r] = u;
          }
        }
      }
      const int gnext = (c + 1) >> 5;  // the group holding row c + 1
      const bool owns_next = gnext % cl == rank && (gnext / cl) % kWarps == warp;
      // row c + 1 of V and W for the next column's step 1 (columns below i;
      // its owner publishes them, column i follows from u and p)
      auto publish_row = [&]() {
        if (!owns_next) return;
        const int r = c + 1, lr = 32 * (gnext / cl) + (r & 31);
        const int q = lane & 15;
        if (q < i) {
          const int4 v = vload((lane & 16) + q, lr, r);
          publish<MULTI>((lane & 16) ? &S.rowW[q] : &S.rowV[q], v, cl);
        }
      };
      if (sc.skip) {
        publish_row();
        finish_column();
        if (t == 0) S.rowV[i] = S.rowW[i] = make_int4(0, 0, 0, 0);
        walker_sync<MULTI>();
        continue;
      }
      walker_sync<MULTI>();
      // ---- 3. tau, by one thread beside the products
      if (t == kThreads - 32) {
        reflector_tau(sc, &S.tau, &S.t2);
      }
      // V^H u and W^H u over the own rows, a warp per column
      for (int it = warp; it < 2 * i; it += kWarps) {
        const int q = it >> 1, vq = (it & 1) ? kNb + q : q;
        Sum s;
        for (int k = max(0, (c + 1) / 32 / cl - 1); k < kmax; ++k) {
          const int r = 32 * (rank + cl * k) + lane, lr = 32 * k + lane;
          if (r > c && r < n) s.add_conj(R.us[r], vload(vq, lr, r));
          if ((k & 7) == 7) s.flush();
        }
        const long long sr = fx::warp_sum(s.re()), si = fx::warp_sum(s.im());
        if (lane == 0) publish<MULTI>(&S.spart[vq][rank], sr, si, cl);
      }
      // y = A u: items of one own group of rows x a run of columns
      int kfirst = (c + 1) / 32;  // first own group with a row > c
      kfirst = kfirst > rank ? (kfirst - rank + cl - 1) / cl : 0;
      const int cnt = kmax - kfirst;
      const int nch = cnt > 0 ? max(1, kWarps / cnt) : 1;
      for (int it = warp; it < cnt * nch; it += kWarps) {
        const int gi = it % cnt, ch = it / cnt;
        const int r = 32 * (rank + cl * (kfirst + gi)) + lane;
        const int m = n - c - 1;
        int j = c + 1 + m * ch / nch;
        const int j1 = c + 1 + m * (ch + 1) / nch;
        const int4* a = R.A + min(r, n - 1);
        Sum s;
        // batches of U columns, the next one's loads in flight (two register
        // sets in turn, so that nothing is copied)
        constexpr int U = 8;
        int4 b0[U], b1[U];
        auto fetch = [&](int4(&b)[U], int jj) {
          if (jj + U <= j1) {
#pragma unroll
            for (int x = 0; x < U; ++x) b[x] = __ldcg(a + (size_t)(jj + x) * ld);
          }
        };
        auto use = [&](const int4(&b)[U]) {
#pragma unroll
          for (int x = 0; x < U; ++x) s.add(b[x], R.us[j + x]);
          s.flush();
          j += U;
        };
        fetch(b0, j);
        while (j + U <= j1) {
          fetch(b1, j + U);
          use(b0);
          if (j + U > j1) break;
          fetch(b0, j + U);
          use(b1);
        }
        for (; j < j1; ++j) s.add(__ldcg(a + (size_t)j * ld), R.us[j]);
        R.part[it * 32 + lane] = make_longlong2(s.re(), s.im());  // unit 2 uA
      }
      walker_sync<MULTI>();
      // ---- 4. corrections, p = tau y, rho
      long long rho = 0;
      {
        // lane x: coefficient column x (V^H u below 16, W^H u above), in limbs
        long long cr = 0, ci = 0;
        if ((lane & 15) < i) {
          for (int x = 0; x < cl; ++x) {
            const longlong2 v = S.spart[lane][x];
            cr += v.x;
            ci += v.y;
          }
        }
        S.scoef[warp][lane] = fx::pack(cr, ci);
        __syncwarp();
      }
      const int4 tau = S.tau;
      // (the own groups from kfirst on, each by the warp that owns it in steps 1 and 5)
      for (int k = warp; k < kmax; k += kWarps) {
        if (k < kfirst) continue;
        const int r = 32 * (rank + cl * k) + lane, lr = 32 * k + lane, gi = k - kfirst;
        long long yr = 0, yi = 0;
        for (int ch = 0; ch < nch; ++ch) {
          const longlong2 v = R.part[(ch * cnt + gi) * 32 + lane];
          yr += v.x;
          yi += v.y;
        }
        long long pr = 0, pi = 0;
        if (r > c && r < n) {
          Sum s;
          for (int q = 0; q < i; ++q) {
            s.add(vload(q, lr, r), S.scoef[warp][kNb + q]);       // V (W^H u)
            s.add(vload(kNb + q, lr, r), S.scoef[warp][q]);       // W (V^H u)
            if (q & 1) s.flush();
          }
          const int4 yq = fx::pack(yr - s.re<2>(), yi - s.im<2>());
          Sum ps;
          ps.add(tau, yq);
          pr = ps.re<3>();  // unit uA
          pi = ps.im<3>();
          rho += real_dot(R.us[r], yq);
          if (r == c + 1) publish<MULTI>(&S.pnext, pr, pi, cl);
        }
        R.part[gi * 32 + lane] = make_longlong2(pr, pi);
      }
      rho = fx::warp_sum(rho);
      if (lane == 0) publish<MULTI>(&S.rho[rank * kWarps + warp], rho, cl);
      publish_row();
      finish_column();
      walker_sync<MULTI>();
      // ---- 5. w = p - (|tau|^2 rho / 2) u
      rho = 0;
      for (int x = lane; x < cl * kWarps; x += 32) rho += S.rho[x];
      rho = fx::warp_sum(rho);
      const fx::Limb cc = w_coef(S.t2, rho);
      for (int k = warp; k < kmax; k += kWarps) {
        if (k < kfirst) continue;
        const int r = 32 * (rank + cl * k) + lane, lr = 32 * k + lane;
        if (r > c && r < n) {
          const longlong2 p = R.part[(k - kfirst) * 32 + lane];
          const int4 w = make_w(p.x, p.y, cc, R.us[r]);
          if constexpr (VWS) *vptr(kNb + i, lr, r) = w;
          if (MULTI || !VWS) R.P[(size_t)(kNb + i) * n + r] = w;
        }
      }
      if (t == kThreads - 1) {
        S.rowV[i] = R.us[c + 1];
        S.rowW[i] = make_w(S.pnext.x, S.pnext.y, cc, R.us[c + 1]);
      }
      __syncthreads();
    }
    walker_sync<MULTI>();
    // ---- trailing update on rows and columns q0 ..: a warp per 32 rows x
    // kStrip columns of the lower triangle, written to both triangles
    const int q0 = p0 + nbp;
    const int z = rescale(S.trace, unpack(S.fro), R.shifted);
    R.shifted += z;
    eunit -= z;
    {
      const int nw = cl * kWarps, gw = rank * kWarps + warp;
      const int c00 = q0 / kStrip * kStrip;
      int base = 0;
      for (int I = q0 >> 5; I < ngroups; ++I) {
        const int cntI = (min(32 * I + 32, n) - c00 + kStrip - 1) / kStrip;
        int s = (gw - base) % nw;
        if (s < 0) s += nw;
        base += cntI;
        for (; s < cntI; s += nw) {
          const int cs = c00 + s * kStrip;
          const int r = 32 * I + lane, rc = min(r, n - 1);
          const int4* st = nullptr;
          if constexpr (MULTI || !VWS) {
            int4* sg = R.stage + warp * (2 * kNb * kStrip);
            __syncwarp();
#pragma unroll
            for (int x = 0; x < kStrip; ++x) {
              const int q = x * (32 / kStrip) + lane / kStrip, cc = cs + lane % kStrip;
              sg[q * kStrip + lane % kStrip] = (q & 15) < nbp && cc < n
                                                   ? __ldcg(R.P + (size_t)q * n + cc)
                                                   : make_int4(0, 0, 0, 0);
            }
            __syncwarp();
            st = sg;
          }
          int4 a[kStrip];
#pragma unroll
          for (int x = 0; x < kStrip; ++x)
            a[x] = __ldcg(R.A + rc + (size_t)min(cs + x, n - 1) * ld);
          Sum sum[kStrip];
#pragma unroll 2
          for (int q = 0; q < nbp; ++q) {
            int4 v, w;
            if constexpr (MULTI || !VWS) {
              v = __ldcg(R.P + (size_t)q * n + rc);
              w = __ldcg(R.P + (size_t)(kNb + q) * n + rc);
            } else {
              v = R.vw[q * own + rc];
              w = R.vw[(kNb + q) * own + rc];
            }
#pragma unroll
            for (int x = 0; x < kStrip; ++x) {
              int4 cv, cw;
              if constexpr (MULTI || !VWS) {
                cv = st[q * kStrip + x];
                cw = st[(kNb + q) * kStrip + x];
              } else {
                cv = R.vw[q * own + min(cs + x, n - 1)];
                cw = R.vw[(kNb + q) * own + min(cs + x, n - 1)];
              }
              sum[x].add_conj(v, cw);
              sum[x].add_conj(w, cv);
            }
            if (q & 1) {
#pragma unroll
              for (int x = 0; x < kStrip; ++x) sum[x].flush();
            }
          }
#pragma unroll
          for (int x = 0; x < kStrip; ++x) {
            const int cc = cs + x;
            if (r >= n || cc > r || cc < q0) continue;
            const long long re = (fx::join(a[x].x, a[x].y) - sum[x].re<2>()) << z;
            const long long im =
                r == cc ? 0 : (fx::join(a[x].z, a[x].w) - sum[x].im<2>()) << z;
            const int4 v = fx::pack(re, im);
            R.A[r + (size_t)cc * ld] = v;
            if (r != cc) R.A[cc + (size_t)r * ld] = fx::pack(re, -im);
          }
        }
      }
    }
    walker_sync<MULTI>();
    if (t == 0) {
      S.trace <<= z;
      S.fro = pack(unpack(S.fro).shifted_left(2 * z));
    }
  }
  R.eunit = eunit;
}

// The reduction of a matrix of order n <= 32 ROWS held in shared memory (both
// triangles, leading dimension 32 ROWS + 1) by W warps, column by column: at
// this order the columns are bound by latency, not by the products, so warp 0
// takes the chain from one column to the next alone (its ROWS rows per lane
// need no barrier) and three barriers part it from what the other warps do: the
// rank-2 update of the previous column beside the norm, square root and u of
// this one, then the product A u beside tau, then w. (As panels of 16 columns
// in the general routine, the last 96 columns took 16 k clocks each; here
// 8 k.) us: u of this column and the last, ws: w.
template <int ROWS, int W>
__device__ __forceinline__ void reduce_tail(int4* A, int n, int4* us, int4* ws, longlong2* part,
                                            double* d, double* e, int eunit, int shifted,
                                            Shared& S) {
  const int t = threadIdx.x, warp = t >> 5, lane = t & 31;
  constexpr int kRows = ROWS;  // rows per lane of warp 0
  constexpr int N = 32 * ROWS, ld = N + 1;
  long long trace = 0;  // (these two in the thread that chooses the next shift)
  fx::U128 fro;
  for (int c = 0; c < n; ++c) {
    // (the previous column's update is scaled up by 2^z)
    const int z = c > 0 ? S.tail_z[(c - 1) & 1] : 0;
    int4* u = us + (c & 1) * N;
    const int4* up = us + ((c & 1) ^ 1) * N;
    if (warp == 0) {
      // ---- column c, with the previous column's update
      fx::U128 sq;
      long long xr[kRows], xi[kRows];
      int4 cu = make_int4(0, 0, 0, 0), cw = cu;
      if (c > 0) {
        cu = up[c];
        cw = ws[c];
      }
#pragma unroll
      for (int k = 0; k < kRows; ++k) {
        const int r = lane + 32 * k;
        xr[k] = xi[k] = 0;
        if (r >= c && r < n) {
          const int4 a = A[r + c * ld];
          xr[k] = fx::join(a.x, a.y);
          xi[k] = fx::join(a.z, a.w);
          if (c > 0) {
            Sum s;
            s.add_conj(up[r], cw);
            s.add_conj(ws[r], cu);
            xr[k] = (xr[k] - s.re<2>()) << z;
            xi[k] = (xi[k] - s.im<2>()) << z;
          }
          if (r >= c + 2) {
            sq.add_square(xr[k]);
            sq.add_square(xi[k]);
          }
        }
      }
      eunit -= z;
      if (c < n - 1) {
        sq = fx::warp_sum(sq);
        const int kd = c >> 5, ka = (c + 1) >> 5;
        long long dr = xr[0], ar = xr[0], ai = xi[0];
#pragma unroll
        for (int k = 1; k < kRows; ++k) {
          if (kd == k) dr = xr[k];
          if (ka == k) {
            ar = xr[k];
            ai = xi[k];
          }
        }
        dr = __shfl_sync(0xFFFFFFFFu, dr, c & 31);
        ar = __shfl_sync(0xFFFFFFFFu, ar, (c + 1) & 31);
        ai = __shfl_sync(0xFFFFFFFFu, ai, (c + 1) & 31);
        const ColumnScalars sc = reflector(sq, ar, ai);
#pragma unroll
        for (int k = 0; k < kRows; ++k) {
          const int r = lane + 32 * k;
          if (r > c && r < n) {
            int4 v = make_int4(0, 0, 0, 0);
            if (!sc.skip)
              v = r == c + 1 ? fx::pack(sc.u0r, sc.u0i)
                             : fx::pack(fx::shift(xr[k], sc.z), fx::shift(xi[k], sc.z));
            u[r] = v;
          }
        }
        if (lane == 0) {
          S.sc = sc;
          S.alpha[c & 1] = make_longlong2(ar, dr);
          S.unit[c & 1] = eunit;
        }
      } else {
        long long dr = xr[0];
#pragma unroll
        for (int k = 1; k < kRows; ++k)
          if ((c >> 5) == k) dr = xr[k];
        if (lane == (c & 31)) {
          d[c] = fx::to_double(dr, eunit);
          e[c] = 0.0;
        }
      }
    } else if (c > 0) {
      // ---- A -= u w^H + w u^H of the previous column on rows and columns
      // above c: a warp per pair of columns j, m - 1 - j (m + 1 elements
      // below and on the diagonal together)
      const int b0 = c + 1, m = n - b0;
      for (int j = warp - 1; 2 * j < m; j += W - 1) {
        const int first = m - j, len = 2 * j == m - 1 ? first : m + 1;
        for (int x = lane; x < len; x += 32) {
          const int cc = b0 + (x < first ? j : m - 1 - j);
          const int r = x < first ? cc + x : cc + (x - first);
          const int4 a = A[r + cc * ld];
          Sum s;
          s.add_conj(up[r], ws[cc]);
          s.add_conj(ws[r], up[cc]);
          const long long re = (fx::join(a.x, a.y) - s.re<2>()) << z;
          const long long im = r == cc ? 0 : (fx::join(a.z, a.w) - s.im<2>()) << z;
          A[r + cc * ld] = fx::pack(re, im);
          if (r != cc) A[cc + r * ld] = fx::pack(re, -im);
        }
      }
    }
    if (c == n - 1) break;
    __syncthreads();
    const ColumnScalars sc = S.sc;
    const int m = n - c - 1;
    const int g0 = (c + 1) >> 5, cnt = ((n + 31) >> 5) - g0;  // groups of 32 rows with one > c
    const int nch = (W - 1) / cnt;
    // the column's results and the next shift, by a warp that has no part in w
    auto finish_column = [&]() {
      if (t != 32 * W - 64) return;
      const long long dr = S.alpha[c & 1].y;
      trace = (c > 0 ? trace << z : S.trace) - (dr >> kTraceUnit);
      fro = c > 0 ? fro.shifted_left(2 * z) : unpack(S.fro);
      fro.subtract(fro_column(dr, sc.sum));
      const int zn = rescale(trace, fro, shifted);
      shifted += zn;
      S.tail_z[c & 1] = zn;
      d[c] = fx::to_double(dr, S.unit[c & 1]);
      e[c] = column_beta(sc, S.alpha[c & 1].x, S.unit[c & 1]);
    };
    if (sc.skip) {  // H = I: w = 0 like u
      if (warp == 0)
        for (int r = c + 1 + lane; r < n; r += 32) ws[r] = make_int4(0, 0, 0, 0);
      finish_column();
      __syncthreads();
      continue;
    }
    if (warp == W - 1) {
      if (lane == 0) reflector_tau(sc, &S.tau, &S.t2);
    } else if (warp < cnt * nch) {
      // ---- y = A u: one group of rows x a run of columns
      const int g = g0 + warp % cnt, ch = warp / cnt;
      const int r = min(32 * g + lane, n - 1);
      int j = c + 1 + m * ch / nch;
      const int j1 = c + 1 + m * (ch + 1) / nch;
      Sum s;
      for (; j < j1; ++j) {
        s.add(A[r + j * ld], u[j]);
        if ((j & 15) == 15) s.flush();
      }
      part[warp * 32 + lane] = make_longlong2(s.re(), s.im());
    }
    __syncthreads();
    finish_column();
    if (warp == 0) {
      // ---- p = tau y, rho, w
      const int4 tau = S.tau;
      long long pr[kRows], pi[kRows], rho = 0;
#pragma unroll
      for (int k = 0; k < kRows; ++k) {
        const int r = lane + 32 * k;
        pr[k] = pi[k] = 0;
        if (r > c && r < n) {
          long long yr = 0, yi = 0;
#pragma unroll 5
          for (int ch = 0; ch < nch; ++ch) {
            const longlong2 v = part[(ch * cnt + k - g0) * 32 + lane];
            yr += v.x;
            yi += v.y;
          }
          const int4 yq = fx::pack(yr, yi);
          Sum ps;
          ps.add(tau, yq);
          pr[k] = ps.re<3>();
          pi[k] = ps.im<3>();
          rho += real_dot(u[r], yq);
        }
      }
      const fx::Limb cc = w_coef(S.t2, fx::warp_sum(rho));
#pragma unroll
      for (int k = 0; k < kRows; ++k) {
        const int r = lane + 32 * k;
        if (r > c && r < n) ws[r] = make_w(pr[k], pi[k], cc, u[r]);
      }
    }
    __syncthreads();
  }
}

// |x| 2^-e as a float rounded down by at most 2^-20 of itself (inf for a
// non-finite x, 0 below 2^-126).
__device__ __forceinline__ float scaled_abs(double x, int e) {
  const uint32_t h = (uint32_t)__double2hiint(x) & 0x7FFFFFFFu;
  const int eb = (int)(h >> 20);
  const int ef = eb - 1023 - e + 127;
  if (eb == 0x7FF || ef >= 255) return __int_as_float(0x7F800000);
  if (ef <= 0 || eb == 0) return 0.0f;
  return __int_as_float((ef << 23) | (int)((h & 0xFFFFFu) << 3));
}

// The whole reduction of walker blockIdx.x / cl by W warps. ROWS: n <= 32 ROWS,
// the matrix goes straight to shared memory (0: any order above kTail). Bound by the multiply pipe (77%
// of a busy SM's cycles at n = 256, 1.7 times what the products need) and, in the
// last columns and for few walkers, by the latency of a column. Measured
// against panels with an FP64 product, split GEMMs between them and an FP64
// kernel for the last 64 columns: 128 matrices of order 256 12.6 -> 5.3 ms, 16
// of 1024 382 -> 52.8 ms (6 CTAs each), 4 of 64 0.89 -> 0.25 ms; against the
// FP64 kernel alone 32 of 128 4.5 -> 1.0 ms.
template <bool MULTI, bool VWS, int ROWS, int W>
__global__ void __launch_bounds__(32 * W, W < kWarps ? kPackedCtas : 1) tri_reduce_kernel(const TriArgs g) {
  static_assert(W == kWarps || (ROWS > 0 && !MULTI), "reduce() takes kWarps warps");
  constexpr bool SMALL = ROWS > 0;
  extern __shared__ __align__(16) int4 sm4[];
  __shared__ Shared S;
  const int t = threadIdx.x, warp = t >> 5, lane = t & 31;
  int cl = 1, rank = 0;
  if constexpr (MULTI) {
    asm("mov.u32 %0, %%cluster_nctarank;" : "=r"(cl));
    asm("mov.u32 %0, %%cluster_ctarank;" : "=r"(rank));
  }
  const int n = g.n;
  const size_t w = blockIdx.x / cl;
  double2* G = g.G + w * n * n;
  double* dw = g.d + w * n;
  double* ew = g.e + w * n;
  // ---- the scale: with t the mean eigenvalue (trace / n), the largest one is
  // at most t + sqrt((n - 1) (||G||_F^2 / n - t^2))
  double dm = 0.0;
  for (int i = t; i < n; i += 32 * W) dm = fmax(dm, fabs(__ldcg(&G[i + (size_t)i * n].x)));
  for (int o = 16; o > 0; o >>= 1) dm = fmax(dm, __shfl_xor_sync(0xFFFFFFFFu, dm, o));
  if (lane == 0) S.dred[warp] = dm;
  walker_sync<MULTI>();  // also: every CTA of the cluster runs before its memory is written
  dm = 0.0;
  for (int i = 0; i < W; ++i) dm = fmax(dm, S.dred[i]);
  const int e0 = dm > 0.0 ? (int)((__double2hiint(dm) >> 20) & 0x7FF) - 1022 : 0;
  const int ngroups = (n + 31) >> 5;
  float f2 = 0.0f, tr = 0.0f;
  for (int idx = rank * W + warp; idx < n; idx += cl * W) {
    // a warp per column, its lower part
    for (int r = idx + lane; r < n; r += 32) {
      const double2 z = __ldcg(&G[r + (size_t)idx * n]);
      const float a = scaled_abs(z.x, e0), b = r == idx ? 0.0f : scaled_abs(z.y, e0);
      const float q = fmaf(a, a, b * b);
      f2 += r == idx ? q : 2.0f * q;
      tr += r == idx ? a : 0.0f;
    }
  }
  for (int o = 16; o > 0; o >>= 1) {
    f2 += __shfl_xor_sync(0xFFFFFFFFu, f2, o);
    tr += __shfl_xor_sync(0xFFFFFFFFu, tr, o);
  }
  if (lane == 0) {
    if constexpr (MULTI) {
      for (int x = 0; x < cl; ++x)
        asm volatile("st.shared::cluster.v2.f32 [%0], {%1, %2};" ::"r"(
                         mapa(smem_addr(&S.fsum[rank * W + warp]), x)),
                     "f"(f2), "f"(tr)
                     : "memory");
    } else {
      S.fsum[warp] = make_float2(f2, tr);
    }
  }
  walker_sync<MULTI>();
  float F2 = 0.0f, mean = 0.0f;
  for (int x = 0; x < cl * W; ++x) {
    F2 += S.fsum[x].x;
    mean += S.fsum[x].y;
  }
  mean /= (float)n;
  if (!(F2 < __int_as_float(0x7F800000))) {  // a NaN or infinity in G
    const double nan = __longlong_as_double(0x7FF8000000000000ll);
    if (rank == 0)
      for (int i = t; i < n; i += 32 * W) {
        dw[i] = nan;
        ew[i] = i + 1 < n ? nan : 0.0;
      }
    return;
  }
  // the bound, with 4e-5 of the sum of squares for the float sums' rounding
  const float var = fmaxf(F2 / (float)n - mean * mean, 0.0f) + 4e-5f * F2 / (float)n;
  const float lam = (mean + sqrtf((float)(n - 1) * var)) * 1.0001f;
  // B = 2^eB >= bound / kScaleRoom; a zero matrix takes any scale
  const float B = lam * (1.0f / kScaleRoom);
  const int eB = e0 + (B > 0.0f ? (int)((__float_as_uint(B) >> 23) & 0xFF) - 126 : 0);
  const int eunit = eB - fx::kFull;  // uA = 2^eunit
  Red R;
  R.S = &S;
  R.eunit = eunit;
  R.rank = rank;
  R.cl = cl;
  R.d = dw;
  R.e = ew;
  int4* sm = sm4;
  constexpr int kOrder = SMALL ? 32 * ROWS : kTail, kLd = kOrder + 1;
  const int nt = SMALL ? n : kTail;
  // ---- fixed point, both triangles (in place, or into shared memory)
  int4* tail_us = sm;                                        // 2 kOrder
  int4* tail_ws = tail_us + 2 * kOrder;                      // kOrder
  longlong2* tail_part = reinterpret_cast<longlong2*>(tail_ws + kOrder);
  int4* tail_A = reinterpret_cast<int4*>(tail_part + W * 32);  // kOrder x kLd
  fx::U128 fro;
  {
    int4* A = SMALL ? tail_A : reinterpret_cast<int4*>(G);
    const int ld = SMALL ? kLd : n;
    const int nw = cl * W, gw = rank * W + warp;
    int base = 0;
    for (int I = 0; I < ngroups; ++I) {
      const int cntI = (min(32 * I + 32, n) + kStrip - 1) / kStrip;
      int s = (gw - base) % nw;
      if (s < 0) s += nw;
      base += cntI;
      for (; s < cntI; s += nw) {
        const int r = 32 * I + lane;
        double2 z[kStrip];
#pragma unroll
        for (int x = 0; x < kStrip; ++x) {
          const int cc = s * kStrip + x;
          z[x] = r < n && cc <= r ? __ldcg(&G[r + (size_t)cc * n]) : make_double2(0.0, 0.0);
        }
#pragma unroll
        for (int x = 0; x < kStrip; ++x) {
          const int cc = s * kStrip + x;
          if (r >= n || cc > r) continue;
          const long long re = fx::from_double(z[x].x, -eunit);
          const long long im = r == cc ? 0 : fx::from_double(z[x].y, -eunit);
          const fx::U128 sq = fro_entry(re, im, r == cc);
          fro.add(sq.hi, sq.lo);
          A[r + (size_t)cc * ld] = fx::pack(re, im);
          if (r != cc) A[cc + (size_t)r * ld] = fx::pack(re, -im);
        }
      }
    }
  }
  fro = fx::warp_sum(fro);
  if (lane == 0)  // (norm[1]: column 0 uses norm[0])
    publish<MULTI>(&S.norm[1][rank * W + warp], (long long)fro.hi, (long long)fro.lo, cl);
  walker_sync<MULTI>();
  if (warp == 0) {
    fro = fx::U128();
    for (int x = lane; x < cl * W; x += 32) {
      const longlong2 v = S.norm[1][x];
      fro.add((unsigned long long)v.x, (unsigned long long)v.y);
    }
    fro = fx::warp_sum(fro);
    const int4* A = SMALL ? tail_A : reinterpret_cast<int4*>(G);
    const int ld = SMALL ? kLd : n;
    long long tr0 = 0;
    for (int i = lane; i < n; i += 32) {
      const int4 v = SMALL ? A[i + i * ld] : __ldcg(A + i + (size_t)i * ld);
      tr0 += fx::join(v.x, v.y) >> kTraceUnit;
    }
    tr0 = fx::warp_sum(tr0);
    if (lane == 0) {
      S.trace = tr0;
      S.fro = pack(fro);
    }
    __syncwarp();
  }
  R.shifted = 0;
  if constexpr (!SMALL) {
    R.A = reinterpret_cast<int4*>(G);
    R.ld = n;
    R.n = n;
    R.own = g.own;
    R.P = g.P ? g.P + w * (size_t)(2 * kNb) * n : nullptr;
    R.us = sm;
    R.part = reinterpret_cast<longlong2*>(R.us + n);
    const int nparts = max(kWarps, g.own / 32) * 32;
    R.vw = reinterpret_cast<int4*>(R.part + nparts);
    R.stage = reinterpret_cast<int4*>(R.part + nparts) + (VWS ? 2 * kNb * g.own : 0);
    reduce<MULTI, VWS>(R, n - kTail);  // ends with a barrier of the walker
    if (rank != 0) return;
    const int4* A0 = R.A + (n - kTail) + (size_t)(n - kTail) * n;
    for (int x = t; x < kTail * kTail; x += 32 * W) {
      const int r = x % kTail, c = x / kTail;
      tail_A[r + c * kLd] = __ldcg(A0 + r + (size_t)c * n);
    }
    __syncthreads();
  }
  reduce_tail<kOrder / 32, W>(tail_A, nt, tail_us, tail_ws, tail_part, dw + (n - nt), ew + (n - nt), R.eunit,
              R.shifted, S);
}

constexpr size_t tail_smem(int order, int warps) {
  return ((size_t)3 * order + (size_t)warps * 32 + (size_t)order * (order + 1)) * 16;
}

// The largest shared-memory request of any order. The limit is a property of
// the kernel on a device, shared by all threads that launch it: it is set to
// this one value, so that no plan's launch depends on another's order.
constexpr size_t kSmemLimit = kSmemMax - sizeof(Shared) - 512;

// What an order-n reduction on clusters of cl CTAs asks for.
TriShape shape_for(int n, int cl, bool packed) {
  TriShape s;
  s.warps = packed ? kPackedWarps : kWarps;
  if (n <= kTail) {
    s.smem = packed ? tail_smem(kPacked, kPackedWarps) : tail_smem(kTail, kWarps);
    return s;
  }
  s.cl = cl;
  const int groups = (n + 31) / 32;
  s.own = (groups + cl - 1) / cl * 32;
  const size_t fixed = (size_t)n * 16 + (size_t)std::max(kWarps, s.own / 32) * 32 * 16;
  const size_t vw = (size_t)2 * kNb * s.own * 16;
  const size_t stage = (size_t)kWarps * 2 * kNb * kStrip * 16;
  s.vws = fixed + vw + (cl > 1 ? stage : 0) <= kSmemLimit;
  s.smem = std::max(tail_smem(kTail, kWarps), fixed + (s.vws ? vw : 0) + (cl > 1 || !s.vws ? stage : 0));
  s.panel = cl > 1 || !s.vws ? (size_t)2 * kNb * n * sizeof(int4) : 0;
  return s;
}

void launch_config(const TriShape& s, int64_t walkers, cudaStream_t st, cudaLaunchConfig_t* cfg,
                   cudaLaunchAttribute* at) {
  cfg->gridDim = dim3((unsigned)(walkers * s.cl));
  cfg->blockDim = dim3((unsigned)s.warps * 32);
  cfg->dynamicSmemBytes = s.smem;
  cfg->stream = st;
  at->id = cudaLaunchAttributeClusterDimension;
  at->val.clusterDim.x = (unsigned)s.cl;
  at->val.clusterDim.y = 1;
  at->val.clusterDim.z = 1;
  cfg->attrs = at;
  cfg->numAttrs = s.cl > 1 ? 1 : 0;
}

template <bool MULTI, bool VWS, int ROWS, int W = kWarps>
cudaError_t launch_reduce(const TriArgs& a, int64_t walkers, const TriShape& s, cudaStream_t st) {
  cudaLaunchConfig_t cfg = {};
  cudaLaunchAttribute at[1];
  launch_config(s, walkers, st, &cfg, at);
  const cudaError_t err = cudaLaunchKernelEx(&cfg, tri_reduce_kernel<MULTI, VWS, ROWS, W>, a);
  if (err != cudaSuccess) return err;
  count_launch();
  return cudaGetLastError();
}

// Once per device: five calls of the driver, a sixth of a small plan's making.
cudaError_t set_smem_limits() {
  static std::mutex mu;
  static bool done[kAttrDevices];
  int dev = 0;
  cudaError_t e = cudaGetDevice(&dev);
  if (e != cudaSuccess) return e;
  const bool tracked = dev >= 0 && dev < kAttrDevices;
  std::lock_guard<std::mutex> lk(mu);
  if (tracked && done[dev]) return cudaSuccess;
  // (the packed kernel's request needs no raised limit)
  static_assert(tail_smem(kPacked, kPackedWarps) + sizeof(Shared) <= 48 * 1024, "packed CTA");
  const void* kernels[] = {(const void*)tri_reduce_kernel<false, true, kTail / 32, kWarps>,
                           (const void*)tri_reduce_kernel<true, true, 0, kWarps>,
                           (const void*)tri_reduce_kernel<true, false, 0, kWarps>,
                           (const void*)tri_reduce_kernel<false, true, 0, kWarps>,
                           (const void*)tri_reduce_kernel<false, false, 0, kWarps>};
  for (const void* k : kernels) {
    e = cudaFuncSetAttribute(k, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)kSmemLimit);
    if (e != cudaSuccess) return e;
  }
  if (tracked) done[dev] = true;
  return cudaSuccess;
}

// CTAs per walker: the most (up to 8, and a group of 32 rows each before the
// tail) for which the device holds every walker's cluster at once. Clusters
// of 8 fit 15 times on a GB300 (GPCs of 18 to 20 SMs, one CTA per SM), of 4
// 36 times, so 16 walkers run on clusters of 7 at most; a second wave would
// double the time. The shared-memory limits must be set.
int tri_cluster(int64_t walkers, int n) {
  if (n <= kTail || walkers <= 0) return 1;
  static std::mutex mu;
  static int active[kAttrDevices][kMaxCl + 1];  // clusters the device holds, 0 = not asked yet
  int dev = 0;
  if (cudaGetDevice(&dev) != cudaSuccess || dev < 0 || dev >= kAttrDevices) return 1;
  std::lock_guard<std::mutex> lk(mu);
  for (int cl = std::min(kMaxCl, (n - kTail) / 32); cl > 1; --cl) {
    int& a = active[dev][cl];
    if (a == 0) {
      // the largest request any order makes: one CTA per SM
      cudaLaunchConfig_t cfg = {};
      cudaLaunchAttribute at[1];
      TriShape s;
      s.cl = cl;
      s.warps = kWarps;
      s.smem = kSmemLimit;
      int c = 0;
      launch_config(s, 1, nullptr, &cfg, at);
      if (cudaOccupancyMaxActiveClusters(&c, tri_reduce_kernel<true, true, 0, kWarps>, &cfg) !=
          cudaSuccess) {
        cudaGetLastError();
        return 1;
      }
      a = std::max(c, 1);
    }
    if (a >= walkers) return cl;
  }
  return 1;
}

}  // namespace

cudaError_t tri_shape(int64_t walkers, int n, int sms, TriShape* out) {
  const cudaError_t e = set_smem_limits();
  *out = shape_for(n, e == cudaSuccess ? tri_cluster(walkers, n) : 1,
                   n <= kPacked && walkers > sms);
  return e;
}

cudaError_t launch_tridiag(double2* gram, int64_t walkers, int n, const TriShape& s, void* panel,
                           double* d, double* e, cudaStream_t st) {
  if (walkers <= 0) return cudaSuccess;
  const TriArgs a{gram, static_cast<int4*>(panel), d, e, n, s.own};
  if (s.warps < kWarps)
    return launch_reduce<false, true, kPacked / 32, kPackedWarps>(a, walkers, s, st);
  if (n <= kTail) return launch_reduce<false, true, kTail / 32>(a, walkers, s, st);
  if (s.cl > 1)
    return s.vws ? launch_reduce<true, true, 0>(a, walkers, s, st)
                 : launch_reduce<true, false, 0>(a, walkers, s, st);
  return s.vws ? launch_reduce<false, true, 0>(a, walkers, s, st)
               : launch_reduce<false, false, 0>(a, walkers, s, st);
}

}  // namespace bg
