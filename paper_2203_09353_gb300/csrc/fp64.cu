// FP64 / complex128 path of Eq. (1) (Sec. 2): C_i = alpha A_i B_i + beta C_i.
//
// One persistent kernel walks a list of work items; each item runs one of
// the tile programs below on one tile (or one group of small instances):
//  * small programs: one warp per instance, several instances per CTA (the
//    tiny-matrix idea the paper cites in Sec. 2: several small C per block);
//  * tile programs: a 2-D output tile per CTA (the tiling of Sec. 2), operands
//    staged through shared memory in double-buffered k-slices. A tile of fewer
//    outputs than the full one deals them to the threads in linear order, so
//    that the FP64 instructions grow with the outputs and not with the tile,
//    and ends at the instance's k.
// On GB300 the FP64 pipe issues 2 DFMA per clock per SM (measured 1.19
// TFLOP/s chip-wide, DMMA 1.05), i.e. one warp-wide DFMA per 64 clocks per
// SM sub-partition, so every program here is FP64-issue-bound long before
// memory matters: the design goal is only to keep DFMAs flowing on every SM
// with few non-FMA instructions.
#include <algorithm>
#include <type_traits>

#include "bgemm_internal.h"

namespace bg {

// ---- instance sources ---------------------------------------------------------

struct Desc {
  const double* A;  // complex: interleaved pairs
  const double* B;
  double* C;
  int m, n, k;
  int64_t lda, ldb, ldc;  // elements
  // Hermitian rank-k update (Sec. 3, rho = Psi Psi^H): B is A^H (A^T when
  // real), read from A; only outputs on or below the diagonal are stored,
  // and a complex diagonal gets a zero imaginary part.
  int herm;
};

// Element (p, c) of B (real).
__device__ __forceinline__ double ld_b(const Desc& d, int p, int c) {
  return d.herm ? __ldg(d.A + c + (int64_t)p * d.lda) : __ldg(d.B + p + (int64_t)c * d.ldb);
}

// Element (p, c) of B (complex).
__device__ __forceinline__ double2 ld_bc(const Desc& d, int p, int c) {
  if (d.herm) {
    double2 v = __ldg(reinterpret_cast<const double2*>(d.A) + c + (int64_t)p * d.lda);
    v.y = -v.y;
    return v;
  }
  return __ldg(reinterpret_cast<const double2*>(d.B) + p + (int64_t)c * d.ldb);
}

// Whether output (r, c) is stored (Hermitian updates keep the lower triangle).
__device__ __forceinline__ bool keep_out(const Desc& d, int r, int c) { return !d.herm || r >= c; }

// Fixed-size batch: instance i at constant strides.
struct FixedSrc {
  const double* A;
  const double* B;
  double* C;
  int m, n, k;
  int64_t lda, ldb, ldc, sA, sB, sC;
  int esz;  // doubles per element (1 real, 2 complex)
  __device__ Desc desc(int64_t i) const {
    Desc d;
    d.A = A + i * sA * esz;
    d.B = B + i * sB * esz;
    d.C = C + i * sC * esz;
    d.m = m; d.n = n; d.k = k;
    d.lda = lda; d.ldb = ldb; d.ldc = ldc;
    d.herm = 0;
    return d;
  }
  __device__ int64_t small_inst(int64_t pos) const { return pos; }
};

// Variable-size batch: rows of a device table (m, n, k, lda, ldb, ldc, a_off, b_off, c_off).
struct TableSrc {
  const int64_t* table;
  const int32_t* order;
  const double* A;
  const double* B;
  double* C;
  int esz;
  int herm;  // plan of Hermitian rank-k updates (B unused)
  __device__ Desc desc(int64_t i) const {
    const int64_t* t = table + 9 * i;
    Desc d;
    d.m = (int)t[0]; d.n = (int)t[1]; d.k = (int)t[2];
    d.lda = t[3]; d.ldb = t[4]; d.ldc = t[5];
    d.A = A + t[6] * esz;
    d.B = herm ? d.A : B + t[7] * esz;
    d.C = C + t[8] * esz;
    d.herm = herm;
    return d;
  }
  __device__ int64_t small_inst(int64_t pos) const { return order[pos]; }
};

// One step of the chain: walker w computes U[idx[w]] * Cin_w into Cout_w.
struct ChainSrc {
  const int64_t* wn;
  const int64_t* woff;
  const int64_t* pool_off;
  const int64_t* pool_n;
  int32_t pool_count;
  const int32_t* order;
  const int32_t* idx;
  const double* U;
  const double* Cin;
  double* Cout;
  int esz;
  // An index out of range, or naming a pool matrix of another size, turns the
  // walker's step into a no-op (its output is left as is).
  __device__ Desc desc(int64_t w) const {
    int n = (int)wn[w];
    const int j = idx[w];
    const bool ok = j >= 0 && j < pool_count && pool_n[j] == n;
    if (!ok) n = 0;
    Desc d;
    d.m = d.n = d.k = n;
    d.lda = d.ldb = d.ldc = n > 0 ? n : 1;
    d.A = U + (ok ? pool_off[j] : 0) * esz;
    d.B = Cin + woff[w] * esz;
    d.C = Cout + woff[w] * esz;
    d.herm = 0;
    return d;
  }
  __device__ int64_t small_inst(int64_t pos) const { return order[pos]; }
};

// ---- schedules ------------------------------------------------------------------

struct FixedSched {
  int prog;
  int tm, tn;  // 0: small program
  int64_t tiles_m, tiles_n, batch;
  __device__ WorkItem get(int64_t it) const {
    WorkItem w;
    w.prog = (int16_t)prog;
    if (tm == 0) {
      w.inst = (int32_t)(it * kSmallPerCta);
      const int64_t left = batch - it * kSmallPerCta;
      w.count = (int16_t)(left < kSmallPerCta ? left : kSmallPerCta);
      w.r0 = 0;
      w.c0 = 0;
    } else {
      const int64_t per = tiles_m * tiles_n;
      w.inst = (int32_t)(it / per);
      const int64_t t = it - (it / per) * per;
      w.r0 = (int32_t)((t % tiles_m) * tm);
      w.c0 = (int32_t)((t / tiles_m) * tn);
      w.count = tile_extent(tm, tn);
    }
    return w;
  }
};

struct TableSched {
  const WorkItem* items;
  __device__ WorkItem get(int64_t it) const { return items[it]; }
};

// ---- real tile program: 64x64 outputs, BK = 16, DFMA ----------------------------

constexpr int TR = 64, BKR = 16;

struct SmemR64 {
  double a[2][BKR][TR];  // a[s][kk][row]
  double b[2][BKR][TR];  // b[s][kk][col]
};

// f with beta's part of Eq. (1) in or out: a branch outside the loop over the outputs,
// where the compiler cannot predicate the FP64 instructions that it skips (20000
// complex instances of 16 x 16 x 1 122 us with the test inside, 82 without).
template <class F>
__device__ __forceinline__ void with_beta(const Scalars& s, const F& f) {
  if (s.beta_zero) f(std::false_type{});
  else f(std::true_type{});
}

// alpha acc + beta c (Eq. 1).
template <bool BETA>
__device__ __forceinline__ double combine(double acc, double c, const Scalars& s) {
  double v = s.alpha_re * acc;
  if constexpr (BETA) v = fma(s.beta_re, c, v);
  return v;
}
template <bool BETA>
__device__ __forceinline__ double2 combine(double2 acc, double2 c, const Scalars& s) {
  double2 v;
  v.x = s.alpha_re * acc.x - s.alpha_im * acc.y;
  v.y = s.alpha_re * acc.y + s.alpha_im * acc.x;
  if constexpr (BETA) {
    v.x = fma(s.beta_re, c.x, fma(-s.beta_im, c.y, v.x));
    v.y = fma(s.beta_re, c.y, fma(s.beta_im, c.x, v.y));
  }
  return v;
}
__device__ __forceinline__ void real_diagonal(double&) {}
__device__ __forceinline__ void real_diagonal(double2& v) { v.y = 0.0; }

// Output (r, c) of an instance (T: double or double2).
template <bool BETA, class T>
__device__ __forceinline__ void store_out(const Desc& d, const Scalars& s, int r, int c, T acc) {
  if (!keep_out(d, r, c)) return;
  T* cp = reinterpret_cast<T*>(d.C) + r + (int64_t)c * d.ldc;
  T v = combine<BETA>(acc, BETA ? *cp : T{}, s);
  if (d.herm && r == c) real_diagonal(v);
  *cp = v;
}

// A thread's N x N outputs from (r, c) on; all of C is loaded before the first use.
template <class T, int N>
__device__ __forceinline__ void store_block(const Desc& d, const Scalars& s, int r, int c,
                                            const T (&acc)[N][N]) {
  with_beta(s, [&](auto beta) {
    constexpr bool BETA = decltype(beta)::value;
    T* cp = reinterpret_cast<T*>(d.C) + r + (int64_t)c * d.ldc;
    T cv[N][N];
    bool on[N][N];
#pragma unroll
    for (int j = 0; j < N; ++j)
#pragma unroll
      for (int i = 0; i < N; ++i) {
        on[i][j] = r + i < d.m && c + j < d.n && keep_out(d, r + i, c + j);
        if (BETA && on[i][j]) cv[i][j] = cp[i + (int64_t)j * d.ldc];
      }
#pragma unroll
    for (int j = 0; j < N; ++j)
#pragma unroll
      for (int i = 0; i < N; ++i) {
        if (!on[i][j]) continue;
        T v = combine<BETA>(acc[i][j], BETA ? cv[i][j] : T{}, s);
        if (d.herm && r + i == c + j) real_diagonal(v);
        cp[i + (int64_t)j * d.ldc] = v;
      }
  });
}

// The products of a k-slice for a warp's nj <= NJ outputs in linear order (nj is
// the same in all its lanes). A warp with fewer than NJ takes one output after
// another, so that a branch on nj lies outside the loop over k: inside it the
// compiler may predicate instead, and a DFMA that is off in every lane holds the
// FP64 pipe as long as one that is on (456 complex instances of 32 x 9 x 32 61 us
// so and 35 with the branch outside, 30000 real ones of 2 x 200 x 64 8010 and 3820).
template <int NJ, class F>
__device__ __forceinline__ void linear_products(int nj, int kend, F mul) {
  if (nj >= NJ) {
#pragma unroll 2
    for (int kk = 0; kk < kend; ++kk)
#pragma unroll
      for (int j = 0; j < NJ; ++j) mul(j, kk);
  } else {
#pragma unroll
    for (int j = 0; j < NJ - 1; ++j) {
      if (j >= nj) break;
#pragma unroll 2
      for (int kk = 0; kk < kend; ++kk) mul(j, kk);
    }
  }
}

// Rows r0 .. r0 + tm - 1 and columns c0 .. c0 + tn - 1 (tm, tn <= 64) of one
// instance; FULL: 64 x 64, or what the instance leaves of it, 4 x 4 outputs per
// thread (for more outputs than NJ = 8 holds). Otherwise output o of the tile's
// mb x nb (column-major) goes to thread o mod 256, NJ outputs to a thread: a DFMA takes its 16 clocks per SM
// whether 1 or 32 of the warp's lanes are active (measured), so padding a
// ragged tile to 64 x 64 costs in full, while the two extra shared-memory
// reads per DFMA of this order are hidden behind it.
template <bool FULL, int NJ>
__device__ __forceinline__ void tile_r64(const Desc& d, int r0, int c0, int mb, int nb,
                                         const Scalars& s, SmemR64& sm) {
  const int tid = threadIdx.x;
  const int tx = tid & 15, ty = tid >> 4;
  const int K = s.alpha_zero ? 0 : d.k;
  double acc[FULL ? 4 : 1][FULL ? 4 : 1];
  double lin[FULL ? 1 : NJ];
  int rc[FULL ? 1 : NJ];  // row and column of each output in the tile, row | column << 16
  if constexpr (FULL) {
#pragma unroll
    for (int i = 0; i < 4; ++i)
#pragma unroll
      for (int j = 0; j < 4; ++j) acc[i][j] = 0.0;
  } else {
#pragma unroll
    for (int j = 0; j < NJ; ++j) {
      const int o = tid + kFp64Threads * j;
      lin[j] = 0.0;
      const int col = o / mb;
      rc[j] = col < nb ? (o - col * mb) | col << 16 : 0;  // beyond the tile: computed, not stored
    }
  }
  // outputs of this warp's lanes: a warp past the tile's end issues nothing
  const int nj = (mb * nb - (tid & ~31) + kFp64Threads - 1) / kFp64Threads;

  // global -> register staging: A 64 rows x 16 k, B 16 k x 64 cols
  const int ar = tid & 63, ak = tid >> 6;  // row, k (+4j)
  const int bk = tid & 15, bc = tid >> 4;  // k, col (+16j)
  double ra[4], rb[4];
  auto gload = [&](int k0) {
#pragma unroll
    for (int j = 0; j < 4; ++j) {
      const int r = r0 + ar, kk = k0 + ak + 4 * j;
      ra[j] = (ar < mb && kk < K) ? __ldg(d.A + r + (int64_t)kk * d.lda) : 0.0;
      const int kb = k0 + bk, c = c0 + bc + 16 * j;
      rb[j] = (kb < K && bc + 16 * j < nb) ? ld_b(d, kb, c) : 0.0;
    }
  };
  auto sstore = [&](int st) {
#pragma unroll
    for (int j = 0; j < 4; ++j) {
      sm.a[st][ak + 4 * j][ar] = ra[j];
      sm.b[st][bk][bc + 16 * j] = rb[j];
    }
  };

  if (K > 0) {
    gload(0);
    sstore(0);
  }
  __syncthreads();
  int st = 0;
  for (int k0 = 0; k0 < K; k0 += BKR) {
    const bool more = k0 + BKR < K;
    if (more) gload(k0 + BKR);
    if constexpr (!FULL) {
      const int kend = min(BKR, K - k0);
      linear_products<NJ>(nj, kend, [&](int j, int kk) {
        lin[j] = fma(sm.a[st][kk][rc[j] & 0xFFFF], sm.b[st][kk][rc[j] >> 16], lin[j]);
      });
    } else
#pragma unroll
    for (int kk = 0; kk < BKR; ++kk) {
      const double2 a01 = *reinterpret_cast<const double2*>(&sm.a[st][kk][ty * 4]);
      const double2 a23 = *reinterpret_cast<const double2*>(&sm.a[st][kk][ty * 4 + 2]);
      const double2 b01 = *reinterpret_cast<const double2*>(&sm.b[st][kk][tx * 4]);
      const double2 b23 = *reinterpret_cast<const double2*>(&sm.b[st][kk][tx * 4 + 2]);
      const double a[4] = {a01.x, a01.y, a23.x, a23.y};
      const double b[4] = {b01.x, b01.y, b23.x, b23.y};
#pragma unroll
      for (int i = 0; i < 4; ++i)
#pragma unroll
        for (int j = 0; j < 4; ++j) acc[i][j] = fma(a[i], b[j], acc[i][j]);
    }
    if (more) sstore(st ^ 1);
    __syncthreads();
    st ^= 1;
  }

  if constexpr (!FULL) {
    with_beta(s, [&](auto beta) {
#pragma unroll
      for (int j = 0; j < NJ; ++j)
        if (tid + kFp64Threads * j < mb * nb)
          store_out<decltype(beta)::value>(d, s, r0 + (rc[j] & 0xFFFF), c0 + (rc[j] >> 16), lin[j]);
    });
    return;
  } else
  store_block(d, s, r0 + ty * 4, c0 + tx * 4, acc);
}

// ---- real tile program on the FP64 tensor cores: mma.sync m8n8k4 -----------------
// 8 warps as 2 (rows) x 4 (cols); each warp owns 32x16 outputs = 4x2 fragments.
// Fragment layout (PTX ISA, mma .f64 m8n8k4, row.col): lane = 4*g + t;
// A(g, t), B(t, g), C(g, 2t + {0,1}).

__device__ __forceinline__ void dmma_884(double& c0, double& c1, double a, double b) {
  asm volatile("mma.sync.aligned.m8n8k4.row.col.f64.f64.f64.f64 {%0,%1}, {%2}, {%3}, {%0,%1};\n"
               : "+d"(c0), "+d"(c1)
               : "d"(a), "d"(b));
}

__device__ __forceinline__ void tile_r64_dmma(const Desc& d, int r0, int c0, const Scalars& s,
                                              SmemR64& sm) {
  const int tid = threadIdx.x;
  const int lane = tid & 31, warp = tid >> 5;
  const int wm = warp & 1, wn = warp >> 1;
  const int g = lane >> 2, t = lane & 3;
  const int K = s.alpha_zero ? 0 : d.k;
  double acc[4][2][2];
#pragma unroll
  for (int i = 0; i < 4; ++i)
#pragma unroll
    for (int j = 0; j < 2; ++j) acc[i][j][0] = acc[i][j][1] = 0.0;

  const int ar = tid & 63, ak = tid >> 6;
  const int bk = tid & 15, bc = tid >> 4;
  double ra[4], rb[4];
  auto gload = [&](int k0) {
#pragma unroll
    for (int j = 0; j < 4; ++j) {
      const int r = r0 + ar, kk = k0 + ak + 4 * j;
      ra[j] = (r < d.m && kk < K) ? __ldg(d.A + r + (int64_t)kk * d.lda) : 0.0;
      const int kb = k0 + bk, c = c0 + bc + 16 * j;
      rb[j] = (kb < K && c < d.n) ? ld_b(d, kb, c) : 0.0;
    }
  };
  auto sstore = [&](int st) {
#pragma unroll
    for (int j = 0; j < 4; ++j) {
      sm.a[st][ak + 4 * j][ar] = ra[j];
      sm.b[st][bk][bc + 16 * j] = rb[j];
    }
  };
  if (K > 0) {
    gload(0);
    sstore(0);
  }
  __syncthreads();
  int st = 0;
  for (int k0 = 0; k0 < K; k0 += BKR) {
    const bool more = k0 + BKR < K;
    if (more) gload(k0 + BKR);
#pragma unroll
    for (int k4 = 0; k4 < BKR; k4 += 4) {
      double a[4], b[2];
#pragma unroll
      for (int i = 0; i < 4; ++i) a[i] = sm.a[st][k4 + t][wm * 32 + i * 8 + g];
#pragma unroll
      for (int j = 0; j < 2; ++j) b[j] = sm.b[st][k4 + t][wn * 16 + j * 8 + g];
#pragma unroll
      for (int i = 0; i < 4; ++i)
#pragma unroll
        for (int j = 0; j < 2; ++j) dmma_884(acc[i][j][0], acc[i][j][1], a[i], b[j]);
    }
    if (more) sstore(st ^ 1);
    __syncthreads();
    st ^= 1;
  }
#pragma unroll
  for (int i = 0; i < 4; ++i) {
    const int r = r0 + wm * 32 + i * 8 + g;
    if (r >= d.m) continue;
#pragma unroll
    for (int j = 0; j < 2; ++j)
#pragma unroll
      for (int h = 0; h < 2; ++h) {
        const int c = c0 + wn * 16 + j * 8 + 2 * t + h;
        if (c >= d.n || !keep_out(d, r, c)) continue;
        double* cp = d.C + r + (int64_t)c * d.ldc;
        double v = s.alpha_re * acc[i][j][h];
        if (!s.beta_zero) v = fma(s.beta_re, *cp, v);
        *cp = v;
      }
  }
}

// ---- complex tile program: 32x32 complex outputs, BK = 16 ---------------------------

constexpr int TC = 32, BKC = 16;

struct SmemC128 {
  double2 a[2][BKC][TC];
  double2 b[2][BKC][TC];
};

__device__ __forceinline__ void cmac(double2& acc, double2 a, double2 b) {
  acc.x = fma(a.x, b.x, acc.x);
  acc.x = fma(-a.y, b.y, acc.x);
  acc.y = fma(a.x, b.y, acc.y);
  acc.y = fma(a.y, b.x, acc.y);
}

// As tile_r64: FULL is a whole 32 x 32 tile (2 x 2 outputs per thread), NJ the
// outputs per thread in linear order otherwise.
template <bool FULL, int NJ>
__device__ __forceinline__ void tile_c128(const Desc& d, int r0, int c0, int mb, int nb,
                                          const Scalars& s, SmemC128& sm) {
  const int tid = threadIdx.x;
  const int tx = tid & 15, ty = tid >> 4;
  const int K = s.alpha_zero ? 0 : d.k;
  const double2* A = reinterpret_cast<const double2*>(d.A);
  double2 acc[FULL ? 2 : 1][FULL ? 2 : 1];
  double2 lin[FULL ? 1 : NJ];
  int rc[FULL ? 1 : NJ];
  if constexpr (FULL) {
#pragma unroll
    for (int i = 0; i < 2; ++i)
#pragma unroll
      for (int j = 0; j < 2; ++j) acc[i][j] = make_double2(0.0, 0.0);
  } else {
#pragma unroll
    for (int j = 0; j < NJ; ++j) {
      const int o = tid + kFp64Threads * j;
      lin[j] = make_double2(0.0, 0.0);
      const int col = o / mb;
      rc[j] = col < nb ? (o - col * mb) | col << 16 : 0;
    }
  }
  // outputs of this warp's lanes: a warp past the tile's end issues nothing
  const int nj = (mb * nb - (tid & ~31) + kFp64Threads - 1) / kFp64Threads;

  const int ar = tid & 31, ak = tid >> 5;  // row, k (+8j)
  const int bk = tid & 15, bc = tid >> 4;  // k, col (+16j)
  double2 ra[2], rb[2];
  const double2 z = make_double2(0.0, 0.0);
  auto gload = [&](int k0) {
#pragma unroll
    for (int j = 0; j < 2; ++j) {
      const int r = r0 + ar, kk = k0 + ak + 8 * j;
      ra[j] = (ar < mb && kk < K) ? __ldg(A + r + (int64_t)kk * d.lda) : z;
      const int kb = k0 + bk, c = c0 + bc + 16 * j;
      rb[j] = (kb < K && bc + 16 * j < nb) ? ld_bc(d, kb, c) : z;
    }
  };
  auto sstore = [&](int st) {
#pragma unroll
    for (int j = 0; j < 2; ++j) {
      sm.a[st][ak + 8 * j][ar] = ra[j];
      sm.b[st][bk][bc + 16 * j] = rb[j];
    }
  };
  if (K > 0) {
    gload(0);
    sstore(0);
  }
  __syncthreads();
  int st = 0;
  for (int k0 = 0; k0 < K; k0 += BKC) {
    const bool more = k0 + BKC < K;
    if (more) gload(k0 + BKC);
    if constexpr (!FULL) {
      const int kend = min(BKC, K - k0);
      linear_products<NJ>(nj, kend, [&](int j, int kk) {
        cmac(lin[j], sm.a[st][kk][rc[j] & 0xFFFF], sm.b[st][kk][rc[j] >> 16]);
      });
    } else
#pragma unroll
    for (int kk = 0; kk < BKC; ++kk) {
      const double2 a0 = sm.a[st][kk][ty * 2], a1 = sm.a[st][kk][ty * 2 + 1];
      const double2 b0 = sm.b[st][kk][tx * 2], b1 = sm.b[st][kk][tx * 2 + 1];
      cmac(acc[0][0], a0, b0);
      cmac(acc[0][1], a0, b1);
      cmac(acc[1][0], a1, b0);
      cmac(acc[1][1], a1, b1);
    }
    if (more) sstore(st ^ 1);
    __syncthreads();
    st ^= 1;
  }
  if constexpr (!FULL) {
    with_beta(s, [&](auto beta) {
#pragma unroll
      for (int j = 0; j < NJ; ++j)
        if (tid + kFp64Threads * j < mb * nb)
          store_out<decltype(beta)::value>(d, s, r0 + (rc[j] & 0xFFFF), c0 + (rc[j] >> 16), lin[j]);
    });
    return;
  } else
  store_block(d, s, r0 + ty * 2, c0 + tx * 2, acc);
}

// ---- small programs: a warp per instance --------------------------------------
// The m*n outputs in column-major order, 32 MAXOUT at a time: lane t owns outputs
// o = t + 32 j (j < MAXOUT) of them, (r, c) = (o mod m, o div m). When m divides 32
// the row is the same for every j and the column steps by 32 / m, so one A load
// feeds up to MAXOUT DFMAs; otherwise every output loads its own A element.

// Runs f with the smallest of the powers of two up to MAXOUT that is not below cnt
// (the outputs per lane, the same in all lanes): a DFMA that is off in every
// lane would take the FP64 pipe as long as one that is on.
template <int MAXOUT, class F>
__device__ __forceinline__ void with_outputs(int cnt, const F& f) {
  if constexpr (MAXOUT > 1) {
    if (cnt <= MAXOUT / 2) {
      with_outputs<MAXOUT / 2>(cnt, f);
      return;
    }
  }
  f(std::integral_constant<int, MAXOUT>{});
}

__device__ __forceinline__ void small_product(double& acc, double a, double b) {
  acc = fma(a, b, acc);
}
__device__ __forceinline__ void small_product(double2& acc, double2 a, double2 b) {
  cmac(acc, a, b);
}
__device__ __forceinline__ double small_b(const Desc& d, int p, int c, double) {
  return ld_b(d, p, c);
}
__device__ __forceinline__ double2 small_b(const Desc& d, int p, int c, double2) {
  return ld_bc(d, p, c);
}
// T: double or double2.
template <class T, int MAXOUT>
__device__ __forceinline__ void small_instance(const Desc& d, const Scalars& s) {
  const int lane = threadIdx.x & 31;
  const int m = d.m, n = d.n, mn = m * n;
  const int K = s.alpha_zero ? 0 : d.k;
  const T* A = reinterpret_cast<const T*>(d.A);
  const T* B = reinterpret_cast<const T*>(d.B);
  const bool divides = m > 0 && (32 % m) == 0;
  for (int o0 = 0; o0 < mn; o0 += 32 * MAXOUT) {
    with_outputs<MAXOUT>((mn - o0 + 31) / 32, [&](auto outputs) {
      constexpr int N = decltype(outputs)::value;
      T acc[N] = {};
      if (divides) {
        const int r = lane % m, cstep = 32 / m, c0 = o0 / m + lane / m;
        const T* ap = A + r;
        const T* bp = B + (int64_t)c0 * d.ldb;
        const int64_t bstep = (int64_t)cstep * d.ldb;
#pragma unroll 1
        for (int p = 0; p < K; ++p) {
          const T a = __ldg(ap + (int64_t)p * d.lda);
#pragma unroll
          for (int j = 0; j < N; ++j)
            if (c0 + j * cstep < n)
              small_product(acc[j], a, d.herm ? small_b(d, p, c0 + j * cstep, T{})
                                              : __ldg(bp + p + j * bstep));
        }
        with_beta(s, [&](auto beta) {
#pragma unroll
          for (int j = 0; j < N; ++j)
            if (c0 + j * cstep < n)
              store_out<decltype(beta)::value>(d, s, r, c0 + j * cstep, acc[j]);
        });
      } else {
        int rc[N];  // row | column << 16
#pragma unroll
        for (int j = 0; j < N; ++j) {
          const int o = min(o0 + lane + 32 * j, mn - 1), c = o / m;
          rc[j] = (o - c * m) | c << 16;
        }
#pragma unroll 1
        for (int p = 0; p < K; ++p) {
          const T* ap = A + (int64_t)p * d.lda;
#pragma unroll
          for (int j = 0; j < N; ++j)
            small_product(acc[j], __ldg(ap + (rc[j] & 0xFFFF)), small_b(d, p, rc[j] >> 16, T{}));
        }
        with_beta(s, [&](auto beta) {
#pragma unroll
          for (int j = 0; j < N; ++j)
            if (o0 + lane + 32 * j < mn)
              store_out<decltype(beta)::value>(d, s, rc[j] & 0xFFFF, rc[j] >> 16, acc[j]);
        });
      }
    });
  }
}

// Outputs that a small program holds at once: MAXOUT 8 real, 4 complex.
constexpr int kSmallR64 = 256, kSmallC128 = 128;

// ---- the persistent kernel ---------------------------------------------------------

// CTAS: CTAs per SM. Several hide each other's start (work item, first operand
// loads): two where tiles are ragged (33^3 x 1000: 150 -> 102 us), three where
// all are small, in the registers that the small tiles leave (32^3 x 20000:
// 2710, 1540 and 1257 us with one, two and three). Full tiles run 2-5% faster
// alone (128^3 x 100: 430 -> 411 us).
// A kernel per element type: with both types' programs in one, either's registers
// and order of instructions came to depend on the other's.
template <int CTAS, bool CPLX, class Src, class Sched>
__global__ void __launch_bounds__(kFp64Threads, CTAS)
    fp64_persistent(Src src, Sched sched, int64_t n_items, Scalars s) {
  __shared__ __align__(16) std::conditional_t<CPLX, SmemC128, SmemR64> sm;
  const int warp = threadIdx.x >> 5;
  for (int64_t it = blockIdx.x; it < n_items; it += gridDim.x) {
    const WorkItem w = sched.get(it);
    if constexpr (CTAS < 3) {  // (three CTAs: small tiles only)
      if (w.prog == (CPLX ? PROG_C128_SMALL : PROG_R64_SMALL)) {
        if (warp < w.count) {
          const Desc d = src.desc(src.small_inst((int64_t)w.inst + warp));
          if constexpr (CPLX) small_instance<double2, kSmallC128 / 32>(d, s);
          else small_instance<double, kSmallR64 / 32>(d, s);
        }
        continue;
      }
      if constexpr (!CPLX) {
        if (w.prog == PROG_R64_DMMA) {
          tile_r64_dmma(src.desc(w.inst), w.r0, w.c0, s, sm);
          continue;
        }
      }
    }
    const Desc d = src.desc(w.inst);
    int tm, tn;
    tile_extent_of(w.count, CPLX ? TC : TR, &tm, &tn);
    const int mb = min(tm, d.m - w.r0), nb = min(tn, d.n - w.c0);
    if (mb <= 0 || nb <= 0) continue;  // (a chain index that names no matrix)
    if constexpr (CPLX) {
      const int per = tile_program_c128(mb * nb);
      if (CTAS < 3 && mb == TC && nb == TC) tile_c128<true, 1>(d, w.r0, w.c0, mb, nb, s, sm);
      else if (CTAS < 3 && per == 4) tile_c128<false, 4>(d, w.r0, w.c0, mb, nb, s, sm);
      else if (per > 1) tile_c128<false, 2>(d, w.r0, w.c0, mb, nb, s, sm);
      else tile_c128<false, 1>(d, w.r0, w.c0, mb, nb, s, sm);
    } else {
      const int per = tile_program_r64(mb * nb);
      if (CTAS < 3 && per == 16) tile_r64<true, 1>(d, w.r0, w.c0, mb, nb, s, sm);
      else if (CTAS < 3 && per == 8) tile_r64<false, 8>(d, w.r0, w.c0, mb, nb, s, sm);
      else if (per > 2) tile_r64<false, 4>(d, w.r0, w.c0, mb, nb, s, sm);
      else tile_r64<false, 2>(d, w.r0, w.c0, mb, nb, s, sm);
    }
  }
}

// ---- host side -----------------------------------------------------------------------

bool prog_is_small(int prog) { return prog == PROG_R64_SMALL || prog == PROG_C128_SMALL; }

void prog_tile(int prog, int* tm, int* tn) {
  switch (prog) {
    case PROG_R64_TILE:
    case PROG_R64_DMMA: *tm = TR; *tn = TR; break;
    case PROG_C128_TILE: *tm = TC; *tn = TC; break;
    default: *tm = 0; *tn = 0; break;
  }
}

// The small programs take what they hold at once, and four times as many outputs
// where k is short: a tile's start (descriptor, operands to shared memory, barriers)
// then costs more than its products, above all for a few rows or columns, of
// which a tile holds 64. Measured with sizes at the lines below, tiles and small
// program, us for 30000 real or 20000 complex instances: 1 x 300 x 16 1476 and 693,
// 2 x 200 x 16 1191 and 758 (x 32 2033 and 1499, but 3000 of them 207 and 229),
// 5 x 100 x 8 546 and 400 (x 16 736 and 735), 20 x 20 x 4 260 and 185 (x 8 342 and
// 328), 3000 of 32 x 32 x 3 40 and 39 (x 4 43 and 47); complex 1 x 300 x 32 3162 and
// 1520, 16 x 16 x 8 390 and 329 (x 16 654 and 620, but 3000 of them 106 and 112).
static bool small_fits(bg_dtype dt, int64_t m, int64_t n, int64_t k) {
  const int64_t held = dt == BG_R64 ? kSmallR64 : kSmallC128, thin = std::min(m, n);
  const int64_t k_max = dt == BG_C128       ? (thin <= 2 ? 32 : 8)
                        : thin < 8          ? (thin <= 2 ? 16 : 8)
                        : m * n <= 2 * held ? 4
                                            : 3;
  return m * n <= (k <= k_max ? 4 * held : held);
}

// Whether the small programs are to run `instances` that fit them: where groups of
// 8 fill two CTAs per SM, and fewer where a warp's chain of products is so short
// that tiles take longer to start: 6 per SM up to k = 4, 4 per SM with one or two rows
// or columns up to k = 8 (tiles and small program, us for 1000: 1 x 300 x 2 34.9
// and 8.3, 300 x 1 x 8 39.0 and 24.6, 8 x 64 x 2 12.4 and 10.3, complex 4 x 100 x 4
// 34.9 and 24.2; but 20 x 20 x 8 16.4 and 24; for 400: 4 x 100 x 2 9.3 and 10.2).
bool small_pays(int64_t m, int64_t n, int64_t k, int64_t instances, int sms) {
  if ((instances + kSmallPerCta - 1) / kSmallPerCta >= 2 * (int64_t)sms) return true;
  const bool thin = std::min(m, n) <= 2;
  return k <= (thin ? 8 : 4) && m * n * k <= 2400 && instances >= (thin ? 4 : 6) * (int64_t)sms;
}

bool prog_fits(int prog, bg_dtype dt, int64_t m, int64_t n, int64_t k) {
  switch (prog) {
    case PROG_R64_SMALL: return dt == BG_R64 && small_fits(dt, m, n, k);
    case PROG_C128_SMALL: return dt == BG_C128 && small_fits(dt, m, n, k);
    case PROG_R64_TILE:
    case PROG_R64_DMMA: return dt == BG_R64;
    case PROG_C128_TILE: return dt == BG_C128;
    default: return false;
  }
}

bool fp64_tile_ok(bg_dtype dt, int64_t tm, int64_t tn) {
  const int64_t T = dt == BG_C128 ? TC : TR;
  if (tm > T || tn > T) return false;
  return (tm == T && tn == T) || tm * tn <= (dt == BG_C128 ? 4 : 8) * kFp64Threads;
}

void fp64_tile_split(bg_dtype dt, int64_t m, int64_t n, int64_t k, int64_t batch, int sms, int* tm,
                     int* tn) {
  const int64_t T = dt == BG_C128 ? TC : TR;
  *tm = (int)T;
  *tn = dt == BG_C128 ? (int)T : (int)T / 2;
  if (m < 1 || n < 1) return;
  // (the search takes a good part of a microsecond: a caller's next call most
  // often has the same shape)
  struct Last {
    int64_t key[6];
    int tm, tn;
  };
  static thread_local Last last = {{-1, 0, 0, 0, 0, 0}, 0, 0};
  const int64_t key[6] = {(int64_t)dt, m, n, k, batch, sms};
  if (std::equal(key, key + 6, last.key)) {
    *tm = last.tm;
    *tn = last.tn;
    return;
  }
  // time in clocks: the tiles' DFMAs (16 clocks of an SM per warp and k), in
  // whole rounds over the SMs, plus what starting a tile costs where the two
  // CTAs of an SM cannot hide it
  const double dfma = (dt == BG_C128 ? 4.0 : 1.0) * 16.0 * (double)std::max<int64_t>(k, 1);
  double best = 1e300;
  const int64_t pm0 = (m + T - 1) / T, pn0 = (n + T - 1) / T;
  for (int64_t pm = pm0; pm <= pm0 + 3 && pm <= m; ++pm)
    for (int64_t pn = pn0; pn <= pn0 + 15 && pn <= n; ++pn) {
      const int64_t a = (m + pm - 1) / pm, b = (n + pn - 1) / pn;
      if (!fp64_tile_ok(dt, a, b)) continue;
      // (outputs in linear order measured 10% slower than a full tile)
      const double rate = a == T && b == T ? 1.0 : 1.12;
      const int64_t items = batch * ((m + a - 1) / a) * ((n + b - 1) / b);
      const double rounds = (double)((items + sms - 1) / sms);
      const double cost = rounds * ((double)((a * b + 31) / 32) * dfma * rate + 1500.0);
      if (cost < 0.97 * best) {
        best = cost;
        *tm = (int)a;
        *tn = (int)b;
      }
    }
  std::copy(key, key + 6, last.key);
  last.tm = *tm;
  last.tn = *tn;
}

int default_prog(bg_dtype dt, int64_t m, int64_t n, int64_t k, int64_t batch, int sms) {
  const int small = dt == BG_R64 ? PROG_R64_SMALL : PROG_C128_SMALL;
  if (prog_fits(small, dt, m, n, k) && small_pays(m, n, k, batch, sms)) return small;
  return dt == BG_R64 ? PROG_R64_TILE : PROG_C128_TILE;
}

template <bool CPLX, class Src, class Sched>
static void launch_typed(int ctas, int grid, cudaStream_t st, const Src& src, const Sched& sched,
                         int64_t n_items, const Scalars& s) {
  if (ctas == 1)
    fp64_persistent<1, CPLX, Src, Sched><<<grid, kFp64Threads, 0, st>>>(src, sched, n_items, s);
  else if (ctas == 3)
    fp64_persistent<3, CPLX, Src, Sched><<<grid, kFp64Threads, 0, st>>>(src, sched, n_items, s);
  else
    fp64_persistent<2, CPLX, Src, Sched><<<grid, kFp64Threads, 0, st>>>(src, sched, n_items, s);
}

template <class Src, class Sched>
static void launch_persistent(bg_dtype dt, int ctas, int sms, cudaStream_t st, const Src& src,
                              const Sched& sched, int64_t n_items, const Scalars& s) {
  const int grid = (int)std::min<int64_t>(n_items, (int64_t)sms * ctas);
  if (dt == BG_C128) launch_typed<true>(ctas, grid, st, src, sched, n_items, s);
  else launch_typed<false>(ctas, grid, st, src, sched, n_items, s);
}

cudaError_t launch_fp64_fixed(bg_dtype dt, int prog, int64_t m, int64_t n, int64_t k,
                              const Scalars& s, const void* A, int64_t lda, int64_t sA,
                              const void* B, int64_t ldb, int64_t sB, void* C, int64_t ldc,
                              int64_t sC, int64_t batch, int sms, cudaStream_t st) {
  FixedSrc src;
  src.A = static_cast<const double*>(A);
  src.B = static_cast<const double*>(B);
  src.C = static_cast<double*>(C);
  src.m = (int)m; src.n = (int)n; src.k = (int)k;
  src.lda = lda; src.ldb = ldb; src.ldc = ldc;
  src.sA = sA; src.sB = sB; src.sC = sC;
  src.esz = dt == BG_C128 ? 2 : 1;
  FixedSched sched;
  sched.prog = prog;
  prog_tile(prog, &sched.tm, &sched.tn);
  sched.batch = batch;
  int64_t n_items;
  if (sched.tm == 0) {
    sched.tiles_m = sched.tiles_n = 1;
    n_items = (batch + kSmallPerCta - 1) / kSmallPerCta;
  } else {
    if (prog != PROG_R64_DMMA)
      fp64_tile_split(dt, m, n, k, batch, sms, &sched.tm, &sched.tn);
    sched.tiles_m = (m + sched.tm - 1) / sched.tm;
    sched.tiles_n = (n + sched.tn - 1) / sched.tn;
    n_items = batch * sched.tiles_m * sched.tiles_n;
  }
  if (n_items <= 0) return cudaSuccess;
  const int T = dt == BG_C128 ? TC : TR;
  const int ctas = sched.tm == T && sched.tn == T ? 1
                   : sched.tm > 0 && sched.tm * sched.tn <= (dt == BG_C128 ? 2 : 4) * kFp64Threads
                       ? 3
                       : 2;
  launch_persistent(dt, ctas, sms, st, src, sched, n_items, s);
  count_launch();
  return cudaGetLastError();
}

cudaError_t launch_fp64_table(bg_dtype dt, const int64_t* d_table, const int32_t* d_order,
                              const WorkItem* d_items, int64_t n_items, const void* A,
                              const void* B, void* C, const Scalars& s, int ctas, int sms,
                              cudaStream_t st, bool herm) {
  if (n_items <= 0) return cudaSuccess;
  TableSrc src;
  src.herm = herm ? 1 : 0;
  src.table = d_table;
  src.order = d_order;
  src.A = static_cast<const double*>(A);
  src.B = static_cast<const double*>(B);
  src.C = static_cast<double*>(C);
  src.esz = dt == BG_C128 ? 2 : 1;
  TableSched sched{d_items};
  launch_persistent(dt, ctas, sms, st, src, sched, n_items, s);
  count_launch();
  return cudaGetLastError();
}

cudaError_t launch_fp64_chain(bg_dtype dt, const int64_t* d_wn, const int64_t* d_woff,
                              const int64_t* d_pool_off, const int64_t* d_pool_n,
                              int32_t pool_count, const int32_t* d_order,
                              const int32_t* d_idx_row, const WorkItem* d_items, int64_t n_items,
                              const void* U, const void* Cin, void* Cout, int ctas, int sms,
                              cudaStream_t st) {
  if (n_items <= 0) return cudaSuccess;
  ChainSrc src;
  src.wn = d_wn;
  src.woff = d_woff;
  src.pool_off = d_pool_off;
  src.pool_n = d_pool_n;
  src.pool_count = pool_count;
  src.order = d_order;
  src.idx = d_idx_row;
  src.U = static_cast<const double*>(U);
  src.Cin = static_cast<const double*>(Cin);
  src.Cout = static_cast<double*>(Cout);
  src.esz = dt == BG_C128 ? 2 : 1;
  Scalars s;
  s.alpha_re = 1.0; s.alpha_im = 0.0; s.beta_re = 0.0; s.beta_im = 0.0;
  s.alpha_zero = 0; s.beta_zero = 1;
  TableSched sched{d_items};
  launch_persistent(dt, ctas, sms, st, src, sched, n_items, s);
  count_launch();
  return cudaGetLastError();
}

}  // namespace bg
