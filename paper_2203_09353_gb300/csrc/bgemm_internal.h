// Internal declarations shared by the library's translation units.
// Nothing here is part of the public ABI (include/bgemm.h).
#pragma once

#include <cuda_runtime.h>
#include <stdint.h>

#include <string>

#include "bgemm.h"

namespace bg {

// ---- work description --------------------------------------------------------

// Tile programs of the FP64 path. A work item names one program and the part
// of the batch it covers.
enum Prog : int16_t {
  PROG_R64_SMALL = 0,   // a warp per instance, 8 per CTA
  PROG_R64_TILE = 1,    // 64x64 output tile, DFMA, 4x4 outputs per thread
  PROG_R64_DMMA = 2,    // 64x64 output tile, FP64 tensor-core mma.sync m8n8k4
  PROG_C128_SMALL = 3,  // one warp per complex instance
  PROG_C128_TILE = 4,   // 32x32 complex output tile, DFMA, 2x2 per thread
  PROG_COUNT = 5
};

// One unit of work of the persistent FP64 kernel (16 bytes).
//  - tile programs: `inst` = instance id, (r0, c0) = first row/col of the tile,
//    `count` = its rows and columns (tile_extent)
//  - small programs: `inst` = first position in the class-ordered instance
//    list, `count` = number of consecutive instances (<= 8), r0 = c0 = 0
struct WorkItem {
  int32_t inst;
  int16_t prog;
  int16_t count;
  int32_t r0;
  int32_t c0;
};
static_assert(sizeof(WorkItem) == 16, "WorkItem must stay 16 bytes");

// Rows and columns (1..64 each) of a tile in WorkItem.count; 0 and 1 mean the
// program's full tile.
__host__ __device__ inline int16_t tile_extent(int tm, int tn) { return (int16_t)(2 + (tm - 1) * 64 + (tn - 1)); }
__host__ __device__ inline void tile_extent_of(int count, int full, int* tm, int* tn) {
  *tm = *tn = full;
  if (count >= 2) {
    *tm = (count - 2) / 64 + 1;
    *tn = (count - 2) % 64 + 1;
  }
}

constexpr int kSmallPerCta = 8;   // warps (instances) per CTA in the small programs
constexpr int kFp64Threads = 256;

// Outputs per thread of the program that runs a tile with `out` outputs inside
// its instance: the smallest that holds them all. The largest is the
// register-blocked one of the full tile; it guards its edges, so it also runs
// what an instance leaves of a full tile (127 rows are 64 + 63).
__host__ __device__ constexpr int tile_program_r64(int out) {
  return out > 8 * kFp64Threads ? 16 : out > 4 * kFp64Threads ? 8 : out > 2 * kFp64Threads ? 4 : 2;
}
__host__ __device__ constexpr int tile_program_c128(int out) {
  return out > 2 * kFp64Threads ? 4 : out > kFp64Threads ? 2 : 1;
}

struct Scalars {
  double alpha_re, alpha_im, beta_re, beta_im;
  int alpha_zero, beta_zero;
};

// Program of a fixed-size batch (FP64 path).
int default_prog(bg_dtype dt, int64_t m, int64_t n, int64_t k, int64_t batch, int sms);
// Output-tile extent of a tile program (rows, cols); small programs return 0.
void prog_tile(int prog, int* tm, int* tn);
bool prog_is_small(int prog);
// Whether a tile of tm x tn outputs can run: the full tile, or at most as many
// outputs as the threads hold in linear order.
bool fp64_tile_ok(bg_dtype dt, int64_t tm, int64_t tn);
// Rows and columns of the tiles that `batch` instances of one shape are cut
// into (at most 64 x 64 real, 32 x 32 complex, evenly split), so that a batch
// smaller than the chip still spreads over its SMs.
void fp64_tile_split(bg_dtype dt, int64_t m, int64_t n, int64_t k, int64_t batch, int sms, int* tm,
                     int* tn);
bool prog_fits(int prog, bg_dtype dt, int64_t m, int64_t n, int64_t k);
// Whether a batch of `instances` that the small program fits is to run on it.
bool small_pays(int64_t m, int64_t n, int64_t k, int64_t instances, int sms);

// ---- FP64 launchers (fp64.cu) ---------------------------------------------------

cudaError_t launch_fp64_fixed(bg_dtype dt, int prog, int64_t m, int64_t n, int64_t k,
                              const Scalars& s, const void* A, int64_t lda, int64_t sA,
                              const void* B, int64_t ldb, int64_t sB, void* C, int64_t ldc,
                              int64_t sC, int64_t batch, int sms, cudaStream_t st);

// ctas: CTAs per SM: 1 (most work in full tiles), 2, or 3 (no small programs,
// tiles of at most 1024 real or 512 complex outputs).
// herm: the plan's instances are Hermitian rank-k updates (B = A^H, lower
// triangle stored).
cudaError_t launch_fp64_table(bg_dtype dt, const int64_t* d_table, const int32_t* d_order,
                              const WorkItem* d_items, int64_t n_items, const void* A,
                              const void* B, void* C, const Scalars& s, int ctas, int sms,
                              cudaStream_t st, bool herm = false);

cudaError_t launch_fp64_chain(bg_dtype dt, const int64_t* d_wn, const int64_t* d_woff,
                              const int64_t* d_pool_off, const int64_t* d_pool_n,
                              int32_t pool_count, const int32_t* d_order,
                              const int32_t* d_idx_row, const WorkItem* d_items, int64_t n_items,
                              const void* U, const void* Cin, void* Cout, int ctas, int sms,
                              cudaStream_t st);

// ---- split-BF16 path (split.cu) ---------------------------------------------------

struct SplitParams;  // defined in split.cu

// ---- measurement and diagnostics (util.cu) ------------------------------------------

cudaError_t launch_rel_err(bg_dtype dt, int64_t count, const int64_t* d_table, const void* A,
                           const void* B, const void* Ct, const void* Cr, double* out,
                           cudaStream_t st);
cudaError_t launch_drift(bg_dtype dt, int64_t count, const int64_t* d_n, const int64_t* d_off,
                         const void* C, double* out, cudaStream_t st);
cudaError_t launch_bounded_wait(int64_t spin_limit, int* d_err, cudaStream_t st);
cudaError_t run_fp64_peak_probe(int mma_kind, int sms, double* tflops, cudaStream_t st);
// Local two-spin gate on a batch of complex128 state vectors (gate.cu), from
// src to dst (the same array for the gate in place).
cudaError_t launch_local_gate(int64_t walkers, int spins, const int32_t* sites, const void* gates,
                              const void* src, int64_t src_stride, void* dst, int64_t dst_stride,
                              int* d_err, int sms, cudaStream_t st);

// Device error word layout: [0] = first error code, [1] = location id,
// [2] = detail, [3] = count of events.
enum DevErrLoc : int {
  ERRLOC_NONE = 0,
  ERRLOC_TEST_WAIT = 1,
  ERRLOC_SPLIT_FULL_BARRIER = 2,
  ERRLOC_SPLIT_EMPTY_BARRIER = 3,
  ERRLOC_SPLIT_ACC_FULL = 4,
  ERRLOC_SPLIT_ACC_EMPTY = 5,
  ERRLOC_SPLIT_TMEM_ALLOC = 6,
  ERRLOC_CHAIN_INDEX = 7,
  ERRLOC_GATE_SITE = 8
};

// Host bookkeeping.
void count_launch(int n = 1);

// ---- static scratch (noalloc.cu) ----
// Capacity of the per-device static scratch array, in bytes.
size_t static_scratch_capacity();
// Address of the static scratch on the current device (looked up once per device).
bg_status static_scratch(void** out, size_t* bytes, std::string* err);

// Householder reduction of each walker's Hermitian positive semidefinite
// n x n Gram matrix (lower triangle, overwritten) to a real tridiagonal matrix
// (tridiag.cu). The shape is chosen once, for the current device, and kept with
// the panel memory that it needs: the device's answer to how many clusters fit
// may differ from one query to the next. panel: walkers x TriShape::panel bytes
// of device memory, or null where that is 0.
struct TriShape {
  int cl = 1;        // CTAs per walker
  int warps = 0;     // warps per CTA
  int own = 0;       // rows a CTA owns at most
  bool vws = true;   // the panel's own rows are in shared memory
  size_t smem = 0;   // dynamic shared memory of a CTA
  size_t panel = 0;  // bytes of panel vectors per walker in device memory
};
// (also sets the kernels' shared-memory limits on the current device)
cudaError_t tri_shape(int64_t walkers, int n, int sms, TriShape* out);
cudaError_t launch_tridiag(double2* gram, int64_t walkers, int n, const TriShape& shape,
                           void* panel, double* d, double* e, cudaStream_t st);

// Eigenvalues of the tridiagonal matrices and the entropies (entropy.cu).
// lam: workspace of walkers x n doubles; eigs: optional device [walkers][n],
// ascending.
cudaError_t launch_entropy_bisect(const double* d, const double* e, int64_t walkers, int n,
                                  double* lam, double* entropy, double* eigs, int sms,
                                  cudaStream_t st);

// Metropolis decision per walker and copy of the accepted proposals over the
// current states (anneal.cu). prop / cur may be null when amps == 0.
cudaError_t launch_metropolis(int64_t walkers, double T, int direction, const double* u,
                              const double* e_new, double* e_cur, int32_t* acc,
                              const void* prop, int64_t pstride, void* cur, int64_t cstride,
                              int64_t amps, int sms, cudaStream_t st);

}  // namespace bg
