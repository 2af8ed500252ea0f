// SpMV kernels y = alpha*A*x + beta*y for the formats the paper lists
// (Section 1: Coo, Csr, Ell, Hybrid) and the internal dispatch used by the
// C ABI and the Krylov solvers.  All kernels are deterministic: a fixed
// launch shape and fixed summation order give bit-identical results on
// every call, with no floating-point atomics.
#pragma once

#include "common.cuh"

namespace gko {

// Fused dot epilogue: result[0] = sum_i w[i] * y[i] and result[1] =
// sum_i y[i]^2, in FP64 over the rows the SpMV writes.  Blocks store partial
// sums; the last block to arrive (integer ticket) adds them in index order,
// so the values are deterministic.
struct DotSpec {
  const void* w = nullptr;  // same element type as y
  double* partials = nullptr;  // 2 * kDotSlots doubles
  unsigned* counter = nullptr;  // zero on entry; the last block resets it
  double* result = nullptr;     // 2 doubles
  int want_yy = 1;              // 0: skip y.y (result[1] = 0)
};
constexpr int kDotSlots = 4096;  // blocks a fused reduction may use

// Scratch bytes one SpMV of A needs (long-row partials or COO carries).
size_t spmv_scratch_bytes(const gko_matrix_s* A);
// Whether spmv_run can fuse the dot epilogue for this format.
bool spmv_fuses_dot(const gko_matrix_s* A);

// x, y: device vectors (double for F64 matrices, float otherwise).
// gate (nullable): two device ints; every kernel returns at once when either
// is nonzero (used by the solvers to turn finished iterations into no-ops).
int spmv_run(const gko_matrix_s* A, const void* x, void* y, double alpha, double beta, cudaStream_t s,
             void* scratch, const DotSpec* dot, const int* gate = nullptr);

// Per value type entry points (one translation unit each).
int spmv_run_f64(const gko_matrix_s* A, const double* x, double* y, double alpha, double beta, cudaStream_t s,
                 void* scratch, const DotSpec* dot, const int* gate);
int spmv_run_f32(const gko_matrix_s* A, const float* x, float* y, double alpha, double beta, cudaStream_t s,
                 void* scratch, const DotSpec* dot, const int* gate);
int spmv_run_bf16(const gko_matrix_s* A, const float* x, float* y, double alpha, double beta, cudaStream_t s,
                  void* scratch, const DotSpec* dot, const int* gate);

// Jacobi preconditioner: d = inverse diagonal of the FP64 matrix A (any
// format; zero diagonal -> 1), and its FP32 rounding for inner solves.
int jacobi_inverse(const gko_matrix_s* A, double* d, cudaStream_t s);
int narrow_to_f32(const double* d, float* f, int64_t n, cudaStream_t s);

constexpr int kCooThreads = 128;
constexpr int kCooItems = 8;
constexpr int kCooTile = kCooThreads * kCooItems;

// Row-aligned tiles of W nonzeros (a multiple of 8, for 16-byte loads).  A
// block's window is the kCooTile entries from t W on; W leaves room for the
// rest of the tile's last row where rows are short, so the window nearly
// always holds the whole tile.
// Used where the launch and the workspace that go away (6-8 us) are worth more
// than the overlapping windows and the rest of a row behind the window, which
// one block adds.  Both grow with the nonzeros, the latter also with the
// longest row L (at most kTileRowMax), in FP64 twice as fast as in FP32.
// Speedup of COO over the kernels with carries, FP64 / FP32, rows of L entries
// next to the diagonal:
//   L = 27    4 M 1.28 / 1.27   8 M 1.16 / 1.19   16 M 1.05 / 1.02   40 M 1.04 / 0.91
//   L = 96    4 M 1.20 / 1.31   6 M 1.15 / 1.16    8 M 1.13 / 1.15
//   L = 200   1 M 1.24 / 1.32   2 M 1.09 / 1.31    4 M 1.00 / 1.22    8 M 0.93 / 1.15
//   L = 500   1 M 1.18 / 1.24   2 M 1.10 / 1.18    4 M 0.92 / 1.23    8 M 0.85 / 1.10
//   L = 1800  1 M 1.16 / 1.40   2 M 1.04 / 1.18    4 M 0.88 / 1.13    8 M 0.80 / 0.97
// Random columns, rows of 1..L: FP64 L = 64 4 M 1.09, 8 M 0.95; L = 500 2 M 1.04,
// 4 M 0.98; FP32 L = 300 8 M 1.05; L = 900 3 M 1.10, 8 M 1.06.  CSR gains 3-10%
// less than COO.
constexpr int32_t kTileRowMax = 2048;
inline bool tiles_worth(int64_t nnz, int32_t max_len, gko_dtype dtype) {
  if (nnz == 0 || max_len > kTileRowMax) return false;
  if (dtype == GKO_F64) {
    if (max_len <= 48) return nnz <= 1 << 23;
    return nnz <= 3 << 19 || (nnz <= 3 << 21 && nnz * max_len <= 9ll << 26);
  }
  return nnz <= 1 << 21 || (nnz <= 1 << 23 && nnz * max_len <= 3ll << 30);
}
// COO handles and hybrid tails carry the tile starts where any type wants them.
inline bool coo_tiles(const gko_matrix_s* A) {
  return A->plan.tiles > 0 && tiles_worth(A->coo_nnz, A->plan.tile_len, A->dtype);
}
inline int32_t tile_width_for(int32_t max_len) {
  const int32_t room = max_len < 64 ? max_len : 64;
  return (kCooTile - room) / 8 * 8;
}

}  // namespace gko
