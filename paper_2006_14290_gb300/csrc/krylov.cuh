// Solver state and host-side specifications shared by the Krylov solvers'
// translation units: the multi-kernel solvers (krylov.cu) and the
// single-launch solvers of small systems (persist.cuh, persist_*.cu).
#pragma once

#include <math.h>

#include "blas1.cuh"
#include "reduce.cuh"
#include "spmv.cuh"

namespace gko {

enum : int { kRun = 0, kConverged = 1, kBreakdown = 2, kNotConverged = 3, kCheck = 4 };

// Device-resident solver state.  The first three ints are gate words: an
// SpMV gated on &done runs unless done|zero; gated on &phase it also stops
// when `phase` is set (BiCGSTAB half step converged / GMRES cycle ended).
struct Ctl {
  int phase;
  int done;
  int zero;
  int status;
  int iter;
  int maxit;
  int replace;
  int check_true;
  int cycles;
  int k;         // GMRES: columns of the finished cycle
  int noreorth;  // GMRES: this step skips the second Gram-Schmidt pass
  int pad;
  double nb, tol_abs;
  double rho, rho_new, alpha, beta, omega;
  double red[4];  // fused SpMV dots: red[0] = w.y, red[1] = y.y
  double rr;
  // reliable updates (mixed precision): an update is due when the recurrence
  // residual drops below delta times maxrr, its largest norm since the last
  // update (delta = 0: only at convergence); half: the last check came from
  // BiCGSTAB's half step
  double maxrr, delta;
  int half;
  int gave_up;  // single-launch solves: a wait of some block timed out
};

__device__ __forceinline__ double wd(double v) { return v; }
__device__ __forceinline__ double wd(float v) { return widen(v); }

// What a reliable-update solve needs beyond the recurrences' operator.
struct RelSpec {
  const gko_matrix_s* A64;  // FP64 matrix for the replaced residuals
  const double* b64;        // right-hand side
  double* x64;              // FP64 solution (x0 on entry)
  double* q64;              // n doubles of workspace
  void* scratch;            // SpMV scratch of A64
  double delta;
};

// Bump allocator over one pool allocation.
struct Carve {
  char* base;
  size_t off = 0;
  template <typename T>
  T* take(size_t count) {
    off = (off + 255) / 256 * 256;
    T* p = reinterpret_cast<T*>(base + off);
    off += sizeof(T) * count + 64;
    return p;
  }
};

// Pinned host mirror of Ctl for polling.
inline Ctl* host_ctl() {
  thread_local Ctl* h = nullptr;
  if (!h) {
    if (cudaMallocHost((void**)&h, sizeof(Ctl)) != cudaSuccess) {
      cudaGetLastError();
      static thread_local Ctl fallback;
      h = &fallback;
    }
  }
  return h;
}

inline int read_ctl(const Ctl* d, Ctl* h, cudaStream_t s) {
  GKO_TRY_CUDA(cudaMemcpyAsync(h, d, sizeof(Ctl), cudaMemcpyDeviceToHost, s));
  GKO_TRY_CUDA(cudaStreamSynchronize(s));
  return GKO_OK;
}

struct SolveSpec {
  int solver;  // 0 CG, 1 BiCGSTAB, 2 GMRES
  double rel_tol;
  int maxit;
  int restart;
  int check_true;
  int check_every;
  const void* minv = nullptr;  // Jacobi inverse diagonal (vector of T), or none
  const RelSpec* rel = nullptr;  // reliable updates (FP32 recurrences only)
  const void* bj = nullptr;  // block-Jacobi inverse blocks (n x bs, of T), or none
  int bs = 0;                  // block-Jacobi block size
};

struct SolveOut {
  int status;
  int iterations;
  int cycles;
  // set by the single-launch FP64 solves: ||b - A x|| / ||b|| of the x they
  // return (no separate residual pass needed)
  bool have_residual = false;
  double rel_residual = 0.0;
};

// Largest system the single-launch solvers take (rows); larger ones run the
// multi-kernel solvers.
constexpr int64_t kSmallRows = 1 << 18;

// One CG, BiCGSTAB or GMRES solve in one launch, a cluster or a cooperative grid
// (persist.cuh, persist_gmres.cuh), or GKO_NOT_SUPPORTED when it does not apply (the caller then takes the
// multi-kernel solve).  x: T vector (double for an FP64 matrix, else float).
int persist_solve(const gko_matrix_s* A, const double* b, void* x, bool x_zero, const SolveSpec& sp, cudaStream_t s,
                  SolveOut* out);

}  // namespace gko
