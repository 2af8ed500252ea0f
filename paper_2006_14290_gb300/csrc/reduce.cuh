// Deterministic block and grid reductions (FP64) shared by the SpMV,
// BLAS-1 and solver kernels.  No floating-point atomics: blocks publish
// partial sums and the last block to take an integer ticket adds them in a
// fixed order, then runs an optional scalar operation on the totals.
#pragma once

#include "fx.cuh"
#include "spmv.cuh"

namespace gko {

// Sum of NV values over a block; the totals are valid in thread 0.  Added as
// fixed-point integers (fx.cuh), the warps' sums by warp k for value k: the
// FP64 tree (five shuffles, then eight additions by thread 0) held the SM's
// one FP64 pipe for 48 warp instructions, a fifth of a Gram-Schmidt block's
// work, and took 1,100 cycles where this takes 700.
template <int THREADS, int NV>
__device__ __forceinline__ void block_sum_n(double (&v)[NV]) {
  constexpr int W = THREADS / kWarp;
  static_assert(W <= 32 && NV <= W, "one warp adds one value");
  __shared__ double red[NV][W];  // doubles: csr_rowblock_kernel's blocks per SM hang on these bytes
  const int w = threadIdx.x >> 5, lane = threadIdx.x & 31;
#pragma unroll
  for (int k = 0; k < NV; ++k) {
    const Fx f = warp_fx_sum(fx_of(v[k]));
    if (lane == 0) red[k][w] = fx_double(f);
  }
  __syncthreads();
  if (w < NV) {
    const Fx f = warp_fx_sum(lane < W ? fx_of(red[w][lane]) : Fx{0, 1});
    if (lane == 0) red[w][0] = fx_double(f);
  }
  __syncthreads();
  if (threadIdx.x == 0) {
#pragma unroll
    for (int k = 0; k < NV; ++k) v[k] = red[k][0];
  }
  __syncthreads();
}

// The same sums as an FP64 tree, for the update of large unpreconditioned FP64
// CG (kTreeRows in krylov.cu, with both sides' times): a kernel alone takes
// the same time with either (128^3: 23.7 us with block_sum_n, 24.2 here), but
// the iteration is 3-6% shorter with this one.
template <int THREADS, int NV>
__device__ __forceinline__ void block_tree_n(double (&v)[NV]) {
  __shared__ double red[NV][THREADS / kWarp];
  const int w = threadIdx.x >> 5;
#pragma unroll
  for (int k = 0; k < NV; ++k) {
    v[k] = subwarp_sum<32>(v[k], 0xffffffffu);
    if ((threadIdx.x & 31) == 0) red[k][w] = v[k];
  }
  __syncthreads();
  if (threadIdx.x == 0) {
#pragma unroll
    for (int k = 0; k < NV; ++k) {
      double s = 0.0;
#pragma unroll
      for (int i = 0; i < THREADS / kWarp; ++i) s += red[k][i];
      v[k] = s;
    }
  }
  __syncthreads();
}

template <int THREADS>
__device__ __forceinline__ double block_sum(double v) {
  double a[1] = {v};
  block_sum_n<THREADS, 1>(a);
  return a[0];
}

struct NoOp {
  template <int NV>
  __device__ void operator()(const double (&)[NV]) const {}
};

// Store this block's NV partials in `slot`; the block that takes the last of
// `expected` tickets adds all partials in a fixed order and calls op(totals)
// from its thread 0, then re-arms the counter.
template <int THREADS, int NV, bool TREE = false, typename Op>
__device__ void grid_reduce(double (&v)[NV], double* partials, unsigned* counter, int slot, int expected, Op op) {
  __shared__ int is_last;
  auto block = [](double (&u)[NV]) {
    if constexpr (TREE) block_tree_n<THREADS, NV>(u);
    else block_sum_n<THREADS, NV>(u);
  };
  block(v);
  if (threadIdx.x == 0) {
#pragma unroll
    for (int k = 0; k < NV; ++k) partials[(int64_t)slot * NV + k] = v[k];
    __threadfence();
    const unsigned t = atomicAdd(counter, 1u);
    is_last = (t == (unsigned)expected - 1u);
  }
  __syncthreads();
  if (!is_last) return;
  __threadfence();
  double acc[NV];
#pragma unroll
  for (int k = 0; k < NV; ++k) acc[k] = 0.0;
#pragma unroll 4
  for (int i = threadIdx.x; i < expected; i += THREADS)
#pragma unroll
    for (int k = 0; k < NV; ++k) acc[k] += __ldcg(partials + (int64_t)i * NV + k);
  block(acc);
  if (threadIdx.x == 0) {
    op(acc);
    *counter = 0u;
  }
}

struct StoreOp2 {
  double* result;
  __device__ void operator()(const double (&t)[2]) const {
    result[0] = t[0];
    result[1] = t[1];
  }
};

// Fused dot epilogue of the SpMV kernels: result[0] = w . y, result[1] = y . y.
template <int THREADS>
__device__ __forceinline__ void dot_epilogue2(double wy, double yy, const DotSpec& d, int slot, int expected) {
  double v[2] = {wy, yy};
  grid_reduce<THREADS, 2>(v, d.partials, d.counter, slot, expected, StoreOp2{d.result});
}

// A kernel is gated off when either gate word is nonzero (solver state:
// converged/stopped, or a phase that skips this product).
__device__ __forceinline__ bool gated(const int* g) {
  if (!g) return false;
  return (*(volatile const int*)g | *((volatile const int*)g + 1)) != 0;
}

}  // namespace gko
