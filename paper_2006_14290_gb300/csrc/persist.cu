// Host side of the single-launch solvers (persist.cuh): which systems they
// take, the launch shape and the workspace.
#include "persist_gmres.cuh"

namespace gko {

template <>
PkKernel<double, double> pk_cg<double, double>(int, bool);
template <>
PkKernel<float, float> pk_cg<float, float>(int, bool);
template <>
PkKernel<float, __nv_bfloat16> pk_cg<float, __nv_bfloat16>(int, bool);
template <>
PkKernel<double, double> pk_bicg<double, double>(int, bool);
template <>
PkKernel<float, float> pk_bicg<float, float>(int, bool);
template <>
PkKernel<float, __nv_bfloat16> pk_bicg<float, __nv_bfloat16>(int, bool);
template <>
PkGmresKernel<double, double> pk_gmres<double, double>(int, bool);
template <>
PkGmresKernel<float, float> pk_gmres<float, float>(int, bool);
template <>
PkGmresKernel<float, __nv_bfloat16> pk_gmres<float, __nv_bfloat16>(int, bool);

namespace {

// A matrix's column and value arrays in the formats served here.
const Buf& cols_of(const gko_matrix_s* A) {
  return A->fmt == GKO_CSR ? A->col : A->fmt == GKO_ELL ? A->ell_col : A->sellp_col;
}
const Buf& vals_of(const gko_matrix_s* A) {
  return A->fmt == GKO_CSR ? A->val : A->fmt == GKO_ELL ? A->ell_val : A->sellp_val;
}

// Lines between these kernels and the multi-kernel solve, by the longest row K.
// Figures: speedup over the multi-kernel solve, band matrix / random columns,
// FP64, CSR unless ELL is said (whose multi-kernel product is the faster one).
//
// A published vector costs an exchange, recomputing it (kPkFly) one gather more
// per entry in CG, two and one in BiCGSTAB's products.  CG, 14,000 rows, kPkFly /
// published: K = 7 2.9 / 2.5, 17 2.7 / 2.6, 65 1.7 / 2.3; random columns, K = 65 1.4 / 1.9.
// BiCGSTAB, 25,000 rows: K = 7 2.6 / 2.5, 17 2.2 / 2.7, 65 1.4 / 2.3; random 0.9 / 1.7.
constexpr int64_t kPkFlyRow = 16;
// In a cluster 16 SMs read each other's shared memory, fast from neighbours, not
// at random: CG, 4,096 rows, cluster / published, K = 17 3.2 / 2.4, 27 3.0 / 2.2, 49 2.4 / 1.9;
// random 1.5 / 2.3, 1.0 / 2.1, 0.6 / 1.8.  More entries than this take the grid; in
// FP32 CG, whose grid shapes are as fast there, fewer (the second line).
constexpr int64_t kPkClusterEntries = 7 << 14, kPkClusterEntriesCg32 = 1 << 16;
// Entries that do not fit in shared memory are read from the matrix, a row to a
// lane, which long rows and few SMs make slow:
//   a row a thread:  CG 38,000 rows K = 129 2.0 / 1.5, 257 1.1 / 1.2   25,000 257 1.7 / 1.3
//                    14,000 201 1.3 / 0.9, 401 1.2 / 0.9   9,700 401 0.6 / 0.6; ELL 1.6 / 1.1
//   two rows:        CG 79,000 K = 97 1.3 / 1.1   120,000 97 1.3 / 1.4; ELL 79,000 65 1.3 / 0.95, 129 0.8 / 0.8
//                    ELL 120,000 65 1.9 / 1.4, 97 1.3 / 1.1
//                    BiCGSTAB 79,000 97 1.1 / 1.0, 129 0.9 / 1.0
//   four rows:       CG 262,144 K = 33 1.8 / 1.7, 49 1.0 / 1.3; ELL 27 1.5 / 1.3, 49 0.9 / 0.9
//                    BiCGSTAB 262,144 33 1.4 / 1.5, 49 0.8 / 1.2; ELL 27 1.2 / 1.2, 33 0.8 / 0.9
// FP32: 1.2-3 at all of these but ELL, two rows, K = 129 0.9.  GMRES (few
// products a step): FP64 CSR 25,000 257 1.6 / 1.4, 5,000 321 1.0, 1,000 401 0.9; the
// others win at every K measured, to 999.
bool pk_unstaged_worth(int solver, bool csr, bool f64, int rows, int64_t n, int64_t K) {
  const bool bicg = solver == 1;
  if (solver == 2) return !csr || !f64 || K <= 320;
  if (rows == 1) return !csr || !f64 || K <= (n >= 16384 ? 320 : n > 9728 ? 160 : 0);
  if (rows == 2) return K <= (csr ? (bicg && f64 ? 112 : 160) : f64 && n < 98304 ? 64 : 96);
  return K <= (csr ? (bicg && f64 ? 40 : 72) : bicg && f64 ? 32 : 40);
}

// What every kernel is given: the matrix, right-hand side, x and options.
template <typename T, typename VT>
PkArgs<T, VT> args_of(const gko_matrix_s* A, const double* b, T* x, bool x_zero, const SolveSpec& sp, size_t K) {
  PkArgs<T, VT> a{};
  a.n = (int32_t)A->n_rows;
  a.K = (int32_t)K;
  a.fmt = A->fmt;
  a.rp = A->fmt == GKO_CSR ? ptr<int32_t>(A->row_ptr) : A->fmt == GKO_SELLP ? ptr<int32_t>(A->sellp_sets) : nullptr;
  a.col = ptr<int32_t>(cols_of(A));
  a.val = ptr<VT>(vals_of(A));
  a.stride = A->stride;
  a.slice = A->slice;
  a.b = b;
  a.x = x;
  a.d = static_cast<const T*>(sp.minv);
  a.bj = static_cast<const T*>(sp.bj);
  a.bs = sp.bs;
  a.rel_tol = sp.rel_tol;
  a.maxit = sp.maxit;
  a.check_true = sp.check_true;
  a.x_zero = x_zero ? 1 : 0;
  if (sp.rel) {
    a.val64 = ptr<double>(vals_of(sp.rel->A64));
    a.b64 = sp.rel->b64;
    a.x64 = sp.rel->x64;
    a.delta = sp.rel->delta;
  }
  a.err = device_error_word();
  return a;
}

// Waits for the solve and reads its result.
template <typename T>
int finish(const Ctl* c, cudaStream_t s, SolveOut* out) {
  Ctl* hc = host_ctl();
  GKO_TRY(read_ctl(c, hc, s));
  if (hc->gave_up) return fail(GKO_TIMEOUT, "single-launch solve: a grid reduction's wait timed out");
  out->status = hc->status;
  out->iterations = hc->iter;
  out->cycles = hc->cycles;
  if (sizeof(T) == 8) {
    out->have_residual = true;
    out->rel_residual = hc->nb == 0.0 ? 0.0 : sqrt(hc->rr) / hc->nb;
  }
  return GKO_OK;
}

// Static shared memory of a CG or BiCGSTAB kernel, at most.
constexpr size_t kPkStaticMax = sizeof(PkShared<512, kPkCluster>) + 1024;

template <typename T, typename VT>
int launch(const gko_matrix_s* A, const double* b, T* x, bool x_zero, const SolveSpec& sp, cudaStream_t s, SolveOut* out,
           int shape, bool staged, int G, size_t K, size_t smem) {
  const int64_t n = A->n_rows;
  const PkShape sh = kPkShapes[shape];
  const bool cluster = sh.mode == kPkCluster;
  const PkKernel<T, VT> kern = sp.solver == 0 ? pk_cg<T, VT>(shape, staged) : pk_bicg<T, VT>(shape, staged);
  if (!kern) return GKO_NOT_SUPPORTED;
  // The default limit of 48 KB holds static and dynamic shared memory together.
  // Always the largest request, so that concurrent solves (serving threads)
  // never lower each other's limit.
  if (smem > 48 * 1024 - kPkStaticMax)
    GKO_TRY_CUDA(cudaFuncSetAttribute(kern, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)kPkSmemMax));
  cudaLaunchConfig_t cfg = {};
  cfg.gridDim = dim3((unsigned)G);
  cfg.blockDim = dim3((unsigned)sh.nt);
  cfg.dynamicSmemBytes = smem;
  cfg.stream = s;
  cudaLaunchAttribute at[1];
  if (cluster) {
    if (G > 8) GKO_TRY_CUDA(cudaFuncSetAttribute(kern, cudaFuncAttributeNonPortableClusterSizeAllowed, 1));
    at[0].id = cudaLaunchAttributeClusterDimension;
    at[0].val.clusterDim.x = (unsigned)G;
    at[0].val.clusterDim.y = at[0].val.clusterDim.z = 1;
  } else {
    at[0].id = cudaLaunchAttributeCooperative;
    at[0].val.cooperative = 1;
  }
  cfg.attrs = at;
  cfg.numAttrs = 1;
  if (cluster) {
    int fit = 0;
    if (cudaOccupancyMaxActiveClusters(&fit, kern, &cfg) != cudaSuccess || fit < 1) {
      cudaGetLastError();
      return GKO_NOT_SUPPORTED;
    }
  }

  const int nvec = cluster ? 0 : sp.solver == 0 ? (sh.mode == kPkFly ? 3 : 1) : (sh.mode == kPkFly ? 5 : 2);
  const size_t slot_bytes = cluster ? 0 : sizeof(ulonglong2) * 2 * kPkMaxBlocks * kPkSlot;
  Scratch mem;
  GKO_TRY(mem.get(sizeof(Ctl) + slot_bytes + 1024 + (size_t)nvec * (sizeof(T) * (size_t)n + 320), s));
  Carve cv{static_cast<char*>(mem.data())};
  PkArgs<T, VT> a = args_of<T, VT>(A, b, x, x_zero, sp, K);
  a.c = cv.take<Ctl>(1);
  if (!cluster) a.slots = cv.take<ulonglong2>(2 * kPkMaxBlocks * kPkSlot);
  for (int k = 0; k < nvec; ++k) a.vec[k] = cv.take<T>((size_t)n);
  if (!cluster)  // the state and the slots behind it
    GKO_TRY_CUDA(cudaMemsetAsync(a.c, 0, (size_t)((char*)a.slots - (char*)a.c) + slot_bytes, s));
  const cudaError_t e = cudaLaunchKernelEx(&cfg, kern, a);
  if (e == cudaErrorCooperativeLaunchTooLarge) {  // the blocks cannot all be resident
    cudaGetLastError();
    return GKO_NOT_SUPPORTED;
  }
  GKO_TRY_CUDA(e);
  return finish<T>(a.c, s, out);
}

template <typename T, typename VT>
int run(const gko_matrix_s* A, const double* b, T* x, bool x_zero, const SolveSpec& sp, cudaStream_t s,
        SolveOut* out) {
  const int64_t n = A->n_rows;
  const size_t K = (size_t)std::max<int32_t>(1, A->fmt == GKO_CSR ? A->plan.max_len : A->K);
  // the first shape that covers n and whose entries fit in shared memory;
  // where none does, the first that reads its entries from the matrix
  auto smem_of = [&](const PkShape& h, bool st) {
    const size_t rb = (size_t)h.nt * h.rpt;
    return (st ? K * rb * (sizeof(VT) + sizeof(int32_t)) : 0) +
           ((h.mode == kPkCluster ? kPkClusterVecs : 0) + (sp.bj ? 1 : 0)) * rb * sizeof(T);
  };
  auto blocks_of = [&](const PkShape& h) { return (n + h.nt * h.rpt - 1) / (h.nt * h.rpt); };
  auto covers = [&](const PkShape& h) {
    return blocks_of(h) <= (h.mode == kPkCluster ? kPkCluster16 : std::min(sm_count(), kPkMaxBlocks));
  };
  const bool f64 = sizeof(T) == 8, bicg = sp.solver == 1;
  const bool twins = (bicg && sp.bj) || (int64_t)K > kPkFlyRow;
  auto worth = [&](const PkShape& h, bool staged) {
    if (h.mode == kPkCluster) return n * (int64_t)K <= (!bicg && !f64 ? kPkClusterEntriesCg32 : kPkClusterEntries);
    return staged || pk_unstaged_worth(sp.solver, A->fmt == GKO_CSR, f64, h.rpt, n, (int64_t)K);
  };
  auto attempt = [&](int i, bool staged) -> int {
    const PkShape& h = kPkShapes[i];
    if (!covers(h) || (bicg && sp.bj && h.mode == kPkFly) || smem_of(h, staged) > kPkSmemMax || !worth(h, staged))
      return GKO_NOT_SUPPORTED;
    return launch<T, VT>(A, b, x, x_zero, sp, s, out, i, staged, (int)blocks_of(h), K, smem_of(h, staged));
  };
  for (bool staged : {true, false}) {
    const int first = staged ? 0 : kPkFirstGlobal;
    for (int i = first; i <= kPkLastGlobal; ++i) {
      if (twins && kPkShapes[i].mode == kPkFly) {  // its published twin
        const int rc = attempt(i + kPkTwin, staged);
        if (rc != GKO_NOT_SUPPORTED) return rc;
      }
      const int rc = attempt(i, staged);
      if (rc != GKO_NOT_SUPPORTED) return rc;
    }
  }
  return GKO_NOT_SUPPORTED;
}

// GMRES: grid shapes only; the smallest that covers n with one block per SM.
template <typename T, typename VT>
int run_gmres(const gko_matrix_s* A, const double* b, T* x, bool x_zero, const SolveSpec& sp, cudaStream_t s,
              SolveOut* out) {
  const int64_t n = A->n_rows;
  const size_t K = (size_t)std::max<int32_t>(1, A->fmt == GKO_CSR ? A->plan.max_len : A->K);
  for (bool staged : {true, false})
    for (int shape : {11, 12, 13, 14, 9, 10}) {
      const PkShape h = kPkShapes[shape];
      const int64_t rb = (int64_t)h.nt * h.rpt, G = (n + rb - 1) / rb;
      const size_t smem = staged ? K * (size_t)rb * (sizeof(VT) + sizeof(int32_t)) : 0;
      const PkGmresKernel<T, VT> kern = pk_gmres<T, VT>(shape, staged);
      if (!kern || G > std::min(sm_count(), kPkMaxBlocks) || smem > kPkSmemMax) continue;
      if (!staged && !pk_unstaged_worth(2, A->fmt == GKO_CSR, sizeof(T) == 8, h.rpt, n, (int64_t)K)) continue;
      if (smem > 24 * 1024)
        GKO_TRY_CUDA(cudaFuncSetAttribute(kern, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)kPkSmemMax));
      const int64_t ld = (n + 63) / 64 * 64;
      const size_t words = 2 * kPkMaxBlocks * kPkSlot + 2 * 32 * kPkMaxBlocks + 2 * 32 * 2;
      Scratch mem;
      GKO_TRY(mem.get(sizeof(Ctl) + sizeof(ulonglong2) * words + 2048 + sizeof(T) * ((size_t)n + (size_t)ld * (sp.restart + 1)),
                      s));
      Carve cv{static_cast<char*>(mem.data())};
      PkGmresArgs<T, VT> g{};
      g.a = args_of<T, VT>(A, b, x, x_zero, sp, K);
      g.a.c = cv.take<Ctl>(1);
      g.a.slots = cv.take<ulonglong2>(words);
      g.sums = g.a.slots + 2 * kPkMaxBlocks * kPkSlot;
      g.totals = g.sums + 2 * 32 * kPkMaxBlocks;
      g.a.vec[0] = cv.take<T>((size_t)n);
      g.V = cv.take<T>((size_t)ld * (sp.restart + 1));
      g.ld = ld;
      g.m = sp.restart;
      GKO_TRY_CUDA(cudaMemsetAsync(g.a.c, 0, (size_t)((char*)g.a.slots - (char*)g.a.c) + sizeof(ulonglong2) * words, s));
      void* args[] = {&g};
      const cudaError_t e = cudaLaunchCooperativeKernel((const void*)kern, dim3((unsigned)G), dim3((unsigned)h.nt), args,
                                                        smem, s);
      if (e == cudaErrorCooperativeLaunchTooLarge) {  // the blocks cannot all be resident
        cudaGetLastError();
        continue;
      }
      GKO_TRY_CUDA(e);
      return finish<T>(g.a.c, s, out);
    }
  return GKO_NOT_SUPPORTED;
}

}  // namespace

int persist_solve(const gko_matrix_s* A, const double* b, void* x, bool x_zero, const SolveSpec& sp, cudaStream_t s,
                  SolveOut* out) {
  // CSR under the row-block plan (regular rows: other plans keep their SpMV
  // kernels), ELL and SELL-P; reliable updates for BiCGSTAB only
  if (A->n_rows <= 0 || A->n_rows > kSmallRows) return GKO_NOT_SUPPORTED;
  if (sp.bj && (sp.bs & (sp.bs - 1))) return GKO_NOT_SUPPORTED;  // diagonal blocks end with thread blocks
  if (!(A->fmt == GKO_CSR && A->plan.kind == 1) && A->fmt != GKO_ELL && A->fmt != GKO_SELLP) return GKO_NOT_SUPPORTED;
  if (sp.rel && (sp.solver != 1 || sp.rel->A64->fmt != A->fmt)) return GKO_NOT_SUPPORTED;
  int dev = 0, coop = 0;
  if (cudaGetDevice(&dev) != cudaSuccess ||
      cudaDeviceGetAttribute(&coop, cudaDevAttrCooperativeLaunch, dev) != cudaSuccess) {
    cudaGetLastError();
    return GKO_NOT_SUPPORTED;
  }
  if (!coop) return GKO_NOT_SUPPORTED;
  const bool gmres = sp.solver == 2;
  if (gmres && sp.restart > kPkRestart) return GKO_NOT_SUPPORTED;
  switch (A->dtype) {
    case GKO_F64:
      if (gmres) return run_gmres<double, double>(A, b, static_cast<double*>(x), x_zero, sp, s, out);
      return run<double, double>(A, b, static_cast<double*>(x), x_zero, sp, s, out);
    case GKO_F32:
      if (gmres) return run_gmres<float, float>(A, b, static_cast<float*>(x), x_zero, sp, s, out);
      return run<float, float>(A, b, static_cast<float*>(x), x_zero, sp, s, out);
    case GKO_BF16:
      if (gmres) return run_gmres<float, __nv_bfloat16>(A, b, static_cast<float*>(x), x_zero, sp, s, out);
      return run<float, __nv_bfloat16>(A, b, static_cast<float*>(x), x_zero, sp, s, out);
  }
  return GKO_NOT_SUPPORTED;
}

}  // namespace gko
