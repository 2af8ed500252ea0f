// Single-launch restarted GMRES for small systems (Saad-Schultz; the method
// of krylov.cu's multi-kernel solve: classical Gram-Schmidt with selective
// reorthogonalisation, Givens rotations), on persist.cuh's grid exchanges.
//
// The multi-kernel solve takes nine launches an Arnoldi step, 57-80 us
// whatever n; in one launch 33 us for 1,000 rows, 35 for 29,791 and 65 for
// 238,328 (7-point convection-diffusion, restart 30, FP64).  Here a step is the SpMV, one exchange of the j + 2 sums V_i . w
// and w . w, one exchange of the new norm, and the two again where the basis
// needs the second pass.  The j + 2 sums travel in two hops (pk_gather_sums):
// value i is added by block i mod G alone and comes back as one word, since
// every block polling G x (j + 2) slots would be quadratic.  The next basis
// vector is published unscaled with the norm's exchange and A w is scaled
// instead of w (PkScaled), so no exchange stands between the norm and the next SpMV.
// Each thread keeps its rows of the basis to itself in global memory (its own
// loads and stores only); the Hessenberg column, rotations and back
// substitution are the same few operations in warp 0 of every block.
#pragma once

#include "persist.cuh"

namespace gko {

constexpr int kPkRestart = 31;  // the sums of a step fit one warp's lanes

template <typename T, typename VT>
struct PkGmresArgs {
  PkArgs<T, VT> a;  // vec[0]: the published vector
  T* V;             // (m + 1) columns of leading dimension ld
  int64_t ld;
  int m;
  ulonglong2* sums;   // 2 x 32 x kPkMaxBlocks: every block's partial sums
  ulonglong2* totals; // 2 x 32 x 2: the totals, 32 bytes apart
};

template <int NT>
struct PkGmresShared {
  Fx part[32][NT / 32];
  double h[32], h1[32];            // totals of a gather; the first pass's coefficients
  double H[kPkRestart + 1][kPkRestart], cs[kPkRestart], sn[kPkRestart], g[kPkRestart + 1], y[kPkRestart];
  double hi[32], lo[32];           // coefficients of an update, as Lin<T>
  int ok;
};

// Totals over the grid of `count` <= 32 values, whose warp sums are in
// sh.part, into sh.h.  False when a wait timed out (block-uniform).  `all`
// (every cycle's first gather) also stores the words that it does not use, so
// that no word keeps a tag from before its cycle, at most 4 x 31 steps ago.
template <int NT, typename S>
__device__ __forceinline__ bool pk_gather_sums(int count, bool all, S& sh, ulonglong2* sums, ulonglong2* totals,
                                               int* err, unsigned& seq) {
  constexpr unsigned kAll = 0xffffffffu;
  constexpr int NW = NT / 32;
  const int lane = threadIdx.x & 31, w = threadIdx.x >> 5, G = gridDim.x, me = blockIdx.x;
  if (threadIdx.x == 0) sh.ok = 1;
  __syncthreads();
  ++seq;
  ulonglong2* sb = sums + (size_t)(seq & 1u) * 32 * kPkMaxBlocks;
  ulonglong2* tb = totals + (size_t)(seq & 1u) * 32 * 2;
  for (int i = w; i < count; i += NW) {
    const Fx f = NW > 1 ? warp_fx_sum(lane < NW ? sh.part[i][lane] : Fx{0, 1}) : sh.part[i][0];
    if (lane == 0) pk_put(sb + (size_t)i * kPkMaxBlocks + me, pk_word(f, seq));
  }
  if (all && w == 0 && lane >= count) {
    pk_put(sb + (size_t)lane * kPkMaxBlocks + me, pk_word(Fx{0, 1}, seq));
    if (lane % G == me) pk_put(tb + 2 * lane, pk_word(Fx{0, 1}, seq));
  }
  bool dead = false;
  // poll(i): until all the words that this lane reads carry the tag
  auto poll = [&](auto load, ulonglong2 (&v)[kPkPolls]) {
    long long t0 = 0;
    for (unsigned spins = 0;; ++spins) {
      load(v);
      bool ready = true;
#pragma unroll
      for (int k = 0; k < kPkPolls; ++k) ready = ready && pk_tagged(v[k], seq);
      if (__all_sync(kAll, ready)) break;
      if (spins == 64) t0 = clock64();
      if (spins > 64 && clock64() - t0 > kPkWait) dead = true;
      if (__any_sync(kAll, dead)) {
        dead = true;
        break;
      }
    }
  };
  int mine = 0;  // this block's values, spread over its warps
  for (int i = me; i < count && !dead; i += G, ++mine) {
    if (mine % NW != w) continue;
    ulonglong2 v[kPkPolls];
    poll([&](ulonglong2 (&u)[kPkPolls]) {
#pragma unroll
      for (int k = 0; k < kPkPolls; ++k)
        u[k] = lane + 32 * k < G ? pk_get(sb + (size_t)i * kPkMaxBlocks + lane + 32 * k) : pk_word(Fx{0, 1}, seq);
    }, v);
    Fx part[kPkPolls];
#pragma unroll
    for (int k = 0; k < kPkPolls; ++k) part[k] = pk_value(v[k]);
    const Fx f = warp_fx_sum(G > 32 ? lane_fx_sum(part) : part[0]);
    if (lane == 0 && !dead) pk_put(tb + 2 * i, pk_word(f, seq));
  }
  if (w == 0 && !dead) {
    ulonglong2 v[kPkPolls];
    poll([&](ulonglong2 (&u)[kPkPolls]) {
#pragma unroll
      for (int k = 1; k < kPkPolls; ++k) u[k] = pk_word(Fx{0, 1}, seq);
      u[0] = lane < count ? pk_get(tb + 2 * lane) : pk_word(Fx{0, 1}, seq);
    }, v);
    sh.h[lane] = fx_double(pk_value(v[0]));
  }
  if (dead && lane == 0) {
    if (err) atomicOr(err, 1 << GKO_TIMEOUT);
    sh.ok = 0;
  }
  __syncthreads();
  return sh.ok != 0;
}

// The product A (c w) of a published, unscaled w with a factor c.  FP64: (A w)
// times c; w . w and (A v) . (A v) were representable, so A w is.  FP32 holds
// norms down to 2^-126 but not their product with the entries of a small A
// (||w|| = 2^-100, ||A|| = 2^-40), so there the gathered w is first brought to
// about 1 by the power of two below c, exactly, and the rest of c follows: bit
// for bit the same where neither form leaves the range.
template <typename T>
struct PkScaled {
  int k;  // FP32: w is taken as 2^k w
  Lin<T> back;
  static __device__ __forceinline__ int power(double c) {
    if (sizeof(T) == 8) return 0;
    return min(max((int)(((unsigned)__double2hiint(c) >> 20) & 0x7ffu) - 1023, -126), 127);
  }
  static __device__ __forceinline__ double rest(double c, int k) {
    return sizeof(T) == 8 ? c : c * __hiloint2double((1023 - k) << 20, 0);
  }
  __device__ __forceinline__ explicit PkScaled(double c) : k(power(c)), back(pk_lin<T>(pk_pack<T>(rest(c, k)))) {}
  __device__ __forceinline__ T in(T w) const { return sizeof(T) == 8 ? w : w * __int_as_float((k + 127) << 23); }
};

template <typename T, typename VT, int NT, int RPT, bool ST>
__global__ void __launch_bounds__(NT) pk_gmres_kernel(PkGmresArgs<T, VT> ga) {
  constexpr int MODE = kPkGrid, U = 8;
  const PkArgs<T, VT>& a = ga.a;
  extern __shared__ __align__(16) unsigned char smem_raw[];
  __shared__ PkShared<NT, MODE> sh;
  __shared__ PkGmresShared<NT> gs;
  PkVecs<T, NT * RPT, MODE> vec;
  vec.init(a, smem_raw);
  constexpr int X = decltype(vec)::kX;
  PkRows<T, VT, NT, RPT, ST> rows;
  rows.init(a, smem_raw);
  unsigned seq = 0;
  const int lane = threadIdx.x & 31, w = threadIdx.x >> 5;
  auto one = [](T v) { return v; };
  auto at = [&](int k) { return [&vec, k](int32_t c) { return vec.get(k, c); }; };
  auto x0 = [&](int32_t c) { return __ldcg(a.x + c); };
  auto nothing = [](const double (&)[1], double*) {};
  T xj[RPT], wj[RPT];
  double v2[2] = {0.0, 0.0};
#pragma unroll
  for (int j = 0; j < RPT; ++j) {
    const int32_t i = rows.row[j];
    xj[j] = wj[j] = T(0);
    if (i < 0) continue;
    const double bi = a.b[i];
    if (!a.x_zero) xj[j] = a.x[i];
    wj[j] = a.x_zero ? (T)bi : (T)(bi - wd((T)rows.template dot<U>(a, j, x0, one)));
    vec.put(0, i, wj[j]);
    v2[0] += bi * bi;
    v2[1] += wd(wj[j]) * wd(wj[j]);
  }
  // scalars: thread 0 of every block (tol also where it is broadcast)
  double nb = 0.0, tol = 0.0, rr_true = 0.0, hn = 0.0, hh = 0.0;
  int status = kRun, it = 0, cycles = 0;
  // out[0]: 0 go on, 1 converged, 2 b == 0; out[1]: 1 / beta; out[2]: beta
  auto start = [&](double rr, double* o) {
    const double beta = sqrt(rr);
    rr_true = rr;
    o[0] = nb == 0.0 ? 2.0 : beta <= tol ? 1.0 : 0.0;
    o[1] = 1.0 / beta;
    o[2] = beta;
  };
  bool known = true;  // rr_true is ||b - A x||^2 of the final x
  if (!pk_step<NT, MODE, kPubVec, 2>(v2, sh, a.slots, a.err, seq, [&](const double (&t)[2], double* o) {
        nb = sqrt(t[0]);
        tol = a.rel_tol * nb;
        start(t[1], o);
      }))
    status = -1;
  while (status == kRun) {
    // cycle start: r published, its norm in sh.out
    if (pk_flag(sh.out[0])) {
      if (sh.out[0] == 2.0)
#pragma unroll
        for (int j = 0; j < RPT; ++j) xj[j] = T(0);
      status = kConverged;
      break;
    }
    if (it >= a.maxit) {
      status = kNotConverged;
      break;
    }
    if (threadIdx.x <= kPkRestart) gs.g[threadIdx.x] = threadIdx.x == 0 ? sh.out[2] : 0.0;
    double inv = sh.out[1];
    Lin<T> sc = pk_lin<T>(pk_pack<T>(inv));
    PkScaled<T> pr(inv);
    int k = 0;
    bool end = false, broke = false, estimate = false;
    known = false;
    for (int j = 0; !end; ++j) {
      // v_j = w / h, kept; w = A v_j = (A w) / h
      T nw[RPT];
#pragma unroll
      for (int u = 0; u < RPT; ++u) {
        const int32_t i = rows.row[u];
        if (i >= 0) ga.V[(int64_t)j * ga.ld + i] = sc.scale(wj[u]);
        nw[u] = pr.back.scale((T)rows.template dot<U>(a, u, at(0), [&](T v) { return pr.in(v); }));
      }
#pragma unroll
      for (int u = 0; u < RPT; ++u) wj[u] = rows.row[u] >= 0 ? nw[u] : T(0);
      bool again = false;
      for (int pass = 0; pass < 2 && status == kRun; ++pass) {
        // h_i = V_i . w for i <= j; w . w as value j + 1 of the first pass
        for (int i = 0; i <= j + 1 - pass; ++i) {
          double s = 0.0;
#pragma unroll
          for (int u = 0; u < RPT; ++u)
            if (rows.row[u] >= 0) {
              const double ww = wd(wj[u]);
              s = __fma_rn(i <= j ? wd(ga.V[(int64_t)i * ga.ld + rows.row[u]]) : ww, ww, s);
            }
          const Fx f = warp_fx_sum(fx_of(s));
          if (lane == 0) gs.part[i][w] = f;
        }
        if (!pk_gather_sums<NT>(j + 2 - pass, j == 0 && pass == 0, gs, ga.sums, ga.totals, a.err, seq)) {
          status = -1;
          break;
        }
        if (threadIdx.x == 0 && pass == 0) hh = gs.h[j + 1];
        if (threadIdx.x < 32) {
          const double h = gs.h[lane];
          if (pass == 0) gs.h1[lane] = h;
          if constexpr (sizeof(T) == 4) {
            const Lin<float> l = lin_of(-h);
            gs.hi[lane] = l.pack();
          } else {
            gs.hi[lane] = -h;
          }
        }
        __syncthreads();
        double v1[1] = {0.0};
#pragma unroll
        for (int u = 0; u < RPT; ++u) {
          const int32_t i = rows.row[u];
          if (i < 0) continue;
          T v = wj[u];
          for (int l = 0; l <= j; ++l) v = pk_lin<T>(gs.hi[l])(ga.V[(int64_t)l * ga.ld + i], v);
          wj[u] = v;
          vec.put(0, i, v);
          const double ow = wd(v);
          v1[0] = __fma_rn(ow, ow, v1[0]);
        }
        // out[0]: orthogonal enough; then the column of H, the rotations and the cycle's end test
        if (!pk_step<NT, MODE, kPubVec, 1>(v1, sh, a.slots, a.err, seq, [&](const double (&t)[1], double* o) {
              const bool last = pass == 1 || t[0] >= 0.5 * hh;
              o[0] = last ? 1.0 : 0.0;
              if (!last) return;
              double b = 0.0, prev = gs.h1[0] + (pass ? gs.h[0] : 0.0);
              for (int i = 0; i < j; ++i) {
                b = gs.h1[i + 1] + (pass ? gs.h[i + 1] : 0.0);
                gs.H[i][j] = gs.cs[i] * prev + gs.sn[i] * b;
                prev = -gs.sn[i] * prev + gs.cs[i] * b;
              }
              hn = sqrt(t[0]);
              const double den = sqrt(prev * prev + hn * hn);
              o[1] = 0.0;  // 1: the estimate meets the tolerance, 2: breakdown
              if (den == 0.0) {
                o[1] = 2.0;
                return;
              }
              const double cj = prev / den, sj = hn / den;
              gs.cs[j] = cj;
              gs.sn[j] = sj;
              gs.H[j][j] = den;
              const double gj = gs.g[j];
              gs.g[j + 1] = -sj * gj;
              gs.g[j] = cj * gj;
              if (hn == 0.0 || fabs(gs.g[j + 1]) <= tol) o[1] = 1.0;
              o[2] = 1.0 / hn;
            })) {
          status = -1;
          break;
        }
        again = !pk_flag(sh.out[0]);
        if (!again) break;
      }
      if (status != kRun) break;
      ++it;
      broke = sh.out[1] == 2.0;
      estimate = sh.out[1] == 1.0;
      k = broke ? j : j + 1;
      inv = sh.out[2];
      sc = pk_lin<T>(pk_pack<T>(inv));
      pr = PkScaled<T>(inv);
      end = broke || estimate || it >= a.maxit || j + 1 == ga.m;
    }
    if (status != kRun) break;
    // back substitution by warp 0: lane i holds g_i and subtracts column by column
    if (threadIdx.x < 32) {
      const double d = lane < k ? 1.0 / gs.H[lane][lane] : 0.0;
      double s = lane < k ? gs.g[lane] : 0.0;
      for (int i = k - 1; i >= 0; --i) {
        const double y = __shfl_sync(0xffffffffu, s * d, i);
        if (lane == i) gs.y[i] = y;
        if (lane < i) s = __fma_rn(-gs.H[lane][i], y, s);
      }
      __syncwarp();
      if (lane < k) gs.hi[lane] = pk_pack<T>(gs.y[lane]);
    }
    __syncthreads();
    ++cycles;
#pragma unroll
    for (int u = 0; u < RPT; ++u) {
      const int32_t i = rows.row[u];
      if (i < 0) continue;
      T v = xj[u];
      for (int l = 0; l < k; ++l) v = pk_lin<T>(gs.hi[l])(ga.V[(int64_t)l * ga.ld + i], v);
      xj[u] = v;
      vec.put(X, i, v);
    }
    if (broke) {
      status = kBreakdown;
      break;
    }
    if (!a.check_true && estimate) {
      status = kConverged;
      break;
    }
    // the next cycle starts from the true residual
    if (!pk_step<NT, MODE, kPubVec, 0>(nullptr, sh, a.slots, a.err, seq, nothing)) {
      status = -1;
      break;
    }
    double v1[1] = {0.0};
#pragma unroll
    for (int j = 0; j < RPT; ++j) {
      const int32_t i = rows.row[j];
      if (i < 0) continue;
      wj[j] = (T)(a.b[i] - wd((T)rows.template dot<U>(a, j, at(X), one)));
      vec.put(0, i, wj[j]);
      v1[0] += wd(wj[j]) * wd(wj[j]);
    }
    if (!pk_step<NT, MODE, kPubVec, 1>(v1, sh, a.slots, a.err, seq,
                                       [&](const double (&t)[1], double* o) { start(t[0], o); })) {
      status = -1;
      break;
    }
    known = true;
  }
  if (sizeof(T) == 8 && status >= 0 && !known) {  // breakdown: the residual of the x that is returned
    double v1[1] = {0.0};
    if (!pk_step<NT, MODE, kPubVec, 0>(nullptr, sh, a.slots, a.err, seq, nothing)) {
      status = -1;
    } else {
#pragma unroll
      for (int j = 0; j < RPT; ++j)
        if (rows.row[j] >= 0) {
          const double t = a.b[rows.row[j]] - wd((T)rows.template dot<U>(a, j, at(X), one));
          v1[0] += t * t;
        }
      if (!pk_step<NT, MODE, kPubNone, 1>(v1, sh, a.slots, a.err, seq,
                                          [&](const double (&t)[1], double*) { rr_true = t[0]; }))
        status = -1;
    }
  }
#pragma unroll
  for (int j = 0; j < RPT; ++j)
    if (rows.row[j] >= 0) a.x[rows.row[j]] = xj[j];
  if (blockIdx.x == 0 && threadIdx.x == 0) {
    a.c->status = status < 0 ? kNotConverged : status;
    a.c->iter = it;
    a.c->cycles = cycles;
    a.c->nb = nb;
    a.c->rr = rr_true;
  }
  pk_leave(sh, status < 0, &a.c->gave_up);
}

template <typename T, typename VT>
using PkGmresKernel = void (*)(PkGmresArgs<T, VT>);
template <typename T, typename VT>
PkGmresKernel<T, VT> pk_gmres(int shape, bool staged);

#define GKO_PK_GMRES(SH, NT, RPT, MODE)                                                              \
  if (shape == SH) {                                                                                 \
    if (staged) return pk_gmres_kernel<T, VT, NT, RPT, true>;                                        \
    if constexpr (NT >= 256) return pk_gmres_kernel<T, VT, NT, RPT, false>;                          \
  }

}  // namespace gko
