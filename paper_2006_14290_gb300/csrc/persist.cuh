// Single-launch CG and BiCGSTAB for small systems (the solvers the paper's
// Section 1 lists; CG: Saad Alg. 6.18 / 9.1, BiCGSTAB: Saad Alg. 7.7).
//
// Small systems are bound by latency, not bandwidth: one kernel per vector
// operation costs 4-11 us each whatever n (31^3 BiCGSTAB: 42 us an iteration
// in five kernels).  Here one launch of at most one block per SM runs the
// whole solve.  A thread owns RPT rows (block row0 + thread + j NT) and keeps
// their vector entries in registers; the block's matrix entries sit in shared
// memory column-major ([slot][row]: conflict-free).
//
// Reductions double as barriers (pk_step): each block stores its partial sums
// as (value, sequence tag) words in slots that warp 0 of every block polls and
// adds in slot order, so one trip carries both the arrival and the data, every
// block holds bit-identical totals, and nothing is reset.  Divisions, square
// roots and tests run in one thread per block (a dependent FP64 operation
// takes 67 cycles on GB300, a division 552, and the pipe retires a warp
// instruction in 16).
//
// Three ways to share vectors and sums (MODE):
//  kPkCluster: one cluster of up to 16 blocks; published vectors and slots in
//    shared memory, read through distributed shared memory.  A sum of one value
//    takes 2,150 cycles over 16 blocks of 64 threads from the threads' values to
//    the total in every block, 1,500 more for each further value; through L2
//    3,430 for 16 blocks on both dies, 4,060 for 117 and 1,700 to 2,300 more
//    (gko_diag_exchange).  But 16 SMs are all the FP64 pipes there are.  A partial sum
//    in a cluster is taken by its tag, never by the barrier alone: a cluster
//    CG that ordered untagged slots by barriers read one before it was written
//    (FP32, two rows a thread) and stopped some inner solves after a step.
//    What the barrier still orders are the published vectors: stored before
//    its release, read after its acquire by volatile loads.
//  kPkGrid, kPkFly: a cooperative grid; vectors in global memory, read with
//    ld.global.cg (inside one launch L1 is not coherent across SMs).
//  kPkFly: the vector an SpMV gathers is not published after it is formed,
//    which would cost an exchange of its own; gatherers recompute it from
//    published parts instead (CG: p = z + beta p_old; BiCGSTAB: p = r + beta
//    (p_old - omega v_old) and s = r - alpha v), the owner's operations on the
//    owner's values, so every copy is bit-identical.  CG then passes two
//    exchanges an iteration instead of three, BiCGSTAB three instead of five,
//    for one to three more gathers and FMAs per matrix entry.
//
// Every wait is bounded (~1 s); a block that gives up records GKO_TIMEOUT and
// leaves (pk_leave), and so do the others, whose next wait for it runs out; in
// a cluster every block stays until all have left, because its shared memory
// may be read until then.
#pragma once

#include <algorithm>

#include "fx.cuh"
#include "krylov.cuh"

namespace gko {

constexpr long long kPkWait = 1ll << 31;   // clock cycles
constexpr int kPkMaxBlocks = 160;
constexpr int kPkPolls = kPkMaxBlocks / 32;
constexpr int kPkSlot = 8;                 // a block's slot: 8 x 16 bytes, a line of its own
constexpr int kPkCluster16 = 16;           // blocks of a cluster (the most there are)
enum : int { kPkGrid = 0, kPkFly = 1, kPkCluster = 2 };
constexpr size_t kPkSmemMax = 200 * 1024;  // staged entries (and published vectors) per block

template <typename T, typename VT>
struct PkArgs {
  int32_t n;
  int32_t K;        // slots per staged row (longest row)
  gko_format fmt;   // CSR, ELL or SELLP
  const int32_t* rp;   // CSR row pointers, SELL-P slice offsets
  const int32_t* col;
  const VT* val;
  int64_t stride;   // ELL
  int32_t slice;    // SELL-P
  const double* b;  // right-hand side (reliable updates: the initial residual)
  T* x;
  const T* d;       // Jacobi inverse diagonal, or null
  const T* bj;      // block-Jacobi inverse blocks (n x bs), or null; bs a power of two up to 32
  int bs;
  double rel_tol;
  int maxit;
  int check_true;
  int x_zero;
  T* vec[5];        // published vectors, n each
  ulonglong2* slots;  // grid: 2 x kPkMaxBlocks slots, zero at launch
  int* err;
  Ctl* c;
  // reliable updates (FP32 BiCGSTAB): the FP64 matrix values in the layout of
  // `val`, right-hand side, solution and update factor
  const double* val64;
  const double* b64;
  double* x64;
  double delta;
};

// ----------------------------------------------------------- reduction --

// A partial sum in flight: its low and its high 32 bits, each in an 8-byte
// word with the exponent and the step's tag.  The words are stored and loaded
// whole, so a reader that sees both tags has the value.  16 bits of tag are
// enough because every step stores all kPkWords words of a slot, used or not:
// whatever a word held before is from two steps ago (were unused words left
// alone, one could keep a tag that the same step number mod 65,536 matches
// much later).
constexpr int kPkWords = 3;
__device__ __forceinline__ ulonglong2 pk_word(const Fx& f, unsigned tag) {
  const unsigned long long meta = (unsigned long long)((tag << 16) | ((unsigned)f.e & 0xffffu)) << 32;
  return make_ulonglong2(meta | (unsigned)f.v, meta | (unsigned)((unsigned long long)f.v >> 32));
}
__device__ __forceinline__ bool pk_tagged(const ulonglong2& w, unsigned tag) {
  return (unsigned)(w.x >> 48) == (tag & 0xffffu) && (unsigned)(w.y >> 48) == (tag & 0xffffu);
}
__device__ __forceinline__ Fx pk_value(const ulonglong2& w) {
  return Fx{(long long)((w.y << 32) | (w.x & 0xffffffffull)), (int)(short)(w.x >> 32)};
}
__device__ __forceinline__ void pk_put(ulonglong2* p, const ulonglong2& w) {
  asm volatile("st.relaxed.gpu.global.v2.u64 [%0], {%1, %2};" ::"l"(p), "l"(w.x), "l"(w.y) : "memory");
}
__device__ __forceinline__ ulonglong2 pk_get(const ulonglong2* p) {
  ulonglong2 w;
  asm volatile("ld.relaxed.gpu.global.v2.u64 {%0, %1}, [%2];" : "=l"(w.x), "=l"(w.y) : "l"(p) : "memory");
  return w;
}
__device__ __forceinline__ uint32_t pk_smem(const void* p) {
  return static_cast<uint32_t>(__cvta_generic_to_shared(p));
}
__device__ __forceinline__ uint32_t pk_mapa(uint32_t a, unsigned rank) {
  uint32_t r;
  asm volatile("mapa.shared::cluster.u32 %0, %1, %2;" : "=r"(r) : "r"(a), "r"(rank));
  return r;
}
__device__ __forceinline__ void pk_put_peer(uint32_t a, const ulonglong2& w) {
  asm volatile("st.relaxed.cluster.shared::cluster.v2.u64 [%0], {%1, %2};" ::"r"(a), "l"(w.x), "l"(w.y) : "memory");
}
__device__ __forceinline__ ulonglong2 pk_get_own(uint32_t a) {
  ulonglong2 w;
  asm volatile("ld.relaxed.cluster.shared::cta.v2.u64 {%0, %1}, [%2];" : "=l"(w.x), "=l"(w.y) : "r"(a) : "memory");
  return w;
}
__device__ __forceinline__ double pk_ld_peer(uint32_t a, double) {
  double v;
  asm volatile("ld.shared::cluster.f64 %0, [%1];" : "=d"(v) : "r"(a) : "memory");
  return v;
}
__device__ __forceinline__ float pk_ld_peer(uint32_t a, float) {
  float v;
  asm volatile("ld.shared::cluster.f32 %0, [%1];" : "=f"(v) : "r"(a) : "memory");
  return v;
}
__device__ __forceinline__ void pk_cluster_barrier() {
  asm volatile("barrier.cluster.arrive.release;\n\tbarrier.cluster.wait.acquire;" ::: "memory");
}

template <int NT, int MODE>
struct PkShared {
  Fx part[3][NT / 32];
  double out[6];
  int ok;
  unsigned left[MODE == kPkCluster ? kPkCluster16 : 1];  // cluster: the peers that are about to leave
  ulonglong2 slots[2][MODE == kPkCluster ? kPkCluster16 : 1][kPkWords + 1];  // cluster: slots written by the peers
};

template <int NT>
__device__ __forceinline__ void pk_sync() {
  if (NT > 32) __syncthreads();
  else __syncwarp();
}

// What a step makes visible to the other blocks: nothing (the totals only),
// the published vectors, or global memory.
enum : int { kPubNone = 0, kPubVec = 1, kPubGlobal = 2 };
template <int MODE, int PUB>
__device__ __forceinline__ void pk_fence() {
  if (PUB == kPubNone) return;
  if (MODE == kPkCluster && PUB == kPubVec) asm volatile("fence.acq_rel.cluster;" ::: "memory");
  else asm volatile("fence.acq_rel.gpu;" ::: "memory");
}

struct PkNothing {
  __device__ void operator()() const {}
};

// Kernel start.  Cluster: no tag and no flag set, and every block's words are
// clear before a peer writes them.  *gave_up is the host's to clear in a grid.
template <int NT, int MODE>
__device__ __forceinline__ void pk_open(PkShared<NT, MODE>& sh, int* gave_up) {
  if constexpr (MODE == kPkCluster) {
    for (int i = threadIdx.x; i < 2 * kPkCluster16 * (kPkWords + 1); i += NT)
      (&sh.slots[0][0][0])[i] = make_ulonglong2(0ull, 0ull);
    if (threadIdx.x < kPkCluster16) sh.left[threadIdx.x] = 0u;
    if (blockIdx.x == 0 && threadIdx.x == 0) *gave_up = 0;
    pk_cluster_barrier();
  }
}

// Kernel end, after a block's last access to another block's shared memory;
// dead: one of its waits ran out.  Cluster: the block tells every peer and
// passes cluster barriers until all have told it.  When all end together that
// is one barrier.  A block that gives up is ahead of the others, who may still
// pass barriers of their own and read its vectors: they find it here, its
// shared memory alive, until a wait for it has run out for each of them too.
// All flags are set before their writers' next arrival, so nobody reads or
// writes a peer once one block has left.
template <int NT, int MODE>
__device__ __forceinline__ void pk_leave(PkShared<NT, MODE>& sh, bool dead, int* gave_up) {
  if (dead && threadIdx.x == 0) *gave_up = 1;
  if constexpr (MODE == kPkCluster) {
    const unsigned G = gridDim.x;
    if (threadIdx.x < G)
      asm volatile("st.relaxed.cluster.shared::cluster.u32 [%0], %1;" ::"r"(
                       pk_mapa(pk_smem(&sh.left[blockIdx.x]), threadIdx.x)),
                   "r"(1u)
                   : "memory");
    unsigned told = 1u;
    do {
      pk_cluster_barrier();
      if (threadIdx.x < G)
        asm volatile("ld.relaxed.cluster.shared::cta.u32 %0, [%1];" : "=r"(told) : "r"(pk_smem(&sh.left[threadIdx.x])) : "memory");
    } while (!__syncthreads_and(told != 0u));
  }
}

// Sum of NV <= 3 values per thread over all blocks (NV = 0: a barrier); thread 0 of every block then
// runs fin(totals, out) and the block reads out[] from sh.out.  `pre` runs in
// thread 0 while the values travel.  False when a wait timed out
// (block-uniform).  The polling loop is warp-uniform: lanes leaving it one by
// one kept the warp diverged through the FP64 additions that follow (7300
// cycles instead of 3300 for two exchanges of 8 blocks).
// Reuse: a slot of parity q is overwritten two steps later, which a block
// reaches only after all blocks contributed to the step between, i.e. had
// read this one; sh.part and sh.out are rewritten after the step's first and
// read before the next step's first block barrier.
template <int NT, int MODE, int PUB, int NV, typename F, typename P = PkNothing>
__device__ __forceinline__ bool pk_step(const double* v, PkShared<NT, MODE>& sh, ulonglong2* slots, int* err,
                                        unsigned& seq, F fin, P pre = P{}, long long wait = kPkWait) {
  constexpr unsigned kAll = 0xffffffffu;
  if constexpr (MODE == kPkCluster && NV == 0 && PUB != kPubGlobal) {
    pk_cluster_barrier();  // the hardware barrier; a peer that gave up passes it in pk_leave
    return true;
  }
  constexpr int NF = NV > 0 ? NV : 1;  // NV = 0: a barrier only
  static_assert(NF <= kPkWords, "a slot holds the values of one step");
  Fx f[NF] = {};
#pragma unroll
  for (int k = 0; k < NV; ++k) {
    f[k] = warp_fx_sum(fx_of(v[k]));
    if (NT > 32 && (threadIdx.x & 31) == 0) sh.part[k][threadIdx.x >> 5] = f[k];
  }
  pk_sync<NT>();
  ++seq;
  if (NT == 32 || threadIdx.x < 32) {
    const int lane = threadIdx.x & 31;
    pk_fence<MODE, PUB>();  // cumulative over the block barrier
    if constexpr (NT > 32) {
#pragma unroll
      for (int k = 0; k < NV; ++k) f[k] = warp_fx_sum(lane < NT / 32 ? sh.part[k][lane] : Fx{0, 1});
    }
    const int G = gridDim.x, me = blockIdx.x;
    constexpr int NP = MODE == kPkCluster ? 1 : kPkPolls;
    ulonglong2 w[NP][NF];
    ulonglong2* base = slots + (size_t)(seq & 1u) * kPkMaxBlocks * kPkSlot;
    if constexpr (MODE == kPkCluster) {
      const uint32_t a = pk_smem(&sh.slots[seq & 1u][me][0]);
      if (lane < G) {
        const uint32_t r = pk_mapa(a, lane);
#pragma unroll
        for (int k = 0; k < kPkWords; ++k) pk_put_peer(r + 16 * k, pk_word(k < NF ? f[k < NF ? k : 0] : Fx{0, 1}, seq));
      }
    } else if (lane < kPkWords) {
      Fx mine = lane == 0 ? f[0] : Fx{0, 1};
      if (NF > 1 && lane == 1) mine = f[NF > 1 ? 1 : 0];
      if (NF > 2 && lane == 2) mine = f[NF > 2 ? 2 : 0];
      pk_put(base + me * kPkSlot + lane, pk_word(mine, seq));
    }
    if (lane == 0) pre();
    __syncwarp();
    long long t0 = 0;
    bool dead = false;
    for (unsigned spins = 0;; ++spins) {
      bool ready = true;
#pragma unroll
      for (int i = 0; i < NP; ++i)
#pragma unroll
        for (int k = 0; k < NF; ++k) {
          w[i][k] = pk_word(Fx{0, 1}, seq);
          if (lane + 32 * i < G)
            w[i][k] = MODE == kPkCluster ? pk_get_own(pk_smem(&sh.slots[seq & 1u][lane][k]))
                                         : pk_get(base + (lane + 32 * i) * kPkSlot + k);
        }
#pragma unroll
      for (int i = 0; i < NP; ++i)
#pragma unroll
        for (int k = 0; k < NF; ++k) ready = ready && pk_tagged(w[i][k], seq);
      if (__all_sync(kAll, ready)) break;
      if (spins == 64) t0 = clock64();
      if (spins > 64 && clock64() - t0 > wait) dead = true;
      if (__any_sync(kAll, dead)) {
        dead = true;
        break;
      }
    }
    pk_fence<MODE, PUB>();
    double t[NF];
#pragma unroll
    for (int k = 0; k < NV; ++k) {
      if constexpr (NP == 1) {
        f[k] = pk_value(w[0][k]);
      } else {
        Fx part[NP];
#pragma unroll
        for (int i = 0; i < NP; ++i) part[i] = pk_value(w[i][k]);
        f[k] = G > 32 ? lane_fx_sum(part) : part[0];
      }
      t[k] = fx_double(warp_fx_sum(f[k]));
    }
    if (lane == 0) {
      if (!dead) fin(reinterpret_cast<const double (&)[NF]>(t), sh.out);
      else if (err) atomicOr(err, 1 << GKO_TIMEOUT);
      sh.ok = !dead;
    }
  }
  pk_sync<NT>();
  return sh.ok != 0;
}

// A scalar for Lin<T>, packed into a double for broadcasting (float: the
// hi/lo pair).
template <typename T>
__device__ __forceinline__ double pk_pack(double a) {
  if constexpr (sizeof(T) == 8) return a;
  else return lin_of(a).pack();
}
template <typename T>
__device__ __forceinline__ Lin<T> pk_lin(double p) {
  if constexpr (sizeof(T) == 8) return Lin<double>(p);
  else return Lin<float>::unpack(p);
}
__device__ __forceinline__ bool pk_flag(double f) { return __double_as_longlong(f) != 0; }

// sqrt(rr) <= tol, without the square root where rr is clearly above tol^2
// (tol2 = tol * tol; the margin covers the rounding of both)
__device__ __forceinline__ bool pk_meets(double rr, double tol, double tol2) {
  if (tol == 0.0) return rr == 0.0;
  if (tol2 > 1e-280 && rr > tol2 * (1.0 + 1e-14)) return false;
  return sqrt(rr) <= tol;
}

// -------------------------------------------------- published vectors --

// Vectors that other blocks gather: in global memory, or (cluster) each block
// its rows of every vector in shared memory.  Vector kX is the iterate, for
// the true residual.
template <typename T, int RB, int MODE>
struct PkVecs {
  static constexpr int kX = 5;
  T* g[6];
  T* own;         // cluster: this block's rows, vector after vector
  uint32_t base;  // their shared-memory address
  template <typename A>
  __device__ __forceinline__ void init(const A& a, unsigned char* smem) {
#pragma unroll
    for (int k = 0; k < 5; ++k) g[k] = a.vec[k];
    g[kX] = a.x;
    own = reinterpret_cast<T*>(smem);
    base = pk_smem(smem);
  }
  __device__ __forceinline__ int slot(int k) const { return k == kX ? 2 : k; }  // cluster: two vectors and x
  __device__ __forceinline__ void put(int k, int32_t row, T v) const {
    if (MODE == kPkCluster) own[slot(k) * RB + (row & (RB - 1))] = v;
    else __stcg(g[k] + row, v);
  }
  __device__ __forceinline__ T get(int k, int32_t c) const {
    if constexpr (MODE == kPkCluster) {
      const uint32_t a = base + (uint32_t)sizeof(T) * (slot(k) * RB + (c & (RB - 1)));
      return pk_ld_peer(pk_mapa(a, (unsigned)c / RB), T(0));
    } else {
      return __ldcg(g[k] + c);
    }
  }
};
constexpr size_t kPkClusterVecs = 3;

// ----------------------------------------------------------- the rows --

// The thread's rows: bounds, and the row products.  ST: entries staged in
// shared memory; otherwise read from the matrix arrays every time.
template <typename T, typename VT, int NT, int RPT, bool ST>
struct PkRows {
  static constexpr int RB = NT * RPT;
  const VT* sval;
  const int32_t* scol;
  int32_t row[RPT];   // -1: none
  int32_t len[RPT];
  int64_t g0[RPT];    // first entry in the matrix arrays
  int64_t step;       // distance between a row's entries there

  __device__ __forceinline__ void init(const PkArgs<T, VT>& a, unsigned char* smem) {
    VT* sv = reinterpret_cast<VT*>(smem);
    int32_t* sc = reinterpret_cast<int32_t*>(smem + (size_t)a.K * RB * sizeof(VT));
    sval = sv;
    scol = sc;
    step = a.fmt == GKO_CSR ? 1 : a.fmt == GKO_ELL ? a.stride : a.slice;
#pragma unroll
    for (int j = 0; j < RPT; ++j) {
      const int lr = threadIdx.x + j * NT;
      const int32_t i = (int32_t)blockIdx.x * RB + lr;
      row[j] = i < a.n ? i : -1;
      len[j] = 0;
      g0[j] = 0;
      if (i >= a.n) continue;
      int32_t w = a.K;
      if (a.fmt == GKO_CSR) {
        g0[j] = __ldg(a.rp + i);
        w = __ldg(a.rp + i + 1) - (int32_t)g0[j];
      } else if (a.fmt == GKO_ELL) {
        g0[j] = i;
      } else {
        const int32_t s = i / a.slice, b = __ldg(a.rp + s);
        g0[j] = (int64_t)b * a.slice + (i - s * a.slice);
        w = __ldg(a.rp + s + 1) - b;
      }
      // padding (column -1) is trailing; the loads of 8 entries go out together
      int k = 0;
      for (bool more = true; more && k < w;) {
        int32_t c[8];
        VT v[8];
#pragma unroll
        for (int u = 0; u < 8; ++u) {
          const int64_t q = g0[j] + (k + u) * step;
          c[u] = k + u < w ? __ldg(a.col + q) : -1;
          if (ST && k + u < w) v[u] = a.val[q];
        }
#pragma unroll
        for (int u = 0; u < 8; ++u) {
          more = more && c[u] >= 0;
          if (more) {
            if (ST) {
              sc[k * RB + lr] = c[u];
              sv[k * RB + lr] = v[u];
            }
            ++k;
          }
        }
      }
      len[j] = k;
    }
  }

  // Row j: sum of entry * comb(load(column)) in storage order; the loads of
  // up to U entries are issued before their FMAs.
  template <int U, typename L, typename C>
  __device__ __forceinline__ acc_t<VT> dot(const PkArgs<T, VT>& a, int j, L load, C comb) const {
    using R = decltype(load(0));
    acc_t<VT> s = acc_t<VT>(0);
    const int lr = threadIdx.x + j * NT;
    for (int k = 0; k < len[j]; k += U) {
      VT w[U];
      R g[U];
#pragma unroll
      for (int u = 0; u < U; ++u) {
        w[u] = VT(0);
        g[u] = R{};
        if (k + u < len[j]) {
          int32_t c;
          if (ST) {
            c = scol[(k + u) * RB + lr];
            w[u] = sval[(k + u) * RB + lr];
          } else {
            const int64_t q = g0[j] + (k + u) * step;
            c = __ldg(a.col + q);
            w[u] = a.val[q];
          }
          g[u] = load(c);
        }
      }
#pragma unroll
      for (int u = 0; u < U; ++u)
        if (k + u < len[j]) s = madd(to_acc(w[u]), to_acc(comb(g[u])), s);
    }
    return s;
  }

  // Row j of A64 x64 in FP64 (replaced residuals)
  __device__ __forceinline__ double dot64(const PkArgs<T, VT>& a, int j) const {
    double s = 0.0;
    const int lr = threadIdx.x + j * NT;
#pragma unroll 4
    for (int k = 0; k < len[j]; ++k) {
      const int64_t q = g0[j] + k * step;
      const int32_t c = ST ? scol[k * RB + lr] : __ldg(a.col + q);
      s = __fma_rn(__ldg(a.val64 + q), __ldcg(a.x64 + c), s);
    }
    return s;
  }
};

// z = M^-1 v for the thread's rows: Jacobi (d_j), block-Jacobi (the rows of a
// diagonal block are consecutive threads of this block; v goes through shared
// memory, the inverse block's row is read from L2) or none.
template <typename T, typename VT, int NT, int RPT>
struct PkPrecond {
  T* s;  // NT * RPT entries, block-Jacobi only
  __device__ __forceinline__ void apply(const PkArgs<T, VT>& a, const int32_t (&row)[RPT], const T (&d)[RPT],
                                        const T (&v)[RPT], T (&z)[RPT]) const {
    if (a.bj) {
      pk_sync<NT>();
#pragma unroll
      for (int j = 0; j < RPT; ++j) s[threadIdx.x + j * NT] = v[j];
      pk_sync<NT>();
#pragma unroll
      for (int j = 0; j < RPT; ++j) {
        const int first = (int)threadIdx.x & -a.bs;  // thread of the diagonal block's first row
        const int32_t base = row[j] - ((int)threadIdx.x - first);
        const int nb = row[j] < 0 ? 0 : min(a.bs, a.n - base);
        const T* B = a.bj + (int64_t)max(row[j], 0) * a.bs;
        T t = T(0);
#pragma unroll 8
        for (int k = 0; k < nb; ++k) t = madd(__ldg(B + k), s[first + j * NT + k], t);
        z[j] = t;
      }
    } else {
#pragma unroll
      for (int j = 0; j < RPT; ++j) z[j] = a.d ? d[j] * v[j] : v[j];
    }
  }
};

// ----------------------------------------------------------------- CG --

template <typename T, typename VT, int NT, int RPT, int MODE, bool ST>
__global__ void __launch_bounds__(NT, 1) pk_cg_kernel(PkArgs<T, VT> a) {
  constexpr bool FLY = MODE == kPkFly;
  extern __shared__ __align__(16) unsigned char smem_raw[];
  __shared__ PkShared<NT, MODE> sh;
  constexpr int U = 8;
  PkVecs<T, NT * RPT, MODE> vec;
  vec.init(a, smem_raw);
  constexpr int X = decltype(vec)::kX;
  PkRows<T, VT, NT, RPT, ST> rows;
  // shared memory: cluster vectors, block-Jacobi's vector, entries
  unsigned char* sm = smem_raw + (MODE == kPkCluster ? kPkClusterVecs * NT * RPT * sizeof(T) : 0);
  const PkPrecond<T, VT, NT, RPT> pre{reinterpret_cast<T*>(sm)};
  rows.init(a, sm + (a.bj ? NT * RPT * sizeof(T) : 0));
  pk_open(sh, &a.c->gave_up);
  unsigned seq = 0;
  const bool pc = a.d != nullptr || a.bj != nullptr;
  // vector 0: FLY z = M^-1 r, else p; FLY: vectors 1 and 2 p, alternating
  struct Zp {
    T z, p;
  };
  auto one = [](T v) { return v; };
  auto at = [&](int k) { return [&vec, k](int32_t c) { return vec.get(k, c); }; };
  auto x0 = [&](int32_t c) { return __ldcg(a.x + c); };
  T xj[RPT], rj[RPT], pj[RPT], dj[RPT], zj[RPT];
  double v3[3] = {0.0, 0.0, 0.0};
#pragma unroll
  for (int j = 0; j < RPT; ++j) {
    const int32_t i = rows.row[j];
    xj[j] = rj[j] = pj[j] = T(0);
    dj[j] = T(1);
    if (i < 0) continue;
    const double bi = a.b[i];
    if (!a.x_zero) xj[j] = a.x[i];
    if (a.d) dj[j] = a.d[i];
    // staged entries are this thread's own: no barrier needed to read them
    rj[j] = a.x_zero ? (T)bi : (T)(bi - wd((T)rows.template dot<U>(a, j, x0, one)));
    v3[0] += bi * bi;
    v3[1] += wd(rj[j]) * wd(rj[j]);
  }
  pre.apply(a, rows.row, dj, rj, zj);
#pragma unroll
  for (int j = 0; j < RPT; ++j) {
    const int32_t i = rows.row[j];
    if (i < 0) continue;
    vec.put(0, i, zj[j]);
    if (FLY) vec.put(2, i, T(0));  // p_old of the first iteration
    else pj[j] = zj[j];
    v3[2] += wd(rj[j]) * wd(zj[j]);
  }
  // scalars of the recurrence: thread 0 of every block, the same in each
  double nb = 0.0, tol = 0.0, tol2 = 0.0, rho = 0.0, rho_prev = 0.0, rr_true = 0.0;
  int status = kRun, it = 0;
  bool known = false;  // rr_true is ||b - A x||^2 of the final x
  if (!pk_step<NT, MODE, kPubVec, 3>(v3, sh, a.slots, a.err, seq, [&](const double (&t)[3], double* o) {
        nb = sqrt(t[0]);
        tol = a.rel_tol * nb;
        tol2 = tol * tol;
        rho = t[2];
        rr_true = t[1];
        o[0] = t[0] == 0.0 ? 1.0 : 0.0;
        o[1] = sqrt(t[1]) <= tol ? 1.0 : 0.0;
      }))
    status = -1;
  if (status == kRun) {
    if (pk_flag(sh.out[0])) {  // b == 0: x = 0 after 0 iterations
#pragma unroll
      for (int j = 0; j < RPT; ++j) xj[j] = T(0);
      status = kConverged;
      known = true;
    } else if (pk_flag(sh.out[1])) {
      status = kConverged;
      known = true;
    } else if (a.maxit <= 0) {
      status = kNotConverged;
      known = true;
    }
  }
  Lin<T> bp = pk_lin<T>(pk_pack<T>(0.0));
  // t = b - A x from the published x; totals {t.t, t.M^-1 t}
  auto true_residual = [&](T (&tj)[RPT], auto fin) -> bool {
#pragma unroll
    for (int j = 0; j < RPT; ++j)
      if (rows.row[j] >= 0) vec.put(X, rows.row[j], xj[j]);
    if (!pk_step<NT, MODE, kPubVec, 0>(nullptr, sh, a.slots, a.err, seq, [](const double (&)[1], double*) {})) return false;
    double vt[2] = {0.0, 0.0};
#pragma unroll
    for (int j = 0; j < RPT; ++j) {
      const int32_t i = rows.row[j];
      tj[j] = i >= 0 ? (T)(a.b[i] - wd((T)rows.template dot<U>(a, j, at(X), one))) : T(0);
      vt[0] += wd(tj[j]) * wd(tj[j]);
    }
    pre.apply(a, rows.row, dj, tj, zj);
#pragma unroll
    for (int j = 0; j < RPT; ++j) vt[1] += wd(tj[j]) * wd(zj[j]);
    return pk_step<NT, MODE, kPubNone, 2>(vt, sh, a.slots, a.err, seq, fin);
  };
  while (status == kRun) {
    double v1[1] = {0.0};
    T qj[RPT];
    if constexpr (FLY) {
      const T* zb = vec.g[0];
      const T* po = it & 1 ? vec.g[1] : vec.g[2];
      T* pn = it & 1 ? vec.g[2] : vec.g[1];
#pragma unroll
      for (int j = 0; j < RPT; ++j) {
        if (rows.row[j] < 0) continue;
        pj[j] = bp(pj[j], zj[j]);
        __stcg(pn + rows.row[j], pj[j]);
      }
#pragma unroll
      for (int j = 0; j < RPT; ++j)
        qj[j] = (T)rows.template dot<U>(
            a, j, [&](int32_t c) { return Zp{__ldcg(zb + c), __ldcg(po + c)}; },
            [&](const Zp& g) { return bp(g.p, g.z); });
    } else {
#pragma unroll
      for (int j = 0; j < RPT; ++j) qj[j] = (T)rows.template dot<U>(a, j, at(0), one);
    }
#pragma unroll
    for (int j = 0; j < RPT; ++j) v1[0] += wd(pj[j]) * wd(qj[j]);
    if (!pk_step<NT, MODE, kPubNone, 1>(v1, sh, a.slots, a.err, seq, [&](const double (&t)[1], double* o) {
          const bool up = t[0] > 0.0;
          const double alpha = up ? fast_div(rho, t[0]) : 0.0;
          o[0] = up ? 1.0 : 0.0;
          o[1] = pk_pack<T>(alpha);
          o[2] = pk_pack<T>(-alpha);
        })) {
      status = -1;
      break;
    }
    if (!pk_flag(sh.out[0])) {
      status = kBreakdown;
      break;
    }
    const Lin<T> ax = pk_lin<T>(sh.out[1]), ar = pk_lin<T>(sh.out[2]);
    double v2[2] = {0.0, 0.0};
#pragma unroll
    for (int j = 0; j < RPT; ++j) {
      const int32_t i = rows.row[j];
      if (i < 0) continue;
      xj[j] = ax(pj[j], xj[j]);
      rj[j] = ar(qj[j], rj[j]);
      const double rw = wd(rj[j]);
      v2[0] = __fma_rn(rw, rw, v2[0]);
    }
    pre.apply(a, rows.row, dj, rj, zj);
#pragma unroll
    for (int j = 0; j < RPT; ++j) {
      if (rows.row[j] < 0) continue;
      if (FLY) vec.put(0, rows.row[j], zj[j]);
      if (pc) v2[1] = __fma_rn(wd(rj[j]), wd(zj[j]), v2[1]);
    }
    double inv = 0.0;  // 1 / rho, formed while the sums travel
    auto ahead = [&] { inv = 1.0 / rho; };
    auto fin2 = [&](double rr, double rz, double* o) {
      o[0] = pk_meets(rr, tol, tol2) ? 1.0 : 0.0;
      // rz / rho: the product's error is removed with its exact residual
      const double q = rz * inv, f = __fma_rn(-rho, q, rz);
      o[1] = pk_pack<T>(isfinite(f) ? __fma_rn(f, inv, q) : rz / rho);
      rho_prev = rho;
      rho = rz;
    };
    bool ok;
    if (pc) {
      ok = pk_step<NT, MODE, FLY ? kPubVec : kPubNone, 2>(v2, sh, a.slots, a.err, seq,
                            [&](const double (&t)[2], double* o) { fin2(t[0], t[1], o); }, ahead);
    } else {
      const double w1[1] = {v2[0]};
      ok = pk_step<NT, MODE, FLY ? kPubVec : kPubNone, 1>(w1, sh, a.slots, a.err, seq,
                            [&](const double (&t)[1], double* o) { fin2(t[0], t[0], o); }, ahead);
    }
    if (!ok) {
      status = -1;
      break;
    }
    ++it;
    bp = pk_lin<T>(sh.out[1]);
    if (pk_flag(sh.out[0])) {
      if (!a.check_true) {
        status = kConverged;
        break;
      }
      T tj[RPT];
      if (!true_residual(tj, [&](const double (&t)[2], double* o) {
            rr_true = t[0];
            // 0 go on, 1 converged, 3 iteration cap (close to the attainable accuracy the
            // recurrence may meet the tolerance in every step and the true residual in none)
            o[0] = sqrt(t[0]) <= tol ? 1.0 : it >= a.maxit ? 3.0 : 0.0;
            o[1] = pk_pack<T>(t[1] / rho_prev);
            rho = t[1];
          })) {
        status = -1;
        break;
      }
      if (pk_flag(sh.out[0])) {
        status = sh.out[0] == 1.0 ? kConverged : kNotConverged;
        known = true;
        break;
      }
      bp = pk_lin<T>(sh.out[1]);  // residual replacement (p is kept)
#pragma unroll
      for (int j = 0; j < RPT; ++j) {
        rj[j] = tj[j];
        if (FLY && rows.row[j] >= 0) vec.put(0, rows.row[j], zj[j]);  // of t
      }
      if (FLY && !pk_step<NT, MODE, kPubVec, 0>(nullptr, sh, a.slots, a.err, seq, [](const double (&)[1], double*) {})) {
        status = -1;
        break;
      }
    } else if (it >= a.maxit) {
      status = kNotConverged;
      break;
    }
    if constexpr (!FLY) {
#pragma unroll
      for (int j = 0; j < RPT; ++j) {
        if (rows.row[j] < 0) continue;
        pj[j] = bp(pj[j], zj[j]);
        vec.put(0, rows.row[j], pj[j]);
      }
      if (!pk_step<NT, MODE, kPubVec, 0>(nullptr, sh, a.slots, a.err, seq, [](const double (&)[1], double*) {})) {
        status = -1;
        break;
      }
    }
  }
  // the residual of the x that is returned (FP64 solves report it)
  if (sizeof(T) == 8 && status >= 0 && !known) {
    T tj[RPT];
    if (!true_residual(tj, [&](const double (&t)[2], double*) { rr_true = t[0]; })) status = -1;
  }
#pragma unroll
  for (int j = 0; j < RPT; ++j)
    if (rows.row[j] >= 0) a.x[rows.row[j]] = xj[j];
  if (blockIdx.x == 0 && threadIdx.x == 0) {
    a.c->status = status < 0 ? kNotConverged : status;
    a.c->iter = it;
    a.c->cycles = 0;
    a.c->nb = nb;
    a.c->rr = rr_true;
  }
  pk_leave(sh, status < 0, &a.c->gave_up);
}

// ----------------------------------------------------------- BiCGSTAB --

// REL (FP32): mixed precision with reliable updates, as krylov.cu's
// multi-kernel solve (RelOp): x accumulates the change of the FP64 solution;
// when the recurrence residual meets the tolerance or drops below delta times
// its largest norm since the last update, the change is added to x64 and r is
// replaced by b64 - A64 x64 computed in FP64.
template <typename T, typename VT, int NT, int RPT, int MODE, bool ST, bool REL>
__global__ void __launch_bounds__(NT, 1) pk_bicg_kernel(PkArgs<T, VT> a) {
  constexpr bool FLY = MODE == kPkFly;
  extern __shared__ __align__(16) unsigned char smem_raw[];
  __shared__ PkShared<NT, MODE> sh;
  constexpr int U = 8;
  PkVecs<T, NT * RPT, MODE> vec;
  vec.init(a, smem_raw);
  constexpr int X = decltype(vec)::kX;
  PkRows<T, VT, NT, RPT, ST> rows;
  // shared memory: cluster vectors, block-Jacobi's vector, entries
  unsigned char* sm = smem_raw + (MODE == kPkCluster ? kPkClusterVecs * NT * RPT * sizeof(T) : 0);
  const PkPrecond<T, VT, NT, RPT> pre{reinterpret_cast<T*>(sm)};
  rows.init(a, sm + (a.bj ? NT * RPT * sizeof(T) : 0));
  pk_open(sh, &a.c->gave_up);
  unsigned seq = 0;
  const bool pc = a.d != nullptr;  // FLY gatherers apply it
  const bool reliable = REL && a.val64 != nullptr;
  // FLY: r, p (two buffers), v (two buffers); else vec[0] = M^-1 p, vec[1] = M^-1 s
  T* rb = vec.g[0];
  struct Rpv {
    T r, p, v, d;
  };
  struct Rv {
    T r, v, d;
  };
  auto one = [](T v) { return v; };
  auto at = [&](int k) { return [&vec, k](int32_t c) { return vec.get(k, c); }; };
  auto x0 = [&](int32_t c) { return __ldcg(a.x + c); };
  auto nothing = [](const double (&)[1], double*) {};
  T xj[RPT], rj[RPT], hj[RPT], pj[RPT], vj[RPT], dj[RPT];
  double v2[2] = {0.0, 0.0};
#pragma unroll
  for (int j = 0; j < RPT; ++j) {
    const int32_t i = rows.row[j];
    xj[j] = rj[j] = hj[j] = pj[j] = vj[j] = T(0);
    dj[j] = T(1);
    if (i < 0) continue;
    const double bi = a.b[i];
    if (!a.x_zero) xj[j] = a.x[i];
    if (a.d) dj[j] = a.d[i];
    rj[j] = a.x_zero ? (T)bi : (T)(bi - wd((T)rows.template dot<U>(a, j, x0, one)));
    hj[j] = rj[j];
    if (FLY) {
      vec.put(0, i, rj[j]);
      vec.put(2, i, T(0));
      vec.put(4, i, T(0));
    }
    v2[0] += bi * bi;
    v2[1] += wd(rj[j]) * wd(rj[j]);
  }
  // scalars: thread 0 of every block
  double nb = 0.0, tol = 0.0, tol2 = 0.0, rr_true = 0.0, maxrr = 0.0;
  double rho = 1.0, rho_new = 0.0, alpha = 1.0, omega = 1.0;
  int status = kRun, it = 0, cycles = 0, par = 0;
  bool known = false;
  Lin<T> bp = pk_lin<T>(pk_pack<T>(0.0)), wv = bp;
  if (!pk_step<NT, MODE, kPubVec, 2>(v2, sh, a.slots, a.err, seq, [&](const double (&t)[2], double* o) {
        nb = sqrt(t[0]);
        tol = a.rel_tol * nb;
        tol2 = tol * tol;
        rr_true = t[1];
        maxrr = sqrt(t[1]);
        rho_new = t[1];  // rhat = r
        o[0] = t[0] == 0.0 ? 1.0 : 0.0;
        o[1] = sqrt(t[1]) <= tol ? 1.0 : 0.0;
        o[2] = pk_pack<T>(t[1]);
        o[3] = pk_pack<T>(-1.0);
      }))
    status = -1;
  if (status == kRun) {
    bp = pk_lin<T>(sh.out[2]);
    wv = pk_lin<T>(sh.out[3]);
    known = true;
    if (pk_flag(sh.out[0])) {  // b == 0: x = 0 after 0 iterations
#pragma unroll
      for (int j = 0; j < RPT; ++j) xj[j] = T(0);
      status = kConverged;
    } else if (pk_flag(sh.out[1])) {
      status = kConverged;
    } else if (a.maxit <= 0) {
      status = kNotConverged;
    } else {
      known = false;
    }
  }
  auto true_residual = [&](T (&tj)[RPT], auto fin) -> bool {
#pragma unroll
    for (int j = 0; j < RPT; ++j)
      if (rows.row[j] >= 0) vec.put(X, rows.row[j], xj[j]);
    if (!pk_step<NT, MODE, kPubVec, 0>(nullptr, sh, a.slots, a.err, seq, nothing)) return false;
    double vt[2] = {0.0, 0.0};
#pragma unroll
    for (int j = 0; j < RPT; ++j) {
      const int32_t i = rows.row[j];
      tj[j] = i >= 0 ? (T)(a.b[i] - wd((T)rows.template dot<U>(a, j, at(X), one))) : T(0);
      vt[0] += wd(tj[j]) * wd(tj[j]);
      vt[1] += wd(hj[j]) * wd(tj[j]);
    }
    return pk_step<NT, MODE, kPubNone, 2>(vt, sh, a.slots, a.err, seq, fin);
  };
  // continue from the replaced residual r (restart: with p = v = 0)
  auto republish = [&](bool restart) -> bool {
    if (restart)
#pragma unroll
      for (int j = 0; j < RPT; ++j) pj[j] = vj[j] = T(0);
    if constexpr (FLY) {
#pragma unroll
      for (int j = 0; j < RPT; ++j) {
        const int32_t i = rows.row[j];
        if (i < 0) continue;
        vec.put(0, i, rj[j]);
        if (restart) {
          vec.put(par ? 1 : 2, i, T(0));
          vec.put(par ? 3 : 4, i, T(0));
        }
      }
      return pk_step<NT, MODE, kPubVec, 0>(nullptr, sh, a.slots, a.err, seq, nothing);
    }
    return true;
  };
  while (status == kRun) {
    // ---- p, v = A M^-1 p, alpha
    T phj[RPT];
    const T* po = par ? vec.g[1] : vec.g[2];
    const T* vo = par ? vec.g[3] : vec.g[4];
    T* pn = par ? vec.g[2] : vec.g[1];
    T* vn = par ? vec.g[4] : vec.g[3];
#pragma unroll
    for (int j = 0; j < RPT; ++j) {
      const int32_t i = rows.row[j];
      phj[j] = T(0);
      if (i < 0) continue;
      pj[j] = bp(wv(vj[j], pj[j]), rj[j]);
      if (FLY) __stcg(pn + i, pj[j]);
    }
    pre.apply(a, rows.row, dj, pj, phj);
    if constexpr (!FLY)
#pragma unroll
      for (int j = 0; j < RPT; ++j)
        if (rows.row[j] >= 0) vec.put(0, rows.row[j], phj[j]);
    if constexpr (!FLY)
      if (!pk_step<NT, MODE, kPubVec, 0>(nullptr, sh, a.slots, a.err, seq, nothing)) {
        status = -1;
        break;
      }
    double v1[1] = {0.0};
#pragma unroll
    for (int j = 0; j < RPT; ++j) {
      if constexpr (FLY) {
        vj[j] = (T)rows.template dot<U>(
            a, j,
            [&](int32_t c) { return Rpv{__ldcg(rb + c), __ldcg(po + c), __ldcg(vo + c), pc ? __ldg(a.d + c) : T(1)}; },
            [&](const Rpv& g) {
              const T p = bp(wv(g.v, g.p), g.r);
              return pc ? g.d * p : p;
            });
        if (rows.row[j] >= 0) __stcg(vn + rows.row[j], vj[j]);
      } else {
        vj[j] = (T)rows.template dot<U>(a, j, at(0), one);
      }
      v1[0] += wd(hj[j]) * wd(vj[j]);
    }
    if (!pk_step<NT, MODE, FLY ? kPubVec : kPubNone, 1>(v1, sh, a.slots, a.err, seq, [&](const double (&t)[1], double* o) {
          const bool up = t[0] != 0.0;
          o[0] = up ? 1.0 : 0.0;
          if (up) alpha = fast_div(rho_new, t[0]);
          o[1] = pk_pack<T>(alpha);
          o[2] = pk_pack<T>(-alpha);
        })) {
      status = -1;
      break;
    }
    if (!pk_flag(sh.out[0])) {
      status = kBreakdown;
      break;
    }
    ++it;
    const Lin<T> ap = pk_lin<T>(sh.out[1]), av = pk_lin<T>(sh.out[2]);
    // ---- s, t = A M^-1 s, omega
    T sj[RPT], tj[RPT], shj[RPT];
    double v3[3] = {0.0, 0.0, 0.0};
#pragma unroll
    for (int j = 0; j < RPT; ++j) {
      sj[j] = T(0);
      if (rows.row[j] < 0) continue;
      sj[j] = av(vj[j], rj[j]);
      const double sw = wd(sj[j]);
      v3[2] = __fma_rn(sw, sw, v3[2]);
    }
    pre.apply(a, rows.row, dj, sj, shj);
    if constexpr (!FLY)
#pragma unroll
      for (int j = 0; j < RPT; ++j)
        if (rows.row[j] >= 0) vec.put(1, rows.row[j], shj[j]);
    if constexpr (!FLY)
      if (!pk_step<NT, MODE, kPubVec, 0>(nullptr, sh, a.slots, a.err, seq, nothing)) {
        status = -1;
        break;
      }
#pragma unroll
    for (int j = 0; j < RPT; ++j) {
      if constexpr (FLY) {
        tj[j] = (T)rows.template dot<U>(
            a, j, [&](int32_t c) { return Rv{__ldcg(rb + c), __ldcg(vn + c), pc ? __ldg(a.d + c) : T(1)}; },
            [&](const Rv& g) {
              const T s = av(g.v, g.r);
              return pc ? g.d * s : s;
            });
      } else {
        tj[j] = (T)rows.template dot<U>(a, j, at(1), one);
      }
      const double tw = wd(tj[j]);
      v3[0] = __fma_rn(wd(sj[j]), tw, v3[0]);
      v3[1] = __fma_rn(tw, tw, v3[1]);
    }
    if (!pk_step<NT, MODE, kPubNone, 3>(v3, sh, a.slots, a.err, seq, [&](const double (&t)[3], double* o) {
          const bool half = pk_meets(t[2], tol, tol2);
          o[0] = half ? 1.0 : 0.0;
          o[1] = t[1] == 0.0 ? 1.0 : 0.0;
          if (!half && t[1] != 0.0) omega = fast_div(t[0], t[1]);
          o[2] = pk_pack<T>(omega);
          o[3] = pk_pack<T>(-omega);
        })) {
      status = -1;
      break;
    }
    const bool half = pk_flag(sh.out[0]);
    bool check = half;
    par ^= 1;
    if (half) {  // ||s|| small: x += alpha M^-1 p
#pragma unroll
      for (int j = 0; j < RPT; ++j)
        if (rows.row[j] >= 0) xj[j] = ap(phj[j], xj[j]);
    } else {
      if (pk_flag(sh.out[1])) {
        status = kBreakdown;
        break;
      }
      const Lin<T> os = pk_lin<T>(sh.out[2]), ot = pk_lin<T>(sh.out[3]);
      wv = ot;
      v2[0] = v2[1] = 0.0;
#pragma unroll
      for (int j = 0; j < RPT; ++j) {
        const int32_t i = rows.row[j];
        if (i < 0) continue;
        xj[j] = os(shj[j], ap(phj[j], xj[j]));
        rj[j] = ot(tj[j], sj[j]);
        if (FLY) vec.put(0, i, rj[j]);
        const double rw = wd(rj[j]);
        v2[0] = __fma_rn(rw, rw, v2[0]);
        v2[1] = __fma_rn(wd(hj[j]), rw, v2[1]);
      }
      double ratio = 0.0;  // (alpha / omega) / rho, formed while the sums travel
      // out[0]: 0 go on, 1 check (converged, or an update is due), 2 breakdown, 3 iteration cap
      if (!pk_step<NT, MODE, FLY ? kPubVec : kPubNone, 2>(v2, sh, a.slots, a.err, seq, [&](const double (&t)[2], double* o) {
            rho = rho_new;
            rho_new = t[1];
            double code = 0.0;
            if (pk_meets(t[0], tol, tol2)) code = 1.0;
            if (REL && code == 0.0 && a.delta > 0.0) {
              const double nr = sqrt(t[0]);
              maxrr = nr > maxrr ? nr : maxrr;
              if (nr < a.delta * maxrr) code = 1.0;
            }
            if (code == 0.0) {
              if (omega == 0.0 || (it < a.maxit && rho_new == 0.0)) code = 2.0;
              else if (it >= a.maxit) code = 3.0;
              else o[1] = pk_pack<T>(rho_new * ratio);
            }
            o[0] = code;
          }, [&] { ratio = (alpha / omega) / rho_new; })) {
        status = -1;
        break;
      }
      const double code = sh.out[0];
      if (code == 2.0 || code == 3.0) {
        status = code == 2.0 ? kBreakdown : kNotConverged;
        break;
      }
      check = pk_flag(code);
      if (!check) bp = pk_lin<T>(sh.out[1]);
    }
    if (!check) continue;
    if constexpr (REL) {
      if (reliable) {  // x64 += x, x = 0, r = fl(b64 - A64 x64)
#pragma unroll
        for (int j = 0; j < RPT; ++j) {
          const int32_t i = rows.row[j];
          if (i < 0) continue;
          __stcg(a.x64 + i, __ldcg(a.x64 + i) + wd(xj[j]));
          xj[j] = T(0);
        }
        if (!pk_step<NT, MODE, kPubGlobal, 0>(nullptr, sh, a.slots, a.err, seq, nothing)) {
          status = -1;
          break;
        }
        v2[0] = v2[1] = 0.0;
#pragma unroll
        for (int j = 0; j < RPT; ++j) {
          const int32_t i = rows.row[j];
          if (i < 0) continue;
          const double ti = a.b64[i] - rows.dot64(a, j);
          rj[j] = (T)ti;
          v2[0] = __fma_rn(ti, ti, v2[0]);
          v2[1] = __fma_rn(wd(hj[j]), wd(rj[j]), v2[1]);
        }
        ++cycles;
        // out[0]: 0 go on, 1 converged, 2 breakdown, 3 iteration cap
        if (!pk_step<NT, MODE, kPubNone, 2>(v2, sh, a.slots, a.err, seq, [&](const double (&t)[2], double* o) {
              const double rn = sqrt(t[0]);
              double code = 0.0;
              if (rn <= tol) {
                code = 1.0;
              } else {
                maxrr = rn;
                if (!half && omega == 0.0) code = 2.0;
                else if (it >= a.maxit) code = 3.0;
                else if (t[1] == 0.0) code = 2.0;
                rho_new = t[1];
                if (half) {
                  rho = alpha = omega = 1.0;
                  o[1] = pk_pack<T>(t[1]);
                } else {
                  o[1] = pk_pack<T>((rho_new / rho) * (alpha / omega));
                }
              }
              o[0] = code;
              o[2] = pk_pack<T>(-omega);
            })) {
          status = -1;
          break;
        }
        const double code = sh.out[0];
        if (code != 0.0) {
          status = code == 1.0 ? kConverged : code == 2.0 ? kBreakdown : kNotConverged;
          break;
        }
        bp = pk_lin<T>(sh.out[1]);
        wv = pk_lin<T>(sh.out[2]);
        if (!republish(half)) {
          status = -1;
          break;
        }
        continue;
      }
    }
    if (!a.check_true) {
      status = kConverged;
      break;
    }
    // out[0]: 0 go on, 1 converged, 2 breakdown, 3 iteration cap
    if (!true_residual(tj, [&](const double (&t)[2], double* o) {
          rr_true = t[0];
          double code = 0.0;
          if (sqrt(t[0]) <= tol) code = 1.0;
          else if (it >= a.maxit) code = 3.0;
          else if (t[1] == 0.0) code = 2.0;
          rho = alpha = omega = 1.0;
          rho_new = t[1];
          o[0] = code;
          o[1] = pk_pack<T>(t[1]);
          o[2] = pk_pack<T>(-1.0);
        })) {
      status = -1;
      break;
    }
    const double code = sh.out[0];
    known = true;
    if (code != 0.0) {
      status = code == 1.0 ? kConverged : code == 2.0 ? kBreakdown : kNotConverged;
      break;
    }
    known = false;
    bp = pk_lin<T>(sh.out[1]);
    wv = pk_lin<T>(sh.out[2]);
#pragma unroll
    for (int j = 0; j < RPT; ++j) rj[j] = tj[j];
    if (!republish(true)) {
      status = -1;
      break;
    }
  }
  if (reliable) {  // what moved since the last update
    if (status >= 0)
#pragma unroll
      for (int j = 0; j < RPT; ++j)
        if (rows.row[j] >= 0) __stcg(a.x64 + rows.row[j], __ldcg(a.x64 + rows.row[j]) + wd(xj[j]));
  } else {
    if (sizeof(T) == 8 && status >= 0 && !known) {
      T tj[RPT];
      if (!true_residual(tj, [&](const double (&t)[2], double*) { rr_true = t[0]; })) status = -1;
    }
#pragma unroll
    for (int j = 0; j < RPT; ++j)
      if (rows.row[j] >= 0) a.x[rows.row[j]] = xj[j];
  }
  if (blockIdx.x == 0 && threadIdx.x == 0) {
    a.c->status = status < 0 ? kNotConverged : status;
    a.c->iter = it;
    a.c->cycles = cycles;
    a.c->nb = nb;
    a.c->rr = rr_true;
  }
  pk_leave(sh, status < 0, &a.c->gave_up);
}

// -------------------------------------------------------------- launch --

template <typename T, typename VT>
using PkKernel = void (*)(PkArgs<T, VT>);

// Shapes: threads x rows per thread and mode, in order of preference; the
// first that covers n (with the 16 blocks of a cluster, else one block per
// SM) and whose entries fit is taken, so the fewest rows per SM; what long rows
// change about that is in persist.cu.  Measured, us per iteration (100 CG or 20 BiCGSTAB iterations, setup included), one step
// to the next shape on either side of each line:
//   cluster -> kPkFly after 16 x 512 rows: CG on 8,100 rows 6.2 in the cluster,
//     7.1 as 64-thread kPkFly blocks; on 4,096 rows 4.5 and 6.7
//   kPkFly -> kPkGrid after 512 rows per block (CG on 29,791 rows 7.6 as kPkFly
//     blocks of 256 rows, 12.5 as kPkGrid blocks of 1,024), and for rows of
//     more than kPkFlyRow entries, whose extra gathers cost more than the
//     exchange they save
//   512 threads x 2 and 4 rows above that: CG on 91,125 rows 11.6, 238,328
//     rows 16.4 (256 threads x 4 and 8: 12.4 and 20.4)
struct PkShape {
  int nt, rpt, mode;
};
constexpr PkShape kPkShapes[] = {
    {32, 1, kPkCluster}, {64, 1, kPkCluster}, {128, 1, kPkCluster}, {256, 1, kPkCluster}, {256, 2, kPkCluster},
    {64, 1, kPkFly}, {128, 1, kPkFly}, {256, 1, kPkFly}, {512, 1, kPkFly}, {512, 2, kPkGrid}, {512, 4, kPkGrid},
    // instead of kPkFly where rows are long, and for BiCGSTAB with block-Jacobi, whose preconditioned directions no
    // gatherer can recompute
    {64, 1, kPkGrid}, {128, 1, kPkGrid}, {256, 1, kPkGrid}, {512, 1, kPkGrid}};
constexpr int kPkTwin = 6;  // from a kPkFly shape to the published one of its size
// unstaged variants: shapes kPkFirstGlobal to kPkLastGlobal and the twins of these
constexpr int kPkFirstGlobal = 7, kPkLastGlobal = 10;
constexpr bool pk_unstaged(int shape) {
  return (shape >= kPkFirstGlobal && shape <= kPkLastGlobal) || shape >= kPkFirstGlobal + kPkTwin;
}

// The kernel of a shape, with or without staging, or null; one translation
// unit per solver and value type instantiates them (persist_*.cu).
template <typename T, typename VT>
PkKernel<T, VT> pk_cg(int shape, bool staged);
template <typename T, typename VT>
PkKernel<T, VT> pk_bicg(int shape, bool staged);

#define GKO_PK_SHAPES(CASE)                                                                          \
  CASE(0, 32, 1, kPkCluster) CASE(1, 64, 1, kPkCluster) CASE(2, 128, 1, kPkCluster)                  \
  CASE(3, 256, 1, kPkCluster) CASE(4, 256, 2, kPkCluster) CASE(5, 64, 1, kPkFly)                     \
  CASE(6, 128, 1, kPkFly) CASE(7, 256, 1, kPkFly) CASE(8, 512, 1, kPkFly) CASE(9, 512, 2, kPkGrid)   \
  CASE(10, 512, 4, kPkGrid)
#define GKO_PK_BLOCK_SHAPES(CASE)                                                                    \
  CASE(11, 64, 1, kPkGrid) CASE(12, 128, 1, kPkGrid) CASE(13, 256, 1, kPkGrid) CASE(14, 512, 1, kPkGrid)
#define GKO_PK_CG(SH, NT, RPT, MODE)                                                                  \
  if (shape == SH) {                                                                                 \
    if (staged) return pk_cg_kernel<T, VT, NT, RPT, MODE, true>;                                      \
    if constexpr (pk_unstaged(SH)) return pk_cg_kernel<T, VT, NT, RPT, MODE, false>;                  \
  }
#define GKO_PK_BICG(SH, NT, RPT, MODE)                                                                \
  if (shape == SH) {                                                                                 \
    if (staged) return pk_bicg_kernel<T, VT, NT, RPT, MODE, true, sizeof(T) == 4>;                    \
    if constexpr (pk_unstaged(SH)) return pk_bicg_kernel<T, VT, NT, RPT, MODE, false, sizeof(T) == 4>; \
  }

}  // namespace gko
