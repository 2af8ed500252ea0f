// Check and clock of the single-launch solvers' exchanges (persist.cuh): a
// kernel of nothing but steps, whose totals, published vectors and slot words
// are compared with what they must be, and in which one block can be made to
// leave early, as one whose wait ran out does, so that the others' waits run
// out.
#include "persist_gmres.cuh"

namespace gko {
namespace {

constexpr int kExThreads = 64;

struct ExArgs {
  int values, steps;
  int leave_block, leave_step;  // -1: none
  long long wait;   // limit of a wait, clock cycles
  int* err;
  ulonglong2 *slots, *sums, *totals;
  double* vec;      // kExThreads per block
  int* out;         // per block: steps done, wrong values, stale words, gave up
  long long* cycles;
  int* gave_up;
};

template <int MODE>
__global__ void __launch_bounds__(kExThreads) exchange_kernel(ExArgs a) {
  constexpr int NT = kExThreads;
  __shared__ PkShared<NT, MODE> sh;
  __shared__ double own[NT];
  __shared__ PkGmresShared<NT> gs;
  const int G = gridDim.x, me = blockIdx.x, tid = threadIdx.x, peer = (me + 1) % G;
  pk_open(sh, a.gave_up);
  unsigned seq = 0;
  int wrong = 0, stale = 0, s = 0;
  const double N = (double)G * NT, mine = (double)(me * NT + tid + 1), sum = 0.5 * N * (N + 1.0);
  double want[3];
  // one step of NV values: value k is (k + 1) (row + 1) + s, whose sum is exact
  auto step = [&](auto nv) -> bool {
    constexpr int NV = decltype(nv)::value;
    double v[3] = {mine + s, 2.0 * mine + s, 3.0 * mine + s};
    if (NV == 0) {
      if (MODE == kPkCluster) own[tid] = mine + s;
      else __stcg(a.vec + me * NT + tid, mine + s);
    }
    const bool ok = pk_step<NT, MODE, NV == 0 ? kPubVec : kPubNone, NV>(
        v, sh, a.slots, a.err, seq, [&](const auto& t, double*) {
          for (int k = 0; k < NV; ++k) wrong += t[k] != want[k];
        }, [&] {
          for (int k = 0; k < NV; ++k) want[k] = __fma_rn((double)s, N, (k + 1) * sum);
        }, a.wait);
    if (ok && NV == 0) {
      const double got = MODE == kPkCluster ? pk_ld_peer(pk_mapa(pk_smem(own + tid), peer), 0.0)
                                            : __ldcg(a.vec + peer * NT + tid);
      wrong += got != (double)(peer * NT + tid + 1) + s;
      // read before it is overwritten
      return pk_step<NT, MODE, kPubVec, 0>(nullptr, sh, a.slots, a.err, seq, [](const double (&)[1], double*) {},
                                           PkNothing{}, a.wait);
    }
    return ok;
  };
  auto some = [&](int values) -> bool {
    switch (values) {
      case 0: return step(std::integral_constant<int, 0>{});
      case 1: return step(std::integral_constant<int, 1>{});
      case 2: return step(std::integral_constant<int, 2>{});
      default: return step(std::integral_constant<int, 3>{});
    }
  };
  const long long t0 = clock64();
  bool ok = true;
  for (; ok && s < a.steps; s += ok) ok = !(me == a.leave_block && s == a.leave_step) && some(a.values);
  if (me == 0 && tid == 0) *a.cycles = clock64() - t0;
  const int done = s;
  // every word carries the tag of its slot's last step, however few values that had
  for (int k : {3, 3, 1, 1}) ok = ok && some(k);
  const unsigned last = seq;
  ok = ok && pk_step<NT, MODE, kPubGlobal, 0>(nullptr, sh, a.slots, a.err, seq, [](const double (&)[1], double*) {});
  if (ok && tid < G) {
    const ulonglong2* slot = MODE == kPkCluster
                                 ? &sh.slots[last & 1u][tid][0]
                                 : a.slots + (size_t)(last & 1u) * kPkMaxBlocks * kPkSlot + tid * kPkSlot;
    for (int k = 0; k < kPkWords; ++k) stale += !pk_tagged(MODE == kPkCluster ? pk_get_own(pk_smem(slot + k)) : pk_get(slot + k), last);
  }
  if constexpr (MODE != kPkCluster) {  // the gather's words after a cycle's first gather
    if (ok) {
      for (int i = tid; i < 32 * (NT / 32); i += NT) gs.part[i / (NT / 32)][i % (NT / 32)] = Fx{0, 1};
      __syncthreads();
      ok = pk_gather_sums<NT>(2, true, gs, a.sums, a.totals, a.err, seq);
      const unsigned tag = seq;
      ok = ok && pk_step<NT, MODE, kPubGlobal, 0>(nullptr, sh, a.slots, a.err, seq, [](const double (&)[1], double*) {});
      if (ok && tid < 32) {
        stale += !pk_tagged(pk_get(a.sums + (size_t)(tag & 1u) * 32 * kPkMaxBlocks + (size_t)tid * kPkMaxBlocks + peer), tag);
        stale += !pk_tagged(pk_get(a.totals + (size_t)(tag & 1u) * 32 * 2 + 2 * tid), tag);
      }
    }
  }
  atomicAdd(a.out + 4 * me + 1, wrong);
  atomicAdd(a.out + 4 * me + 2, stale);
  if (tid == 0) {
    a.out[4 * me] = done;
    a.out[4 * me + 3] = !ok;
  }
  pk_leave(sh, !ok, a.gave_up);
}

}  // namespace
}  // namespace gko

using namespace gko;

extern "C" int gko_diag_exchange(int32_t cluster, int32_t blocks, int32_t values, int32_t steps, int32_t leave_block,
                                 int32_t leave_step, int64_t wait_cycles, int32_t* out, double* cycles_per_step,
                                 void* stream) {
  if (blocks < 2 || blocks > (cluster ? kPkCluster16 : std::min(sm_count(), kPkMaxBlocks)) || values < 0 ||
      values > kPkWords || steps < 1 || steps > 1000000 || leave_block >= blocks || wait_cycles < 0 || wait_cycles > kPkWait || !out || !cycles_per_step)
    return fail(GKO_INVALID_ARG, "bad exchange check arguments");
  cudaStream_t s = (cudaStream_t)stream;
  const size_t slots = 2 * kPkMaxBlocks * kPkSlot, sums = 2 * 32 * kPkMaxBlocks, totals = 2 * 32 * 2;
  const size_t words = slots + sums + totals;
  Scratch mem;
  const size_t bytes = sizeof(ulonglong2) * words + sizeof(long long) + sizeof(double) * kExThreads * blocks +
                       sizeof(int) * (4 * blocks + 1) + 2048;
  GKO_TRY(mem.get(bytes, s));
  GKO_TRY_CUDA(cudaMemsetAsync(mem.data(), 0, bytes, s));
  Carve cv{static_cast<char*>(mem.data())};
  ExArgs a{};
  a.values = values;
  a.steps = steps;
  a.leave_block = leave_block;
  a.leave_step = leave_step;
  a.wait = wait_cycles ? wait_cycles : kPkWait;
  a.err = device_error_word();
  a.slots = cv.take<ulonglong2>(words);
  a.sums = a.slots + slots;
  a.totals = a.sums + sums;
  a.cycles = cv.take<long long>(1);
  a.vec = cv.take<double>((size_t)kExThreads * blocks);
  a.gave_up = cv.take<int>(1);
  a.out = cv.take<int>((size_t)4 * blocks);
  auto kern = cluster ? exchange_kernel<kPkCluster> : exchange_kernel<kPkGrid>;
  cudaLaunchConfig_t cfg = {};
  cfg.gridDim = dim3((unsigned)blocks);
  cfg.blockDim = dim3(kExThreads);
  cfg.stream = s;
  cudaLaunchAttribute at[1];
  if (cluster) {
    if (blocks > 8) GKO_TRY_CUDA(cudaFuncSetAttribute(kern, cudaFuncAttributeNonPortableClusterSizeAllowed, 1));
    at[0].id = cudaLaunchAttributeClusterDimension;
    at[0].val.clusterDim.x = (unsigned)blocks;
    at[0].val.clusterDim.y = at[0].val.clusterDim.z = 1;
  } else {
    at[0].id = cudaLaunchAttributeCooperative;
    at[0].val.cooperative = 1;
  }
  cfg.attrs = at;
  cfg.numAttrs = 1;
  GKO_TRY_CUDA(cudaLaunchKernelEx(&cfg, kern, a));
  long long cycles = 0;
  GKO_TRY_CUDA(cudaMemcpyAsync(out, a.out, sizeof(int) * 4 * blocks, cudaMemcpyDeviceToHost, s));
  GKO_TRY_CUDA(cudaMemcpyAsync(&cycles, a.cycles, sizeof(cycles), cudaMemcpyDeviceToHost, s));
  GKO_TRY_CUDA(cudaStreamSynchronize(s));
  *cycles_per_step = (double)cycles / steps;
  return GKO_OK;
}
