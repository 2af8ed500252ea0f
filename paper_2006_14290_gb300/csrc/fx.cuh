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

// Sum of N <= 8 products a[i] * b[i] of FP32 numbers, exact like the FP64
// products would be (24 x 24 = 48 bits), added on the scale of the largest:
// about 25 integer instructions a product instead of two widenings and an
// FP64 FMA, whose 16 cycles of the SM's one FP64 pipe are its cost.  FP32
// subnormals count as zero (as in widen); infinities and NaN go through FP64.
template <int N>
__device__ __forceinline__ Fx fx_dot(const float (&a)[N], const float (&b)[N]) {
  static_assert(N <= 8, "eight 60-bit products");
  long long x[N];
  unsigned e[N], E = 1u << 23, top = 0u;
#pragma unroll
  for (int i = 0; i < N; ++i) {
    const unsigned ua = __float_as_uint(a[i]), ub = __float_as_uint(b[i]);
    const unsigned fa = ua & 0x7f800000u, fb = ub & 0x7f800000u;
    top = max(top, max(fa, fb));
    const bool zero = min(fa, fb) == 0u;
    const int s = (int)(ua ^ ub) >> 31;
    int ma = (int)(((ua << 5) & 0x0fffffe0u) | 0x10000000u);  // 24 bits, up by 5
    ma = zero ? 0 : (ma ^ s) - s;
    x[i] = (long long)ma * (int)(((ub << 7) & 0x3fffff80u) | 0x40000000u);  // 24 bits, up by 7
    e[i] = zero ? 0u : fa + fb;
    E = max(E, e[i]);
  }
  if (top == 0x7f800000u) {
    double s = 0.0;
#pragma unroll
    for (int i = 0; i < N; ++i) s = __fma_rn(widen(a[i]), widen(b[i]), s);
    return fx_of(s);
  }
  long long s = 0;
#pragma unroll
  for (int i = 0; i < N; ++i) s += x[i] >> min((E - e[i]) >> 23, 63u);
  // m 2^(e - 300) = (m 2^12) 2^(e - 312)
  return Fx{s, (int)(E >> 23) - 312 + kFxBias};
}

// a / b, b != 0: reciprocal estimate, one Newton-Raphson step (40 correct
// bits), quotient and one correction of it with its exact residual (Markstein,
// IBM J. Res. Dev. 34, 1990), which leaves about the rounding error of the
// quotient: 5 dependent FP64 operations of 67 cycles instead of 552 cycles of
// IEEE division, on the critical path of every iteration.  Operands whose
// estimate or residual could leave the normal range divide as usual.
__device__ __forceinline__ double fast_div(double a, double b) {
  const unsigned eb = ((unsigned)__double2hiint(b) >> 20) & 0x7ffu, ea = ((unsigned)__double2hiint(a) >> 20) & 0x7ffu;
  if (eb - 523u > 1000u || ea - 523u > 1000u) return a / b;  // exponents outside 2^-500 .. 2^500
  double r;
  asm("rcp.approx.ftz.f64 %0, %1;" : "=d"(r) : "d"(b));
  r = __fma_rn(r, __fma_rn(-b, r, 1.0), r);
  const double q = a * r;
  return __fma_rn(r, __fma_rn(-b, q, a), q);
}

// The float pair of an FP64 scalar (Lin<float>: hi = a rounded to FP32, lo =
// what is left, rounded) in integer operations: about 110 cycles on the
// critical path of a step instead of 365 for the conversions and the FP64
// subtraction.  Scalars outside 2^-60 .. 2^120 convert as usual.
__device__ __forceinline__ Lin<float> lin_of(double a) {
  const unsigned h = (unsigned)__double2hiint(a);
  const unsigned e = (h >> 20) & 0x7ffu;
  if (e - 963u > 180u) return Lin<float>(a);
  const long long m = (long long)(((unsigned long long)__double_as_longlong(a) & 0xfffffffffffffull) | (1ull << 52));
  const unsigned top = (unsigned)((m + (1ll << 28)) >> 29);  // 24 bits, or 2^24
  const int rest = (int)(m - ((long long)top << 29));
  const unsigned sign = h & 0x80000000u;
  const float lo = __int2float_rn(rest);  // times 2^(e - 1075)
  const unsigned lb = rest ? __float_as_uint(lo) + ((e - 1075u) << 23) : 0u;
  return Lin<float>(__uint_as_float(sign | (((e - 896u) << 23) + (top - (1u << 23)))), __uint_as_float(lb ^ sign));
}

}  // namespace gko
