// sc_fixed.cuh -- finite-difference sums in aligned integers.
//
// The FP64 pipe of this GPU starts about 2 operations per SM and clock, its
// integer pipes about 110 (measured: 60.9 IADD3 and 61.0 IMAD per SM and
// clock, on two pipes that run side by side, beside FP64 instructions too).  A
// finite-difference stencil has small integer weights, so its sum needs no
// floating point until the end: the stencil's values are aligned to the
// exponent of the largest of them, as signed integers with 2 (4th order) or 6
// (8th order) bits below that value's last place, summed exactly, and the sum
// is rounded once on its way back to FP64.  The alignment drops what lies
// below 2^-54 (2^-58) of the stencil's own largest value, always downwards, so
// that its mean cancels in sums whose weights add up to zero; the halves of an
// 8th-order sum are joined at 2^-47 of its largest term or less.  A chain of FP64
// additions instead rounds every partial sum at 2^-53 of its size, which the
// weights make several (8th order: thousands of) times the largest value.
// The result depends on the stencil's values alone, not on tiles or boxes.
//
// Stencils that hold an infinity or a NaN, or whose largest value lies near
// either end of the exponent range, are left to the FP64 form (aligned_ok).
#pragma once

#include "sc_internal.h"

namespace sc {

// An unpacked value: the signed mantissa (hi, lo), shifted up by the guard
// bits (floor(-m) - 1 ulp of the guard bits for negative values), and the
// biased exponent in place (bits 20..30 of the high word).
struct Fx {
  int hi;
  unsigned lo;
  int t;
};

template <int GUARD>
__device__ __forceinline__ Fx fx_unpack(double v) {
  const int h = __double2hiint(v);
  const unsigned l = (unsigned)__double2loint(v);
  const int s = h >> 31;
  Fx r;
  r.t = h & 0x7ff00000;
  r.hi = (int)__funnelshift_l(l, (unsigned)((h & 0xfffff) | 0x100000), GUARD) ^ s;
  r.lo = (l << GUARD) ^ (unsigned)s;
  return r;
}

// The exponent field of a value, in place.
__device__ __forceinline__ int fx_exp(double v) { return __double2hiint(v) & 0x7ff00000; }

// The value in units of 2^(exponent of E - 52 - GUARD), rounded down.  E is at
// least the value's own t.  (PTX defines shr.s64 for every count: 64 and more
// give the sign, which is how zeros and denormals, t = 0, become 0 or -1.)
__device__ __forceinline__ long long fx_align(const Fx& f, int E) {
  const long long x = ((long long)f.hi << 32) | f.lo;
  long long r;
  asm("shr.s64 %0, %1, %2;" : "=l"(r) : "l"(x), "r"((E - f.t) >> 20));
  return r;
}

// Whether stencils whose largest value has exponent field E may be summed in
// integers: every alignment shift of a zero is 64 or more, and the result's
// exponent stays inside the normal range whatever the sum.
__device__ __forceinline__ bool aligned_ok(int E) { return (unsigned)(E - (120 << 20)) <= (unsigned)(1880 << 20); }

// A value that several stencils will read, unpacked once: the signed mantissa in
// the high 54 bits, and in the low 10 the exponent less 512 (0 for what is
// smaller, 1023 for what is larger, an infinity or a NaN).
__device__ __forceinline__ long long fx_pack(double v) {
  const int h = __double2hiint(v);
  const unsigned l = (unsigned)__double2loint(v);
  const int t = min(max(((h >> 20) & 0x7ff) - 512, 0), 1023);
  const unsigned mh = (unsigned)((h & 0xfffff) | 0x100000);
  const long long x = (long long)(((unsigned long long)__funnelshift_l(l, mh, 10) << 32) | (l << 10)), s = h >> 31;
  return ((x ^ s) - s) | t;
}
__device__ __forceinline__ int fx_pexp(long long p) { return (int)p & 1023; }
// The same as fx_align(fx_unpack<GUARD>) of a packed value.
template <int GUARD>
__device__ __forceinline__ long long fx_palign(long long p, int E) {
  long long r;
  asm("shr.s64 %0, %1, %2;" : "=l"(r) : "l"(p & ~1023ll), "r"(E + (10 - GUARD) - fx_pexp(p)));
  return r;
}
// As aligned_ok, for the largest packed exponent of a stencil.
__device__ __forceinline__ bool packed_ok(int E) { return (unsigned)(E - 120) <= 902u; }
__device__ __forceinline__ int packed_field(int E) { return (E + 512) << 20; }

// X units of 2^(exponent of E - 52 - GUARD + SHIFT), rounded to FP64.
template <int GUARD, int SHIFT>
__device__ __forceinline__ double fx_back(long long X, int E) {
  const double d = (double)X;
  const int h = __double2hiint(d);
  return __hiloint2double(h ? h + (E - ((1075 + GUARD - SHIFT) << 20)) : 0, __double2loint(d));
}

// 8th order: weighted sums (sums of weight magnitudes up to 98304) do not fit
// beside a 59-bit value in 64 bits, so the terms are cut into a low half, taken as
// signed, and a high half, and each half is summed by 32 x 32 + 64 bit
// multiply-adds: two instructions a term.  (Four 16-bit limbs summed in 32 bits
// took eight: the pass over 262,144 cells ran in 0.385 ms.)
struct FxWide {
  long long hh = 0, ll = 0;
  __device__ __forceinline__ void add(int w, long long x) {
    int l, h;
    asm("mov.b64 {%0, %1}, %2;" : "=r"(l), "=r"(h) : "l"(x));
    hh += (long long)w * (h + (int)((unsigned)l >> 31));
    ll += (long long)w * l;
  }
  // in units of 2^SHIFT, rounded down
  template <int SHIFT>
  __device__ __forceinline__ long long get() const {
    return (hh << (32 - SHIFT)) + (ll >> SHIFT);
  }
};

// The stencil sums of one order.  lo[m - 1], hi[m - 1] are the values at -m, m.
template <int ORD>
struct FxSums;

template <>
struct FxSums<4> {
  static constexpr int kGuard = 2;  // 53 + 2 bits, weights of the Kreiss-Oliger sum 192 < 2^8
  using Val = long long;
  __device__ static __forceinline__ Val val(double v, int E) { return fx_align(fx_unpack<kGuard>(v), E); }
  // 8 (v_1 - v_-1) - (v_2 - v_-2) = 12 h u'
  __device__ static __forceinline__ double first(const Val* lo, const Val* hi, int E) {
    return fx_back<kGuard, 0>(((hi[0] - lo[0]) << 3) + (lo[1] - hi[1]), E);
  }
  // 16 p1 - p2 - 30 u0 = 12 h^2 u'', pm = v_m + v_-m
  __device__ static __forceinline__ double second(const Val* p, Val u0, int E) {
    return fx_back<kGuard, 0>((p[0] << 4) - p[1] - ((u0 << 5) - (u0 << 1)), E);
  }
  // the three second derivatives' sum, Pm the sum over the six neighbours at distance m (weights: 192)
  __device__ static __forceinline__ double laplacian(const Val* P, Val u0, int E) {
    return fx_back<kGuard, 0>((P[0] << 4) - P[1] - 90 * u0, E);
  }
  // P3 - 6 P2 + 15 P1 - 60 u0, Pm the sum over the six neighbours at distance m
  __device__ static __forceinline__ double ko(Val P1, Val P2, Val P3, Val u0, int E) {
    const Val u60 = (u0 << 6) - (u0 << 2);
    return fx_back<kGuard, 0>(((P1 << 4) - P1) - ((P2 << 2) + (P2 << 1)) + P3 - u60, E);
  }
};

template <>
struct FxSums<8> {
  static constexpr int kGuard = 6;  // 59 bits: sums of six values and their halves stay in range
  using Val = long long;
  __device__ static __forceinline__ Val val(double v, int E) { return fx_align(fx_unpack<kGuard>(v), E); }
  // 672 d1 - 168 d2 + 32 d3 - 3 d4 = 840 h u', dm = v_m - v_-m (weights: 1750 < 2^11)
  __device__ static __forceinline__ double first(const Val* lo, const Val* hi, int E) {
    FxWide s;
    s.add(672, hi[0] - lo[0]);
    s.add(-168, hi[1] - lo[1]);
    s.add(32, hi[2] - lo[2]);
    s.add(-3, hi[3] - lo[3]);
    return fx_back<kGuard, 8>(s.get<8>(), E);
  }
  // 8064 p1 - 1008 p2 + 128 p3 - 9 p4 - 14350 u0 = 5040 h^2 u'' (weights: 2^15)
  __device__ static __forceinline__ double second(const Val* p, Val u0, int E) {
    FxWide s;
    s.add(8064, p[0]);
    s.add(-1008, p[1]);
    s.add(128, p[2]);
    s.add(-9, p[3]);
    s.add(-14350, u0);
    return fx_back<kGuard, 12>(s.get<12>(), E);
  }
  // the three second derivatives' sum, Pm the sum over the six neighbours at distance m (weights: 98304)
  __device__ static __forceinline__ double laplacian(const Val* P, Val u0, int E) {
    FxWide s;
    s.add(8064, P[0]);
    s.add(-1008, P[1]);
    s.add(128, P[2]);
    s.add(-9, P[3]);
    s.add(-43050, u0);
    return fx_back<kGuard, 14>(s.get<14>(), E);
  }
  // (weights: 192)
  __device__ static __forceinline__ double ko(Val P1, Val P2, Val P3, Val u0, int E) {
    FxWide s;
    s.add(15, P1);
    s.add(-6, P2);
    s.add(1, P3);
    s.add(-60, u0);
    return fx_back<kGuard, 5>(s.get<5>(), E);
  }
};

}  // namespace sc
