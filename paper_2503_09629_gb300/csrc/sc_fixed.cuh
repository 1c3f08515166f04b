// sc_fixed.cuh -- finite-difference sums in aligned integers.
//
// The FP64 pipe of this GPU starts about 2 operations per SM and clock, its
// integer pipes about 110 (measured: 60.9 IADD3 and 61.0 IMAD per SM and
// clock, on two pipes that run side by side, beside FP64 instructions too).  A
// finite-difference stencil has small integer weights, so its sum needs no
// floating point until the end: the values are aligned to the exponent of the largest
// of them, as signed integers with some bits below that value's last place,
// summed exactly, and the sum is rounded once on its way back to FP64.  The
// alignment drops what lies below the last of these bits, always downwards, so
// that its mean cancels in sums whose weights add up to zero.
//
// What is aligned together is what the sum weighs: the values along one axis for
// its derivatives, all of the star for its Laplacian and the Kreiss-Oliger sum.  At
// 4th order the weights multiply before the alignment cuts, or the weighted
// values keep more bits, so that a sum's error is a few units of its smallest
// weight: at most 2^-49 of the sum of its weighted values' magnitudes (8th order:
// 2^-48; RMS errors are some 2^-53 of the largest value).  At 8th order the weights
// are too far apart for that (1 to 8192), and sums whose lightly weighted outer
// values are 2^3 to 2^5 times the inner ones are left to FP64, whose error
// is relative to the weighted values (kExcess1 and so on; inside these limits the
// integer sums were the more accurate ones: on random values 1.4e-16 against
// 2.3e-14 for a Laplacian of 4th order, 4.7e-17 against 2.8e-14 of 8th).
// The result depends on the stencil's values alone, not on tiles or boxes.
//
// Stencils that hold an infinity or a NaN, or whose largest value lies near either
// end of the exponent range are left to the FP64 form too (aligned_ok,
// packed_ok), unless they are all zeros (zero_bits), as fields at rest are.
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

// Zero for zeros of either sign only.
__device__ __forceinline__ unsigned zero_bits(double v) {
  return (unsigned)__double2hiint(v) << 1 | (unsigned)__double2loint(v);
}
// The exponent field of a value, in place.
__device__ __forceinline__ int fx_exp(double v) { return __double2hiint(v) & 0x7ff00000; }

// (PTX defines shr.s64 for every count: 64 and more give the sign.)
__device__ __forceinline__ long long fx_shift(long long x, int n) {
  long long r;
  asm("shr.s64 %0, %1, %2;" : "=l"(r) : "l"(x), "r"(n));
  return r;
}

// The value in units of 2^(exponent of E - 52 - GUARD), rounded down.  E is at
// least the value's own t.  (Shifts of 64 and more are how zeros and denormals,
// t = 0, become 0 or -1.)
__device__ __forceinline__ long long fx_align(const Fx& f, int E) {
  return fx_shift(((long long)f.hi << 32) | f.lo, (E - f.t) >> 20);
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
// The same for a packed value (a negative one that loses no bits comes out as it is,
// where fx_unpack's is one unit lower).
template <int GUARD>
__device__ __forceinline__ long long fx_palign(long long p, int E) {
  return fx_shift(p & ~1023ll, E + (10 - GUARD) - fx_pexp(p));
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
  // One axis of a star: by how many powers of two its largest value, u0 or one at +-3, may
  // exceed those at +-1 and those at +-2 (one of the two; RMS error of the first
  // derivative 0.07 units of 2^-53 of the largest, FP64: 3.3 of v_1 or 0.5 of v_2).
  static constexpr int kExcess1 = 4, kExcess2 = 2;
  static constexpr int kLaplacianExcess = 1023;
  // 8 (v_1 - v_-1) - (v_2 - v_-2) = 12 h u'
  __device__ static __forceinline__ double first(const double* lo, const double* hi, int E) {
    const long long l0 = fx_align(fx_unpack<7>(lo[0]), E), h0 = fx_align(fx_unpack<7>(hi[0]), E);
    const long long l1 = fx_align(fx_unpack<4>(lo[1]), E), h1 = fx_align(fx_unpack<4>(hi[1]), E);
    return fx_back<4, 0>((h0 - l0) + (l1 - h1), E);
  }
  // Packed values of one axis, E their largest exponent (u0's among them), with 4 bits
  // below the last place: 12 h u', 12 h^2 u'' = 16 p1 - p2 - 30 u0 (pm = v_m + v_-m) and the axis's share
  // 15 p1 - 6 p2 + p3 - 20 u0 of the Kreiss-Oliger sum.  Weights up to 64, 63 bits.
  struct Axis {
    long long a, b, c, u10;
    long long d;  // 8 (v_1 - v_-1) - (v_2 - v_-2)
    __device__ __forceinline__ Axis(const long long* lo, const long long* hi, long long u0, int E) {
      const long long l0 = fx_palign<7>(lo[0], E), h0 = fx_palign<7>(hi[0], E);
      const long long l1 = fx_palign<4>(lo[1], E), h1 = fx_palign<4>(hi[1], E);
      const long long x = u0 >> 10;  // 160 x: u0 times 10
      a = l0 + h0;                   // 8 p1
      b = l1 + h1;
      c = fx_palign<4>(lo[2], E) + fx_palign<4>(hi[2], E);
      d = (h0 - l0) + (l1 - h1);
      u10 = fx_shift((x << 7) + (x << 5), E - fx_pexp(u0));
    }
    __device__ __forceinline__ double first(int Ef) const { return fx_back<4, 0>(d, Ef); }
    __device__ __forceinline__ double second(int Ef) const { return fx_back<4, 0>((a << 1) - b - ((u10 << 1) + u10), Ef); }
    __device__ __forceinline__ long long ko() const {
      const long long p1 = a >> 3;
      return ((p1 << 4) - p1) - ((b << 2) + (b << 1)) + c - (u10 << 1);
    }
  };
  // The Kreiss-Oliger sum from the axes' shares; E: the star's largest exponent, Ed: the axis's.
  struct Ko {
    long long s = 0;
    __device__ __forceinline__ void add(const Axis& A, int Ed, int E) { s += fx_shift(A.ko(), E - Ed + 2); }
    __device__ __forceinline__ double get(long long, int E) const { return fx_back<4, 2>(s, packed_field(E)); }
  };
  // 12 h^2 times the Laplacian: 16 P1 - P2 - 90 u0, Pm the sum over the six neighbours at distance
  // m, v[m - 1]: packed values, E their largest exponent (weights 192, 2 bits below the last place: 63 bits)
  __device__ static __forceinline__ double laplacian(const long long (*v)[6], long long u0, int E) {
    const long long x = u0 >> 10;  // 360 x: u0 times 90
    long long s = -fx_shift((x << 8) + (x << 6) + (x << 5) + (x << 3), E - fx_pexp(u0));
#pragma unroll
    for (int q = 0; q < 6; ++q) s += fx_palign<6>(v[0][q], E) - fx_palign<2>(v[1][q], E);
    return fx_back<2, 0>(s, packed_field(E));
  }
};

template <>
struct FxSums<8> {
  static constexpr int kGuard = 6;  // 59 bits: sums of six values and their halves stay in range
  // As at 4th order, with the outer values of the derivative itself (+-3, +-4, weights 32 and 3
  // against 672 and 168): 9 units of 2^-53 of the largest, FP64: 270 of v_1 or 67 of v_2.
  static constexpr int kExcess1 = 4, kExcess2 = 3;
  // Values at +-2, +-3, +-4 (1008, 128, 9) against u0 and those at +-1 (43050, 8064):
  // 430 2^-53 against 2e4 2^-53.
  static constexpr int kLaplacianExcess = 5;
  // 672 d1 - 168 d2 + 32 d3 - 3 d4 = 840 h u', dm = v_m - v_-m (weights: 1750 < 2^11)
  __device__ static __forceinline__ double first_of(const long long* l, const long long* h, int Ef) {
    FxWide s;
    s.add(672, h[0] - l[0]);
    s.add(-168, h[1] - l[1]);
    s.add(32, h[2] - l[2]);
    s.add(-3, h[3] - l[3]);
    return fx_back<kGuard, 8>(s.get<8>(), Ef);
  }
  __device__ static __forceinline__ double first(const double* lo, const double* hi, int E) {
    long long l[4], h[4];
#pragma unroll
    for (int m = 0; m < 4; ++m) {
      l[m] = fx_align(fx_unpack<kGuard>(lo[m]), E);
      h[m] = fx_align(fx_unpack<kGuard>(hi[m]), E);
    }
    return first_of(l, h, E);
  }
  struct Axis {
    long long l[4], h[4], u0;
    __device__ __forceinline__ Axis(const long long* lo, const long long* hi, long long u, int E) {
#pragma unroll
      for (int m = 0; m < 4; ++m) {
        l[m] = fx_palign<kGuard>(lo[m], E);
        h[m] = fx_palign<kGuard>(hi[m], E);
      }
      u0 = fx_palign<kGuard>(u, E);
    }
    __device__ __forceinline__ double first(int Ef) const { return first_of(l, h, Ef); }
    // 8064 p1 - 1008 p2 + 128 p3 - 9 p4 - 14350 u0 = 5040 h^2 u'' (weights: 2^15)
    __device__ __forceinline__ double second(int Ef) const {
      FxWide s;
      s.add(8064, l[0] + h[0]);
      s.add(-1008, l[1] + h[1]);
      s.add(128, l[2] + h[2]);
      s.add(-9, l[3] + h[3]);
      s.add(-14350, u0);
      return fx_back<kGuard, 12>(s.get<12>(), Ef);
    }
  };
  // (weights: 192)
  struct Ko {
    long long P[3] = {0, 0, 0};
    __device__ __forceinline__ void add(const Axis& A, int Ed, int E) {
#pragma unroll
      for (int m = 0; m < 3; ++m) P[m] += fx_shift(A.l[m] + A.h[m], E - Ed);
    }
    __device__ __forceinline__ double get(long long u0, int E) const {
      FxWide s;
      s.add(15, P[0]);
      s.add(-6, P[1]);
      s.add(1, P[2]);
      s.add(-60, fx_palign<kGuard>(u0, E));
      return fx_back<kGuard, 5>(s.get<5>(), packed_field(E));
    }
  };
  // 5040 h^2 times the Laplacian (weights: 98304)
  __device__ static __forceinline__ double laplacian(const long long (*v)[6], long long u0, int E) {
    long long P[4];
#pragma unroll
    for (int m = 0; m < 4; ++m) {
      P[m] = fx_palign<kGuard>(v[m][0], E);
#pragma unroll
      for (int q = 1; q < 6; ++q) P[m] += fx_palign<kGuard>(v[m][q], E);
    }
    FxWide s;
    s.add(8064, P[0]);
    s.add(-1008, P[1]);
    s.add(128, P[2]);
    s.add(-9, P[3]);
    s.add(-43050, fx_palign<kGuard>(u0, E));
    return fx_back<kGuard, 14>(s.get<14>(), packed_field(E));
  }
};

}  // namespace sc
