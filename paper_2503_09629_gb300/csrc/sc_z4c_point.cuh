// sc_z4c_point.cuh -- the Z4c right-hand side and constraints at one cell.
//
// FP64 is the scarce resource on this GPU (2 operations per SM and clock), the
// integer pipes stand idle beside it.  So the sums of products over tensor
// indices whose operands or results are used many times over (Christoffel symbols,
// the quadratic part of the Ricci tensor, At with raised indices) are formed in
// integers, all else in FP64.
//
// A number is an integer and an exponent of its own (FxN, 60 bits).  The terms
// of a sum of products are aligned to the largest of them (fx_dot): one operand
// of a product is shifted right by what the product lies below the largest one,
// then a product is three 32 x 32 + 64 bit multiply-adds into two accumulators.
// What the shifts and the dropped low x low parts lose is below 2^-54 of the
// sum's own largest term for each product; a chain of FP64 operations rounds at
// 2^-53 of its partial sum for each.  Nothing is scaled by what other components
// hold, so metrics stretched along an axis and components many orders smaller
// than their neighbours keep their accuracy.
// (One exponent per tensor needs no shifts and ran the stage in 0.269 ms in place
// of 0.327 for 262,144 cells, but its error is relative to the tensor's largest
// component: 3e-6 in the right-hand side of At_xx for gt_xx = 1e4 gt_yy, 3e-9 in that
// of gt_xy for off-diagonal components 1e-8 times the diagonal ones.)
//
// Cells that hold a value the integers do not take (an infinity, a NaN, a
// subnormal number, or a result outside the range of normal doubles) have the
// same sums in FP64 (z4c_connection_fp64).
#pragma once

#include "sc_internal.h"

#include <cmath>
#include <cstring>

namespace sc {

// scratch slots of the derivative pass
constexpr int Q_D1 = 0;    // 3 * f + d: first derivative of field f along d
constexpr int Q_D2 = 66;   // 6 * s + p: second derivative, s = slot (W, gt x6, alpha, beta x3), p = xx,xy,xz,yy,yz,zz
constexpr int Q_KO = 132;  // f: sum_d delta_d^6 u_f (unscaled)

#ifdef __CUDACC__
#define FXD __host__ __device__ __forceinline__
#define FX_NOINLINE __host__ __device__ __noinline__
#else
#define FXD inline
#define FX_NOINLINE inline
using std::fma;
#endif

// symmetric index helpers: xx xy xz yy yz zz
FXD constexpr int sidx(int i, int j) {
  return (i == j) ? (i == 0 ? 0 : (i == 1 ? 3 : 5)) : (i + j == 1 ? 1 : (i + j == 2 ? 2 : 4));
}
FXD constexpr bool fx_pure(int s) { return s == 0 || s == 3 || s == 5; }

FXD int fx_dhi(double v) {
#ifdef __CUDA_ARCH__
  return __double2hiint(v);
#else
  long long b;
  std::memcpy(&b, &v, 8);
  return (int)(b >> 32);
#endif
}
FXD unsigned fx_dlo(double v) {
#ifdef __CUDA_ARCH__
  return (unsigned)__double2loint(v);
#else
  long long b;
  std::memcpy(&b, &v, 8);
  return (unsigned)b;
#endif
}
FXD double fx_make(int hi, int lo) {
#ifdef __CUDA_ARCH__
  return __hiloint2double(hi, lo);
#else
  const long long b = (long long)(((unsigned long long)(unsigned)hi << 32) | (unsigned)lo);
  double v;
  std::memcpy(&v, &b, 8);
  return v;
#endif
}
// x >> n, n >= 0 of any size (64 and more give the sign, as PTX defines it)
FXD long long fx_shr(long long x, int n) {
#ifdef __CUDA_ARCH__
  long long r;
  asm("shr.s64 %0, %1, %2;" : "=l"(r) : "l"(x), "r"(n));
  return r;
#else
  return x >> (n > 63 ? 63 : n);
#endif
}
FXD long long fx_shl(long long x, int n) { return (long long)((unsigned long long)x << n); }
FXD int fx_clz(int x) {
#ifdef __CUDA_ARCH__
  return __clz(x);
#else
  return x ? __builtin_clz((unsigned)x) : 32;
#endif
}
FXD int fx_max(int a, int b) { return a > b ? a : b; }

// A multiplication operand: h * 2^32 + l, the low half signed so that every
// partial product is a signed 32 x 32 multiplication.
struct FxP {
  int h, l;
};
// (As 32-bit shifts of x the compiler would widen the halves again in products,
// and a 32 x 32 multiplication would become a 64 x 64 one.)
FXD FxP fx_split(long long x) {
  FxP r;
#ifdef __CUDA_ARCH__
  asm("mov.b64 {%0, %1}, %2;" : "=r"(r.l), "=r"(r.h) : "l"(x));
#else
  r.l = (int)x;
  r.h = (int)(x >> 32);
#endif
  r.h += (int)((unsigned)r.l >> 31);
  return r;
}

// A sum of products: hh * 2^64 + mm * 2^32, the low x low parts (at most 2^62
// each, signed) dropped.
struct FxDot {
  long long hh = 0, mm = 0;
  FXD void mac(const FxP& a, const FxP& b) {
    hh += (long long)a.h * b.h;
    mm += (long long)a.h * b.l;
    mm += (long long)a.l * b.h;
  }
  // in units of 2^K, 60 <= K <= 62, rounded down
  template <int K>
  FXD long long fin() const {
    return fx_shl(hh, 64 - K) + (mm >> (K - 32));
  }
};

// m * 2^e, |m| < 2^60 unless a comment says otherwise.  Zeros have an exponent far
// below all others, so that they do not count where terms are aligned.
struct FxN {
  long long m;
  int e;
};
// the same as the operand of a product that is not shifted
struct FxA {
  FxP v;
  int e;
};
FXD FxA fx_op(const FxN& n) { return FxA{fx_split(n.m), n.e}; }
FXD FxA fx_twice(const FxA& a) { return FxA{a.v, a.e + 1}; }
constexpr int kFxZero = -(1 << 14);
// What tells that a value is out of range: the largest exponent field loaded, and bits
// that stay zero if there are no subnormal numbers and no results out of range.
struct FxCheck {
  int largest = 0;
  unsigned bad = 0;
  FXD bool ok() const { return largest < 0x7ff && bad == 0; }
};

FXD FxN fx_load(double v, FxCheck& c) {
  const int h = fx_dhi(v), t = (h >> 20) & 0x7ff, s = h >> 31;
  const unsigned l = fx_dlo(v);
  unsigned mh = (unsigned)h & 0xfffff;
  int e = t - (1023 + 59);
  c.largest = fx_max(c.largest, t);
  if (t == 0) {
    c.bad |= mh | l;
    e = kFxZero;
  } else {
    mh |= 0x100000;
  }
  const long long x = (long long)(((unsigned long long)((mh << 7) | (l >> 25)) << 32) | (l << 7));
  return FxN{(x ^ s) - s, e};
}
// The largest bit of a sum below 2^63 moved to bit 59.  (A sum that vanishes in its
// high word moves by 28 places and stays short: its terms cancelled, and their
// errors are of that size.)
FXD FxN fx_norm(const FxN& n) {
  const int h = (int)(n.m >> 32), s = fx_clz(h ^ (h >> 31)) - 1;
  return FxN{fx_shl(n.m, s) >> 3, n.e - s + 3};
}
// a + b and a + b - c of numbers
FXD FxN fx_add(const FxN& a, const FxN& b) {
  const int E = fx_max(a.e, b.e) + 1;
  return FxN{fx_shr(a.m, E - a.e) + fx_shr(b.m, E - b.e), E};
}
FXD FxN fx_add_sub(const FxN& a, const FxN& b, const FxN& c) {
  const int E = fx_max(fx_max(a.e, b.e), c.e) + 2;
  return FxN{fx_shr(a.m, E - a.e) + fx_shr(b.m, E - b.e) - fx_shr(c.m, E - c.e), E};
}
// a + b for sums; their magnitudes add up
FXD FxN fx_acc(const FxN& a, const FxN& b) {
  const int E = fx_max(a.e, b.e);
  return FxN{fx_shr(a.m, E - a.e) + fx_shr(b.m, E - b.e), E};
}
// sum_i a_i b_i, i < N <= 9, below N * 2^60 (N > 6: N * 2^59) for K = 60
template <int N, int K = 60>
FXD FxN fx_dot(const FxA* a, const FxN* b) {
  constexpr int X = N > 6 ? 1 : 0;
  int e[N], E = a[0].e + b[0].e;
  e[0] = E;
#pragma unroll
  for (int i = 1; i < N; ++i) {
    e[i] = a[i].e + b[i].e;
    E = fx_max(E, e[i]);
  }
  FxDot d;
#pragma unroll
  for (int i = 0; i < N; ++i) d.mac(a[i].v, fx_split(fx_shr(b[i].m, E - e[i] + X)));
  return FxN{d.fin<K>(), E + X + K};
}
// rounded to FP64; sums of any size below 2^63
FXD double fx_double(const FxN& n, FxCheck& c) {
  const double d = (double)n.m;
  const int h = fx_dhi(d), t = h & 0x7ff00000;
  if (t == 0) return 0.0;
  c.bad |= (unsigned)((t >> 20) + n.e - 1) > 2045u;
  return fx_make((int)((unsigned)h + ((unsigned)n.e << 20)), (int)fx_dlo(d));
}

// One thread's numbers in shared memory, slot s of thread t at s * T + t: the
// rolled loops below index them at run time, which registers do not allow, and
// a warp's access to one slot is free of bank conflicts.
template <int T>
struct FxMem {
  long long* m;
  short* e;
  FXD FxN ld(int s) const { return FxN{m[s * T], e[s * T]}; }
  FXD void st(int s, const FxN& n) const {
    m[s * T] = n.m;
    e[s * T] = (short)fx_max(n.e, kFxZero);
  }
  FXD double ldd(int s) const { return reinterpret_cast<const double*>(m)[s * T]; }
  FXD void std(int s, double v) const { reinterpret_cast<double*>(m)[s * T] = v; }
  // slots of row i of a symmetric tensor in slots s0..s0 + 5
  FXD void row(int s0, int i, FxA* r) const {
    r[0] = fx_op(ld(s0 + i));
    r[1] = fx_op(ld(s0 + (i == 0 ? 1 : i + 2)));
    r[2] = fx_op(ld(s0 + (i == 0 ? 2 : i + 3)));
  }
};
// slot of a symmetric pair known at run time
FXD int fx_slot(int i, int j) {
  const int a = i < j ? i : j, b = i < j ? j : i;
  return a + b + (a > 0 ? 1 : 0);
}

// The derivatives are stored as stencil sums: a first derivative is 2 u times its
// sum, a mixed second one 4 u^2 times, a pure one `pure` u^2 times, u = 1 / (24 h) or
// 1 / (1680 h).  Sums over them are formed in units of u and u^2, in which the
// factors are whole numbers, and scaled where they enter an equation.
struct Z4cUnits {
  double u, iu, u2;        // u, 1 / u, u^2
  double s1, m2u, m2u2;    // 2 u, -2 u, -2 u^2
  double pure, mh_pure;    // 48 or 560, and -1/2 of it
  double tp, tm;           // a third of the scales of second derivatives
};
// Every scale is formed in a pair of doubles and rounded once: their errors are the
// same in every cell.  (Explicit FMAs, so that every host compiler gives the same values.)
struct FxPair {
  double h, l;
};
inline FxPair fx_pair_times(const FxPair& x, double k) {
  const double h = x.h * k;
  return FxPair{h, std::fma(x.l, k, std::fma(x.h, k, -h))};
}
inline Z4cUnits z4c_units(int order, double h) {
  const double w = order == 8 ? 840.0 : 12.0;
  const FxPair d = fx_pair_times(FxPair{h, 0.0}, 2.0 * w);
  FxPair u{1.0 / d.h, 0.0};
  u.l = u.h * std::fma(-u.h, d.l, std::fma(-u.h, d.h, 1.0));
  FxPair u2 = fx_pair_times(u, u.h);
  u2.l = std::fma(u.h, u.l, u2.l);
  auto third = [](const FxPair& x) {
    const double q = x.h / 3.0;
    return q + (std::fma(-q, 3.0, x.h) + x.l) / 3.0;
  };
  Z4cUnits c;
  c.u = u.h + u.l;
  c.iu = d.h + d.l;
  c.u2 = u2.h + u2.l;
  c.s1 = 2.0 * c.u;
  c.m2u = -2.0 * c.u;
  c.m2u2 = -2.0 * c.u2;
  c.pure = order == 8 ? 560.0 : 48.0;
  c.mh_pure = -0.5 * c.pure;
  c.tp = third(fx_pair_times(u2, c.pure));
  c.tm = third(fx_pair_times(u2, 4.0));
  return c;
}

// slots of one cell
enum {
  // while the integer sums run
  FM_GS = 0,   // Gamma_{k,ij}, 6 k + s
  FM_GU = 18,  // Gamma^k_ij, 6 k + s
  FM_Q = 36,   // as CN_Q
  // afterwards, as doubles in units of the power of u in brackets
  CN_GW = 0,   // Gamma^k_ij d_k W (u^2)
  CN_GD = 6,   // (Gamma_d)^k = gt^ij Gamma^k_ij (u)
  CN_WW = 9,   // gt^ij d_i W d_j W (u^2)
  CN_Q = 36,   // the quadratic part of the Ricci tensor and gt_k(i d_j) Gamt^k (u^2)
  // for the constraints
  CN_GU = 18,  // Gamma^k_ij (u)
  // for the right-hand side
  CN_WA = 10,  // gt^ij d_i W d_j alpha (u^2)
  CN_AA = 11,  // At_ij At^ij
  CN_GA = 12,  // Gamma^k_ij d_k alpha (u^2)
  CN_BR = 18,  // Gamma^k_ij At^ij (u)
  CN_AK = 21,  // At_ik At^k_j
  CN_AW = 27,  // At^ij d_j W (u)
  CN_AL = 30,  // At^ij d_j alpha (u)
  FM_SLOTS = 42
};

FXD double fx_get(const double* p) {
#ifdef __CUDA_ARCH__
  return __ldg(p);
#else
  return *p;
#endif
}
// The same pointer, as one the compiler knows nothing of: values read through it are
// read again rather than kept in registers (and spilled) from an earlier read.
FXD const double* fx_again(const double* p) {
#ifdef __CUDA_ARCH__
  asm volatile("" : "+l"(p));
#endif
  return p;
}
#define FLD(f) fx_get(Y + ((long)(f) * fs + o))
#define D1(f, d) fx_get(S + ((long)(Q_D1 + 3 * (f) + (d)) * fs + o))
#define D2(sl, p) fx_get(S + ((long)(Q_D2 + 6 * (sl) + (p)) * fs + o))

// The sums over tensor indices that the right-hand side (CONS: the constraints)
// takes, into the slots CN_*, from the fields, their derivatives and the inverse
// metric.  Returns false, the slots undefined, where a value is out of range.
template <bool CONS, int T, class KT>
FXD bool z4c_connection_fixed(const double* Y, const double* S, long fs, long o, const Z4cUnits& c,
                              const double* gu, const FxMem<T>& mem, const KT& K) {
  FxCheck bad;
  {
    FxN d[18];
#pragma unroll
    for (int q = 0; q < 18; ++q) d[q] = fx_load(D1(ZG + q / 3, q % 3), bad);
#define DG(i, j, k) d[3 * sidx(i, j) + (k)]
#pragma unroll
    for (int k = 0; k < 3; ++k)
#pragma unroll
      for (int i = 0; i < 3; ++i)
#pragma unroll
        for (int j = i; j < 3; ++j) {
          // where k is i or j two of the three terms cancel, where i = j != k two coincide
          FxN v;
          if (k == i) v = DG(i, i, j);
          else if (k == j) v = DG(j, j, i);
          else if (i == j) v = fx_norm(fx_add(FxN{DG(i, k, i).m, DG(i, k, i).e + 1}, FxN{-DG(i, i, k).m, DG(i, i, k).e}));
          else v = fx_norm(fx_add_sub(DG(j, k, i), DG(i, k, j), DG(i, j, k)));
          mem.st(FM_GS + 6 * k + sidx(i, j), v);
        }
#undef DG
  }
  FxA g[6];
#pragma unroll
  for (int s = 0; s < 6; ++s) g[s] = fx_op(fx_load(gu[s], bad));
  const FxA gr[3][3] = {{g[0], g[1], g[2]}, {g[1], g[3], g[4]}, {g[2], g[4], g[5]}};
#pragma unroll 1
  for (int s = 0; s < 6; ++s) {
    const FxN b[3] = {mem.ld(FM_GS + s), mem.ld(FM_GS + 6 + s), mem.ld(FM_GS + 12 + s)};
#pragma unroll
    for (int k = 0; k < 3; ++k) mem.st(FM_GU + 6 * k + s, fx_norm(fx_dot<3>(gr[k], b)));
  }
  {
    // gt_k(i d_j) Gamt^k
    FxN dG[9];
    FxA h[6];
#pragma unroll
    for (int q = 0; q < 9; ++q) dG[q] = fx_load(fmul(D1(ZGAM + q / 3, q % 3), c.iu, K), bad);
#pragma unroll
    for (int s = 0; s < 6; ++s) h[s] = fx_op(fx_load(FLD(ZG + s), bad));
#pragma unroll
    for (int i = 0; i < 3; ++i)
#pragma unroll
      for (int j = i; j < 3; ++j) {
        const FxA a[6] = {h[sidx(0, i)], h[sidx(1, i)], h[sidx(2, i)], h[sidx(0, j)], h[sidx(1, j)], h[sidx(2, j)]};
        const FxN b[6] = {dG[j], dG[3 + j], dG[6 + j], dG[i], dG[3 + i], dG[6 + i]};
        FxN q = i == j ? fx_dot<3, 62>(a, b) : fx_dot<6, 62>(a, b);  // below 2^60.6
        if (i == j) q.e += 1;
        mem.st(FM_Q + sidx(i, j), q);
      }
  }
  // gt^lm (2 Gamma^k_l(i Gamma_j)km + Gamma^k_im Gamma_klj) = T_ij + T_ji + t3 with
  // U[k][l] = gt^lm Gamma_{J,km}, T_iJ = Gamma^k_li U[k][l], t3 = Gamma^J_im U[j][m] summed over J
#pragma unroll 1
  for (int J = 0; J < 3; ++J) {
    FxN U[9];
    {
      FxN G[6];
#pragma unroll
      for (int s = 0; s < 6; ++s) G[s] = mem.ld(FM_GS + 6 * J + s);
#pragma unroll
      for (int k = 0; k < 3; ++k) {
        const FxN r[3] = {G[sidx(k, 0)], G[sidx(k, 1)], G[sidx(k, 2)]};
#pragma unroll
        for (int l = 0; l < 3; ++l) U[3 * k + l] = fx_norm(fx_dot<3>(gr[l], r));
      }
    }
#pragma unroll 1
    for (int i = 0; i < 3; ++i) {
      FxA r[9];
#pragma unroll
      for (int k = 0; k < 3; ++k) mem.row(FM_GU + 6 * k, i, r + 3 * k);
      FxN t = fx_dot<9, 62>(r, U);  // below 2^60.2, two of these at most in one sum
      if (i == J) t.m += t.m;
      const int s = FM_Q + fx_slot(i, J);
      mem.st(s, fx_acc(mem.ld(s), t));
    }
    FxA G[6];
#pragma unroll
    for (int s = 0; s < 6; ++s) G[s] = fx_op(mem.ld(FM_GU + 6 * J + s));
#pragma unroll
    for (int i = 0; i < 3; ++i) {
      const FxA r[3] = {G[sidx(i, 0)], G[sidx(i, 1)], G[sidx(i, 2)]};
#pragma unroll
      for (int j = i; j < 3; ++j) {
        const int s = FM_Q + sidx(i, j);
        mem.st(s, fx_acc(mem.ld(s), fx_dot<3, 62>(r, U + 3 * j)));  // below 2^59.6, three of these; 2^62.7 in all
      }
    }
  }
#pragma unroll
  for (int s = 0; s < 6; ++s) mem.std(CN_Q + s, fx_double(mem.ld(FM_Q + s), bad));
  FxN w[3], al[3];
#pragma unroll
  for (int k = 0; k < 3; ++k) {
    w[k] = fx_load(D1(ZW, k), bad);
    w[k].e += 1;
    if (!CONS) {
      al[k] = fx_load(D1(ZAL, k), bad);
      al[k].e += 1;
    }
  }
  {
    const FxA t[6] = {g[0], fx_twice(g[1]), fx_twice(g[2]), g[3], fx_twice(g[4]), g[5]};
#pragma unroll 1
    for (int k = 0; k < 3; ++k) {
      FxN v[6];
#pragma unroll
      for (int s = 0; s < 6; ++s) v[s] = mem.ld(FM_GU + 6 * k + s);
      mem.std(CN_GD + k, fx_double(fx_dot<6>(t, v), bad));
    }
  }
  {
    const FxA wo[3] = {fx_op(w[0]), fx_op(w[1]), fx_op(w[2])};
    FxA ao[3];
    if (!CONS)
#pragma unroll
      for (int k = 0; k < 3; ++k) ao[k] = fx_op(al[k]);
    FxN u[3];  // gt^kl d_l W
#pragma unroll
    for (int k = 0; k < 3; ++k) u[k] = fx_norm(fx_dot<3>(gr[k], w));
    mem.std(CN_WW, fx_double(fx_dot<3>(wo, u), bad));
    if (!CONS) mem.std(CN_WA, fx_double(fx_dot<3>(ao, u), bad));
#pragma unroll 1
    for (int s = 0; s < 6; ++s) {
      const FxN v[3] = {mem.ld(FM_GU + s), mem.ld(FM_GU + 6 + s), mem.ld(FM_GU + 12 + s)};
      mem.std(CN_GW + s, fx_double(fx_dot<3>(wo, v), bad));
      if (CONS) {
#pragma unroll
        for (int k = 0; k < 3; ++k) mem.std(CN_GU + 6 * k + s, fx_double(v[k], bad));
      } else {
        mem.std(CN_GA + s, fx_double(fx_dot<3>(ao, v), bad));
      }
    }
  }
  if (!CONS) {
    FxN A[6], Am[9];  // Am: At^i_j, 3 i + j
#pragma unroll
    for (int s = 0; s < 6; ++s) A[s] = fx_load(FLD(ZA + s), bad);
#pragma unroll
    for (int q = 0; q < 9; ++q) {
      const FxN b[3] = {A[sidx(0, q % 3)], A[sidx(1, q % 3)], A[sidx(2, q % 3)]};
      Am[q] = fx_norm(fx_dot<3>(gr[q / 3], b));
    }
    FxA au[6];
#pragma unroll
    for (int i = 0; i < 3; ++i)
#pragma unroll
      for (int j = i; j < 3; ++j) au[sidx(i, j)] = fx_op(fx_norm(fx_dot<3>(gr[j], Am + 3 * i)));
    const FxA t[6] = {au[0], fx_twice(au[1]), fx_twice(au[2]), au[3], fx_twice(au[4]), au[5]};
    mem.std(CN_AA, fx_double(fx_dot<6>(t, A), bad));
    double br[3];
#pragma unroll
    for (int k = 0; k < 3; ++k) {
      FxN v[6];
#pragma unroll
      for (int s = 0; s < 6; ++s) v[s] = mem.ld(FM_GU + 6 * k + s);
      br[k] = fx_double(fx_dot<6>(t, v), bad);
    }
#pragma unroll
    for (int i = 0; i < 3; ++i) {
      mem.std(CN_BR + i, br[i]);
      const FxA a[3] = {au[sidx(i, 0)], au[sidx(i, 1)], au[sidx(i, 2)]};
      mem.std(CN_AW + i, fx_double(fx_dot<3>(a, w), bad));
      mem.std(CN_AL + i, fx_double(fx_dot<3>(a, al), bad));
#pragma unroll
      for (int j = i; j < 3; ++j) {
        const FxA r[3] = {fx_op(A[sidx(0, j)]), fx_op(A[sidx(1, j)]), fx_op(A[sidx(2, j)])};
        const FxN b[3] = {Am[i], Am[3 + i], Am[6 + i]};
        mem.std(CN_AK + sidx(i, j), fx_double(fx_dot<3>(r, b), bad));
      }
    }
  }
  return bad.ok();
}

// The same in FP64, out of line: its registers stay out of the kernel's own budget.
struct InverseMetric {
  double gu[6];
};
template <bool CONS, int T, class KT>
FX_NOINLINE void z4c_connection_fp64(const double* Y, const double* S, long fs, long o, Z4cUnits c, InverseMetric t,
                                     FxMem<T> mem, KT K) {
  double g[6], gu[6], A[6], dW[3], dal[3];
#pragma unroll
  for (int s = 0; s < 6; ++s) {
    g[s] = FLD(ZG + s);
    gu[s] = t.gu[s];
    A[s] = FLD(ZA + s);
  }
#pragma unroll
  for (int k = 0; k < 3; ++k) {
    dW[k] = fmul(2.0, D1(ZW, k), K);
    dal[k] = fmul(2.0, D1(ZAL, k), K);
  }
  double dg[18], Gs[3][6], Gu[3][6];
#pragma unroll
  for (int q = 0; q < 18; ++q) dg[q] = D1(ZG + q / 3, q % 3);
#pragma unroll
  for (int k = 0; k < 3; ++k)
#pragma unroll
    for (int i = 0; i < 3; ++i)
#pragma unroll
      for (int j = i; j < 3; ++j)
        Gs[k][sidx(i, j)] =
            k == i   ? dg[3 * sidx(i, i) + j]
            : k == j ? dg[3 * sidx(j, j) + i]
            : i == j ? fma(2.0, dg[3 * sidx(i, k) + i], -dg[3 * sidx(i, i) + k])
                     : fsub(fadd(dg[3 * sidx(j, k) + i], dg[3 * sidx(i, k) + j], K), dg[3 * sidx(i, j) + k], K);
  auto dot3 = [&](const double* t, int l, double x, double y, double z) {
    return fma(t[sidx(l, 0)], x, fma(t[sidx(l, 1)], y, fmul(t[sidx(l, 2)], z, K)));
  };
  auto trace = [&](const double* t, const double* v) {
    return fma(2.0, fma(t[1], v[1], fma(t[2], v[2], fmul(t[4], v[4], K))),
               fma(t[0], v[0], fma(t[3], v[3], fmul(t[5], v[5], K))));
  };
#pragma unroll
  for (int k = 0; k < 3; ++k) {
#pragma unroll
    for (int s = 0; s < 6; ++s) {
      Gu[k][s] = dot3(gu, k, Gs[0][s], Gs[1][s], Gs[2][s]);
      if (CONS) mem.std(CN_GU + 6 * k + s, Gu[k][s]);
    }
    mem.std(CN_GD + k, trace(gu, Gu[k]));
  }
  double Q[6], dG[9];
#pragma unroll
  for (int q = 0; q < 9; ++q) dG[q] = fmul(D1(ZGAM + q / 3, q % 3), c.iu, K);
#pragma unroll
  for (int i = 0; i < 3; ++i)
#pragma unroll
    for (int j = i; j < 3; ++j)
      Q[sidx(i, j)] = fadd(dot3(g, i, dG[j], dG[3 + j], dG[6 + j]), dot3(g, j, dG[i], dG[3 + i], dG[6 + i]), K);
#pragma unroll
  for (int J = 0; J < 3; ++J) {
    double U[3][3];
#pragma unroll
    for (int k = 0; k < 3; ++k)
#pragma unroll
      for (int l = 0; l < 3; ++l) U[k][l] = dot3(gu, l, Gs[J][sidx(k, 0)], Gs[J][sidx(k, 1)], Gs[J][sidx(k, 2)]);
#pragma unroll
    for (int i = 0; i < 3; ++i) {
      double t = fmul(Gu[0][sidx(0, i)], U[0][0], K);
#pragma unroll
      for (int q = 1; q < 9; ++q) t = fma(Gu[q / 3][sidx(q % 3, i)], U[q / 3][q % 3], t);
      Q[sidx(i, J)] = i == J ? fma(2.0, t, Q[sidx(i, J)]) : fadd(Q[sidx(i, J)], t, K);
#pragma unroll
      for (int j = i; j < 3; ++j)
#pragma unroll
        for (int m = 0; m < 3; ++m) Q[sidx(i, j)] = fma(Gu[J][sidx(i, m)], U[j][m], Q[sidx(i, j)]);
    }
  }
  double u[3];
#pragma unroll
  for (int k = 0; k < 3; ++k) u[k] = dot3(gu, k, dW[0], dW[1], dW[2]);
  auto along = [&](const double* a, double x, double y, double z) {
    return fma(a[0], x, fma(a[1], y, fmul(a[2], z, K)));
  };
  mem.std(CN_WW, along(dW, u[0], u[1], u[2]));
  if (!CONS) mem.std(CN_WA, along(dal, u[0], u[1], u[2]));
#pragma unroll
  for (int s = 0; s < 6; ++s) {
    mem.std(CN_Q + s, Q[s]);
    mem.std(CN_GW + s, along(dW, Gu[0][s], Gu[1][s], Gu[2][s]));
    if (!CONS) mem.std(CN_GA + s, along(dal, Gu[0][s], Gu[1][s], Gu[2][s]));
  }
  if (!CONS) {
    double Am[3][3], Auu[6];
#pragma unroll
    for (int i = 0; i < 3; ++i)
#pragma unroll
      for (int j = 0; j < 3; ++j) Am[i][j] = dot3(gu, i, A[sidx(0, j)], A[sidx(1, j)], A[sidx(2, j)]);
#pragma unroll
    for (int i = 0; i < 3; ++i)
#pragma unroll
      for (int j = i; j < 3; ++j) {
        Auu[sidx(i, j)] = dot3(gu, j, Am[i][0], Am[i][1], Am[i][2]);
        mem.std(CN_AK + sidx(i, j), dot3(A, j, Am[0][i], Am[1][i], Am[2][i]));
      }
    mem.std(CN_AA, trace(A, Auu));
#pragma unroll
    for (int i = 0; i < 3; ++i) {
      mem.std(CN_BR + i, trace(Auu, Gu[i]));
      mem.std(CN_AW + i, dot3(Auu, i, dW[0], dW[1], dW[2]));
      mem.std(CN_AL + i, dot3(Auu, i, dal[0], dal[1], dal[2]));
    }
  }
}

// How a point function gets these sums: in integers, or in FP64 where they do not allow that.
struct Connection {
  template <bool CONS, int T, class KT>
  FXD static void sums(const double* Y, const double* S, long fs, long o, const Z4cUnits& c, const double* gu,
                       const FxMem<T>& mem, const KT& K) {
    if (!z4c_connection_fixed<CONS, T, KT>(Y, S, fs, o, c, gu, mem, K)) {
      InverseMetric t;
#pragma unroll
      for (int s = 0; s < 6; ++s) t.gu[s] = gu[s];
      z4c_connection_fp64<CONS, T, KT>(Y, S, fs, o, c, t, mem, K);
    }
  }
};

// What the right-hand side and the constraints share.  Sums, differences and
// products that do not fuse with a neighbour are written as fadd, fsub, fmul:
// FMAs with the run-time unit constants of an FmaK (measured faster than plain
// DADD/DMUL), or the DADD/DMUL of a PlainK.
struct Z4cGeometry {
  double g[6], gu[6], W, iW;
  double gw[6];  // trace weights: gt^ij X_ij = sum_s gw[s] X[s]

  template <class KT>
  FXD double up(int k, const double* v, const KT& K) const {  // gt^kl v_l
    return fma(gu[sidx(k, 0)], v[0], fma(gu[sidx(k, 1)], v[1], fmul(gu[sidx(k, 2)], v[2], K)));
  }
  template <class KT>
  FXD double trace(const double* v, const KT& K) const {
    double t = fmul(gw[0], v[0], K);
#pragma unroll
    for (int s = 1; s < 6; ++s) t = fma(gw[s], v[s], t);
    return t;
  }

  template <class CONN, bool CONS, int T, class KT>
  FXD void load(const double* Y, const double* S, long fs, long o, const Z4cUnits& c, const FxMem<T>& mem,
                const KT& K) {
    {
      double v[6], f[6];
#pragma unroll
      for (int s = 0; s < 6; ++s) v[s] = FLD(ZG + s);
      const double w = FLD(ZW);
      f[0] = fma(v[3], v[5], fmul(-v[4], v[4], K));
      f[1] = fma(v[2], v[4], fmul(-v[1], v[5], K));
      f[2] = fma(v[1], v[4], fmul(-v[2], v[3], K));
      f[3] = fma(v[0], v[5], fmul(-v[2], v[2], K));
      f[4] = fma(v[1], v[2], fmul(-v[0], v[4], K));
      f[5] = fma(v[0], v[3], fmul(-v[1], v[1], K));
      const double det = fma(v[0], f[0], fma(v[1], f[1], fmul(v[2], f[2], K)));
      const double rdw = 1.0 / fmul(det, w, K);  // one division for 1/det and 1/W
      const double idet = fmul(w, rdw, K);
      iW = fmul(det, rdw, K);
#pragma unroll
      for (int s = 0; s < 6; ++s) gu[s] = fmul(f[s], idet, K);
    }
    CONN::template sums<CONS, T, KT>(Y, S, fs, o, c, gu, mem, K);
    Y = fx_again(Y);
    W = FLD(ZW);
#pragma unroll
    for (int s = 0; s < 6; ++s) {
      g[s] = FLD(ZG + s);
      gw[s] = fx_pure(s) ? gu[s] : fmul(2.0, gu[s], K);
    }
  }

  // -1/2 gt^lm for sums over the stored second derivatives (the pair lm, ml counted once)
  template <class KT>
  FXD void second(const Z4cUnits& c, const KT& K, double* guS) const {
#pragma unroll
    for (int s = 0; s < 6; ++s) guS[s] = fmul(gu[s], fx_pure(s) ? c.mh_pure : -4.0, K);
  }
  // R_ij = R^W_ij + Rt_ij in units of u^2, every term accumulated in one chain of FMAs
  // onto the quadratic part
  template <int T, class KT>
  FXD void ricci(const double* S, long fs, long o, const Z4cUnits& c, const FxMem<T>& mem, const double* guS,
                 const KT& K, double* R) const {
    double DDW[6];
#pragma unroll
    for (int s = 0; s < 6; ++s) DDW[s] = fma(D2(0, s), fx_pure(s) ? c.pure : 4.0, -mem.ldd(CN_GW + s));
    // R^W_ij = D_i D_j W / W + gt_ij (D^l D_l W - 2 |dW|^2 / W) / W
    const double z = fmul(fma(fmul(-2.0, mem.ldd(CN_WW), K), iW, trace(DDW, K)), iW, K);
    const double Gd[3] = {mem.ldd(CN_GD), mem.ldd(CN_GD + 1), mem.ldd(CN_GD + 2)};
#pragma unroll
    for (int s = 0; s < 6; ++s) {
      double r = mem.ldd(CN_Q + s);
#pragma unroll
      for (int q = 0; q < 6; ++q) r = fma(guS[q], D2(1 + s, q), r);  // -1/2 gt^lm d_l d_m gt_ij
      // (Gamma_d)^k Gamma_(ij)k = (Gamma_d)^k d_k gt_ij / 2
#pragma unroll
      for (int k = 0; k < 3; ++k) r = fma(Gd[k], D1(ZG + s, k), r);
      R[s] = fma(g[s], z, fma(DDW[s], iW, r));
    }
  }
};

// Right-hand side of the Z4c system at one cell (Sec. III.A; vacuum, so the
// matter terms vanish): out(f, value, out.load(f)) for every field.
template <class CONN, int T, class KT, class OUT>
FXD void z4c_rhs_point(const double* Y, const double* S, long fs, long o, const Z4cParams& P, double eta,
                       const Z4cUnits& c, const FxMem<T>& mem, const KT& K, const OUT& out) {
  Z4cGeometry G;
  G.load<CONN, false, T, KT>(Y, S, fs, o, c, mem, K);
  Y = fx_again(Y);
  S = fx_again(S);
  const double *g = G.g, *gu = G.gu;
  const double W = G.W, iW = G.iW, AA = mem.ldd(CN_AA);
  const double Kh = FLD(ZK), Th = FLD(ZTH), al = FLD(ZAL);
  double guS[6];
  G.second(c, K, guS);
  // alpha R_ij - D_i D_j alpha and the traces of both, in units of u^2
  double X[6], trR, trDDal;
  {
    double R[6], DDal[6], vW[3], da[3];  // vW: 4 d_k W / W
    G.ricci(S, fs, o, c, mem, guS, K, R);
    const double iW4 = fmul(4.0, iW, K), WAiW = fmul(mem.ldd(CN_WA), iW, K);
#pragma unroll
    for (int k = 0; k < 3; ++k) {
      vW[k] = fmul(D1(ZW, k), iW4, K);
      da[k] = D1(ZAL, k);
    }
#pragma unroll
    for (int i = 0; i < 3; ++i)
#pragma unroll
      for (int j = i; j < 3; ++j) {
        // with Gamma^k_ij - (delta^k_i d_j W + delta^k_j d_i W - gt_ij gt^kl d_l W) / W
        const int s = sidx(i, j);
        const double t = fma(D2(7, s), fx_pure(s) ? c.pure : 4.0, fma(-g[s], WAiW, -mem.ldd(CN_GA + s)));
        DDal[s] = i == j ? fma(fmul(2.0, vW[i], K), da[i], t) : fma(vW[j], da[i], fma(vW[i], da[j], t));
        X[s] = fma(al, R[s], -DDal[s]);
      }
    trR = G.trace(R, K);
    trDDal = G.trace(DDal, K);
  }
  const double W2 = fmul(fmul(W, W, K), c.u2, K);
  const double Rsc = fmul(W2, trR, K);
  const double DiDial = fmul(W2, trDDal, K);
  const double trX = fma(al, trR, -trDDal);

  double A[6], Gd[3];
#pragma unroll
  for (int s = 0; s < 6; ++s) A[s] = FLD(ZA + s);
#pragma unroll
  for (int k = 0; k < 3; ++k) Gd[k] = fmul(mem.ldd(CN_GD + k), c.u, K);
  double dbe[3][3];  // dbe[i][j] = d_j beta^i
#pragma unroll
  for (int i = 0; i < 3; ++i)
#pragma unroll
    for (int j = 0; j < 3; ++j) dbe[i][j] = fmul(D1(ZB + i, j), c.s1, K);
  const double divb = fadd(fadd(dbe[0][0], dbe[1][1], K), dbe[2][2], K);
  const double Kt = fma(2.0, Th, Kh);
  const double third = 1.0 / 3.0, twothird = 2.0 / 3.0;
  const double alKt = fmul(al, Kt, K);
  const double m2al = fmul(-2.0, al, K);
  const double m23divb = fmul(-twothird, divb, K);
  const double m13trX = fmul(-third, trX, K);
  const double cA = fadd(alKt, m23divb, K);  // (alpha Kt - 2/3 div beta), the coefficient of At_ij
  const double be[3] = {FLD(ZB), FLD(ZB + 1), FLD(ZB + 2)};
  // advection beta^i d_i f added onto x, the scale s1 carried by beta
  const double bes[3] = {fmul(be[0], c.s1, K), fmul(be[1], c.s1, K), fmul(be[2], c.s1, K)};
#define ADV_ON(f, x) fma(bes[0], D1(f, 0), fma(bes[1], D1(f, 1), fma(bes[2], D1(f, 2), (x))))
#define ADV(f) fma(bes[0], D1(f, 0), fma(bes[1], D1(f, 1), fmul(bes[2], D1(f, 2), K)))
  // gt_ij and At_ij
#pragma unroll
  for (int i = 0; i < 3; ++i)
#pragma unroll
    for (int j = i; j < 3; ++j) {
      const int s = sidx(i, j);
      const auto pg = out.load(ZG + s), pa = out.load(ZA + s);
      // gt_k(i d_j) beta^k and At_k(i d_j) beta^k with the terms in gt_ij and At_ij; At_ik At^k_j
      double lg = fmul(m23divb, g[s], K), la = fmul(cA, A[s], K);
      if (i == j) {
        lg = fma(2.0, fma(g[sidx(0, i)], dbe[0][i], fma(g[sidx(1, i)], dbe[1][i], fmul(g[sidx(2, i)], dbe[2][i], K))), lg);
        la = fma(2.0, fma(A[sidx(0, i)], dbe[0][i], fma(A[sidx(1, i)], dbe[1][i], fmul(A[sidx(2, i)], dbe[2][i], K))), la);
      } else {
#pragma unroll
        for (int k = 0; k < 3; ++k) {
          lg = fma(g[sidx(k, i)], dbe[k][j], fma(g[sidx(k, j)], dbe[k][i], lg));
          la = fma(A[sidx(k, i)], dbe[k][j], fma(A[sidx(k, j)], dbe[k][i], la));
        }
      }
      out(ZG + s, ADV_ON(ZG + s, fma(m2al, A[s], lg)), pg);
      const double tf = fma(m13trX, g[s], X[s]);
      out(ZA + s, ADV_ON(ZA + s, fma(W2, tf, fma(m2al, mem.ldd(CN_AK + s), la))), pa);
    }
  // Gamt^i and beta^i
  {
    double dd[3];     // -2/3 d_j (2 Khat + Theta) as stencil sums
    double ddivb[3];  // 1/3 d_j d_k beta^k: the k = j term a pure second derivative
#pragma unroll
    for (int j = 0; j < 3; ++j) {
      dd[j] = fma(-4.0 / 3.0, D1(ZK, j), fmul(-twothird, D1(ZTH, j), K));
      ddivb[j] = fma(D2(8, sidx(j, 0)), j == 0 ? c.tp : c.tm,
                     fma(D2(9, sidx(j, 1)), j == 1 ? c.tp : c.tm, fmul(D2(10, sidx(j, 2)), j == 2 ? c.tp : c.tm, K)));
    }
    const double m3iW = fmul(-3.0, iW, K);
    const double twoal = fmul(c.s1, al, K);
    const double twothirddivb = fmul(twothird, divb, K);
    const double m2k1al = fmul(-2.0 * P.kappa1, al, K);
    const double cGd = fsub(twothirddivb, m2k1al, K);
#pragma unroll
    for (int i = 0; i < 3; ++i) {
      const auto pgam = out.load(ZGAM + i), pb = out.load(ZB + i);
      const double gam = FLD(ZGAM + i);
      double t = fmul(guS[0], D2(8 + i, 0), K);  // -1/2 gt^jk d_j d_k beta^i
#pragma unroll
      for (int q = 1; q < 6; ++q) t = fma(guS[q], D2(8 + i, q), t);
      double r = fma(c.m2u2, t, fmul(c.m2u, mem.ldd(CN_AL + i), K));   // -2 At^ij d_j alpha
      double br = fma(m3iW, mem.ldd(CN_AW + i), mem.ldd(CN_BR + i));  // -3 At^ij d_j W / W
#pragma unroll
      for (int j = 0; j < 3; ++j) {
        br = fma(gu[sidx(i, j)], dd[j], br);
        r = fma(gu[sidx(i, j)], ddivb[j], fma(-Gd[j], dbe[i][j], r));
      }
      r = fma(twoal, br, r);
      // 2/3 (Gamma_d)^i div beta - 2 kappa1 alpha (Gamt^i - (Gamma_d)^i)
      r = fma(Gd[i], cGd, fma(m2k1al, gam, r));
      out(ZGAM + i, ADV_ON(ZGAM + i, r), pgam);
      out(ZB + i, ADV_ON(ZB + i, fma(0.75, gam, fmul(-eta, be[i], K))), pb);  // Gamma-driver
    }
  }
  out(ZW, ADV_ON(ZW, fmul(fmul(third, W, K), fma(al, Kt, -divb), K)), out.load(ZW));
  out(ZK, fma(al, fma(fmul(third, Kt, K), Kt, AA),
              fma(fmul(al, P.kappa1 * (1.0 - P.kappa2), K), Th, ADV_ON(ZK, -DiDial))), out.load(ZK));
  out(ZTH, fma(fmul(0.5, al, K), fma(fmul(twothird, Kt, K), Kt, fsub(Rsc, AA, K)),
               fma(fmul(-al, P.kappa1 * (2.0 + P.kappa2), K), Th, ADV(ZTH))), out.load(ZTH));
  out(ZAL, fma(m2al, Kh, ADV(ZAL)), out.load(ZAL));  // 1+log
#undef ADV_ON
#undef ADV
}

// The Z4c constraints at one cell:
//   H   = R + 2/3 (Khat + 2 Theta)^2 - At_ij At^ij      (R the Ricci scalar of gamma)
//   M^i = d_j At^ij + Gamt^i_jk At^jk - 3 At^ij d_j W / W - 2/3 gt^ij d_j (Khat + 2 Theta)
//   G^i = Gamt^i - gt^jk Gamt^i_jk
// out(c, value).  With d_k gt_ij = Gamma_{i,jk} + Gamma_{j,ik} and At^ij's own derivatives,
//   M^i = gt^im (gt^jp d_j At_mp - Gamma^n_mj At_n^j) - At^id Gamma^j_dj - At^i_p (Gamma_d)^p
//         - 3 At^ij d_j W / W - 2/3 gt^ij d_j (Khat + 2 Theta)
template <class CONN, int T, class KT, class OUT>
FXD void z4c_constraints_point(const double* Y, const double* S, long fs, long o, const Z4cUnits& c,
                               const FxMem<T>& mem, const KT& K, const OUT& out) {
  Z4cGeometry G;
  G.load<CONN, true, T, KT>(Y, S, fs, o, c, mem, K);
  const double Kt = fma(2.0, FLD(ZTH), FLD(ZK));
  double R[6], Am[3][3], Auu[6], A[6];
#pragma unroll
  for (int s = 0; s < 6; ++s) A[s] = FLD(ZA + s);
  double guS[6];
  G.second(c, K, guS);
  G.ricci(S, fs, o, c, mem, guS, K, R);
#pragma unroll
  for (int i = 0; i < 3; ++i)
#pragma unroll
    for (int j = 0; j < 3; ++j) {
      const double a[3] = {A[sidx(0, j)], A[sidx(1, j)], A[sidx(2, j)]};
      Am[i][j] = G.up(i, a, K);
    }
#pragma unroll
  for (int i = 0; i < 3; ++i)
#pragma unroll
    for (int j = i; j < 3; ++j) Auu[sidx(i, j)] = G.up(j, Am[i], K);
  const double AA = fma(2.0, fma(A[1], Auu[1], fma(A[2], Auu[2], fmul(A[4], Auu[4], K))),
                        fma(A[0], Auu[0], fma(A[3], Auu[3], fmul(A[5], Auu[5], K))));
  out(0, fma(fmul(fmul(G.W, G.W, K), c.u2, K), G.trace(R, K), fma(fmul(2.0 / 3.0, Kt, K), Kt, -AA)));
  double b[3], t[3], dd[3];
#pragma unroll
  for (int i = 0; i < 3; ++i) {
    double p = 0.0, q = 0.0;
    t[i] = 0.0;
#pragma unroll
    for (int j = 0; j < 3; ++j) {
#pragma unroll
      for (int k = 0; k < 3; ++k) {
        p = fma(G.gu[sidx(j, k)], D1(ZA + sidx(i, k), j), p);
        q = fma(mem.ldd(CN_GU + 6 * k + sidx(i, j)), Am[j][k], q);
      }
      t[i] = fadd(t[i], mem.ldd(CN_GU + 6 * j + sidx(i, j)), K);  // Gamma^j_ij
    }
    b[i] = fma(2.0, p, -q);
    t[i] = fma(fmul(6.0, D1(ZW, i), K), G.iW, t[i]);
    dd[i] = fma(-4.0 / 3.0, D1(ZK, i), fmul(-8.0 / 3.0, D1(ZTH, i), K));
  }
#pragma unroll
  for (int i = 0; i < 3; ++i) {
    double m = fadd(G.up(i, b, K), G.up(i, dd, K), K);
#pragma unroll
    for (int j = 0; j < 3; ++j) m = fma(-Auu[sidx(i, j)], t[j], fma(-Am[i][j], mem.ldd(CN_GD + j), m));
    out(1 + i, fmul(c.u, m, K));
    out(4 + i, fma(-c.u, mem.ldd(CN_GD + i), FLD(ZGAM + i)));
  }
}

#undef FLD
#undef D1
#undef D2

}  // namespace sc
