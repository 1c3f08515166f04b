// sc_z4c_fixed.cuh -- the Z4c right-hand side at one cell in block fixed point.
//
// Nearly all of the right-hand side is small contractions over tensor indices.
// In FP64 one cell takes 1072 instructions of a pipe that starts 2 per SM and
// clock; a 32 x 32 + 64 bit multiply-add takes a fraction of that time on the
// FP32/integer pipes, which the FP64 form leaves idle.  So the tensors are held
// as blocks of signed integers with one exponent per block (value = v * 2^e,
// |v| < 2^59 unless a comment says less), a product is three multiply-adds into
// two 64-bit accumulators (FxDot), and a sum of products is shifted into place
// once.  Blocks are loaded with the largest magnitude at bit 58, 6 bits more
// than a double's significand, and brought back there (fx_norm) after sums and
// products whose largest value may have moved down.  A result therefore carries
// an absolute error of a few 2^-59 of its block's largest value, where a chain of
// FP64 operations carries 2^-53 of the largest partial sum at every step.  What
// is left to FP64: the one division, scalar combinations, and the conversion of
// each result.
//
// Bounds are given as bits: "59.2" at a sum means |sum| < 2^59.2; every 64-bit
// sum stays below 2^63, and everything that fx_norm gets below its BITS.
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
#else
#define FXD inline
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
  const long long b = ((long long)hi << 32) | (unsigned)lo;
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
FXD unsigned long long fx_shr_u(unsigned long long x, unsigned n) {
#ifdef __CUDA_ARCH__
  unsigned long long r;
  asm("shr.u64 %0, %1, %2;" : "=l"(r) : "l"(x), "r"(n));
  return r;
#else
  return n > 63 ? 0 : x >> n;
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

// A multiplication operand: h * 2^32 + l, the low half signed so that every
// partial product is a signed 32 x 32 multiplication.
struct FxP {
  int h, l;
};
// The halves of x.  (As 32-bit shifts of x the compiler would widen them again
// in products, and a 32 x 32 multiplication would become a 64 x 64 one.)
FXD FxP fx_halves(long long x) {
  FxP r;
#ifdef __CUDA_ARCH__
  asm("mov.b64 {%0, %1}, %2;" : "=r"(r.l), "=r"(r.h) : "l"(x));
#else
  r.l = (int)x;
  r.h = (int)(x >> 32);
#endif
  return r;
}
FXD FxP fx_split(long long x) {
  FxP r = fx_halves(x);
  r.h += (int)((unsigned)r.l >> 31);
  return r;
}
FXD long long fx_join(const FxP& p) { return fx_shl((long long)p.h, 32) + p.l; }

// A sum of products: hh * 2^64 + mm * 2^32, the low x low parts (at most 2^62
// each) dropped.  They are signed and below the unit that fin keeps, or 8 units
// of it where a single product is kept to 59 bits.
struct FxDot {
  long long hh = 0, mm = 0;
  FXD void mac(const FxP& a, const FxP& b) {
    hh += (long long)a.h * b.h;
    mm += (long long)a.h * b.l;
    mm += (long long)a.l * b.h;
  }
  FXD void add(const FxDot& d) {
    hh += d.hh;
    mm += d.mm;
  }
  FXD void sub(const FxDot& d) {
    hh -= d.hh;
    mm -= d.mm;
  }
  FXD void twice() {
    hh += hh;
    mm += mm;
  }
  // in units of 2^K, 59 <= K <= 64, rounded down
  template <int K>
  FXD long long fin() const {
    return fx_shl(hh, 64 - K) + (mm >> (K - 32));
  }
};

template <int N>
struct FxBlk {
  FxP v[N];
  int e;
};
// Block sums before they become operands.
template <int N>
struct FxSum {
  long long m[N];
  int e;
};

// Blocks whose largest value is above 2^150 (with that bound no product of the
// right-hand side can overflow a double) or in the lowest ninth of the exponent
// range, or that hold an infinity or a NaN, are left to the FP64 form (bad).  A
// block of zeros is fine: it is aligned to the lower end, so that it stays zero
// and vanishes in sums.
constexpr int kFxLo = 128 << 20, kFxHi = (1023 + 150) << 20;
FXD int fx_out_of_range(int E) { return (unsigned)(E - kFxLo) > (unsigned)(kFxHi - kFxLo) && E != 0; }
// The value v * 2^off (off in place, as an exponent field) in units of the block's.
template <int BITS>
FXD long long fx_mant(double v, int Em, int off) {
  constexpr int G = BITS - 53;
  const int h = fx_dhi(v);
  const unsigned l = fx_dlo(v);
  const int s = h >> 31;
  const unsigned mh = (unsigned)((h & 0xfffff) | 0x100000);
  const unsigned long long x = ((unsigned long long)((mh << G) | (l >> (32 - G))) << 32) | (l << G);
  const long long r = (long long)fx_shr_u(x, (unsigned)(Em - ((h & 0x7ff00000) + off)) >> 20);
  return (r ^ s) - s;  // rounded towards zero: a zero of either sign stays zero
}
// poff: exponent offset (in place) of the pure entries of a block of six second derivatives.
template <int BITS, int N>
FXD void fx_load_raw(const double* x, FxSum<N>& b, int& bad, int poff = 0) {
  int E = 0;
#pragma unroll
  for (int i = 0; i < N; ++i) {
    const int a = fx_dhi(x[i]) & 0x7fffffff;
    const int t = poff && fx_pure(i % 6) ? a + poff : a;
    E = E > t ? E : t;
  }
  bad |= poff ? (E != poff && fx_out_of_range(E)) : fx_out_of_range(E);
  const int Em = E > kFxLo ? E & 0x7ff00000 : kFxLo;
  b.e = (Em >> 20) - (1023 + 52 + BITS - 53);
#pragma unroll
  for (int i = 0; i < N; ++i) b.m[i] = fx_mant<BITS>(x[i], Em, poff && fx_pure(i % 6) ? poff : 0);
}
template <int BITS, int N>
FXD FxBlk<N> fx_load(const double* x, int& bad, int poff = 0) {
  FxSum<N> r;
  fx_load_raw<BITS, N>(x, r, bad, poff);
  FxBlk<N> b;
  b.e = r.e;
#pragma unroll
  for (int i = 0; i < N; ++i) b.v[i] = fx_split(r.m[i]);
  return b;
}
template <int N>
FXD FxBlk<N> fx_plain(const FxSum<N>& r) {
  FxBlk<N> b;
  b.e = r.e;
#pragma unroll
  for (int i = 0; i < N; ++i) b.v[i] = fx_split(r.m[i]);
  return b;
}
// Sums below 2^BITS, the largest moved up to bit BITS - 1 (sums that all vanish in
// the high word move by its 27 places and stay short).
FXD int fx_mag(long long m) {  // bits of the magnitude's high word
  const int h = (int)(m >> 32);
  return h ^ (h >> 31);
}
template <int BITS, int N>
FXD FxBlk<N> fx_norm(const FxSum<N>& r) {
  int o = 0;
#pragma unroll
  for (int i = 0; i < N; ++i) o |= fx_mag(r.m[i]);
  const int s = fx_clz(o) - (64 - BITS);
  FxBlk<N> b;
  b.e = r.e - s;
#pragma unroll
  for (int i = 0; i < N; ++i) b.v[i] = fx_split(fx_shl(r.m[i], s));
  return b;
}
// The same to bit 58 for sums of any size below 2^63.
template <int N>
FXD FxBlk<N> fx_norm_any(const FxSum<N>& r) {
  int o = 0;
#pragma unroll
  for (int i = 0; i < N; ++i) o |= fx_mag(r.m[i]);
  const int s = fx_clz(o) - 1;
  FxBlk<N> b;
  b.e = r.e - s + 4;
#pragma unroll
  for (int i = 0; i < N; ++i) b.v[i] = fx_split(fx_shl(r.m[i], s) >> 4);
  return b;
}
// a += b, in units of the larger exponent
template <int N>
FXD void fx_add(FxSum<N>& a, const FxSum<N>& b) {
  const int d = a.e - b.e, sa = d < 0 ? -d : 0, sb = d > 0 ? d : 0;
#pragma unroll
  for (int i = 0; i < N; ++i) a.m[i] = fx_shr(a.m[i], sa) + fx_shr(b.m[i], sb);
  a.e += sa;
}
FXD void fx_add1(long long& m, int& e, long long bm, int be) {
  const int d = e - be, sa = d < 0 ? -d : 0, sb = d > 0 ? d : 0;
  m = fx_shr(m, sa) + fx_shr(bm, sb);
  e += sa;
}
FXD double fx_double(long long m, int e) {
  const double d = (double)m;
  const int h = fx_dhi(d);
  const int x = ((h >> 20) & 0x7ff) + e;
  return h == 0 || x <= 0 ? 0.0 : fx_make(h + (e << 20), (int)fx_dlo(d));
}
// block times one operand, in units of 2^K
template <int K, int N>
FXD FxSum<N> fx_times(const FxBlk<N>& a, const FxP& c, int ec) {
  FxSum<N> r;
  r.e = a.e + ec + K;
#pragma unroll
  for (int i = 0; i < N; ++i) {
    FxDot d;
    d.mac(a.v[i], c);
    r.m[i] = d.fin<K>();
  }
  return r;
}
// sum_m a_i(m) b_m over a symmetric and a plain index
FXD FxDot fx_row(const FxBlk<6>& a, int i, const FxP* b) {
  FxDot d;
#pragma unroll
  for (int m = 0; m < 3; ++m) d.mac(a.v[sidx(i, m)], b[m]);
  return d;
}
// sum_ij a_ij b_ij of two symmetric tensors
FXD FxDot fx_trace(const FxP* a, const FxP* b) {
  FxDot d;
  d.mac(a[1], b[1]);
  d.mac(a[2], b[2]);
  d.mac(a[4], b[4]);
  d.twice();
  d.mac(a[0], b[0]);
  d.mac(a[3], b[3]);
  d.mac(a[5], b[5]);
  return d;
}

// A constant as an operand (|v| < 2^59, value v * 2^e).
struct FxC {
  FxP v;
  int e;
};
inline FxC fx_const(double x, int e) { return FxC{fx_split((long long)std::ldexp(x, -e)), e}; }
inline int fx_const_exp(double x) {  // the exponent that puts x at bit 58
  return (x == 0.0 ? -1023 : ((fx_dhi(x) >> 20) & 0x7ff) - 1023) - 58;
}
inline FxC fx_const(double x) { return fx_const(x, fx_const_exp(x)); }

// Scales of the stored derivative sums (DerivScales) as operands.
struct FxScales {
  FxC s1, ts1;       // first derivatives, a third of that
  FxC kP, kM;        // second derivatives, one exponent: pure (a value times 2^poff) and mixed
  FxC kP3, kM3;      // a third of those
  FxC twothird;      // exponent -59
  int poff;          // in place
};
inline FxScales fx_scales(const DerivScales& ds) {
  FxScales c{};
  c.s1 = fx_const(ds.s1);
  c.ts1 = fx_const(ds.ts1);
  // s2p / s2m = 12 (4th order) or 140 (8th): the power of two above it goes with the values
  const int r = ds.s2p / ds.s2m > 16.0 ? 8 : 4;
  c.poff = r << 20;
  const double p = ds.s2p / (1 << r);
  const int e = fx_const_exp(p > ds.s2m ? p : ds.s2m);
  c.kP = fx_const(p, e);
  c.kM = fx_const(ds.s2m, e);
  const int e3 = fx_const_exp((p > ds.s2m ? p : ds.s2m) / 3.0);
  c.kP3 = fx_const(p / 3.0, e3);
  c.kM3 = fx_const(ds.s2m / 3.0, e3);
  c.twothird = fx_const(2.0 / 3.0, -59);
  return c;
}

// One thread's tensors in shared memory, slot s of thread t at s * T + t.  The
// rolled loops below index them at run time, which registers do not allow, and a
// warp's access to one slot is free of bank conflicts.
template <int T>
struct FxMem {
  long long* p;
  FXD FxP ld(int s) const { return fx_halves(p[s * T]); }
  FXD void st(int s, const FxP& v) const { p[s * T] = fx_shl((long long)v.h, 32) | (unsigned)v.l; }
  FXD long long ldm(int s) const { return p[s * T]; }
  FXD void stm(int s, long long m) const { p[s * T] = m; }
  // row i of a symmetric tensor in slots s0..s0 + 5
  FXD void row(int s0, int i, FxP* r) const {
    r[0] = ld(s0 + i);
    r[1] = ld(s0 + (i == 0 ? 1 : i + 2));
    r[2] = ld(s0 + (i == 0 ? 2 : i + 3));
  }
  template <int N>
  FXD FxBlk<N> get(int s0, int e) const {
    FxBlk<N> b;
    b.e = e;
#pragma unroll
    for (int i = 0; i < N; ++i) b.v[i] = ld(s0 + i);
    return b;
  }
  template <int N>
  FXD void put(int s0, const FxBlk<N>& b) const {
#pragma unroll
    for (int i = 0; i < N; ++i) st(s0 + i, b.v[i]);
  }
};
FXD FxDot fx_dot3(const FxP* a, const FxP* b) {
  FxDot d;
  d.mac(a[0], b[0]);
  d.mac(a[1], b[1]);
  d.mac(a[2], b[2]);
  return d;
}
// slot of a symmetric pair known at run time, and the pair of a slot
FXD int fx_slot(int i, int j) {
  const int a = i < j ? i : j, b = i < j ? j : i;
  return a + b + (a > 0 ? 1 : 0);
}
FXD int fx_slot_i(int s) { return s < 3 ? 0 : s < 5 ? 1 : 2; }
FXD int fx_slot_j(int s) { return s < 3 ? s : s < 5 ? s - 2 : 2; }

// shared-memory slots of one cell
enum {
  FM_G = 0,    // gt_ij
  FM_GI = 6,   // gt^ij
  FM_GU = 12,  // Gamma^k_ij, 6 k + s; in the end the parts of seven right-hand sides without their advection
  FM_GS = 30,  // Gs[k][s], 6 k + s; then
  FM_TF = 30,  //   the trace-free part of alpha R_ij - D_i D_j alpha
  FM_A = 36,   //   At_ij
  FM_AU = 42,  //   At^ij
  FM_R = 48,   // R_ij as sums, then operands; then
  FM_AB = 48,  //   (Kt delta^k_i - 2 At^k_i) At_kj
  FM_GD = 54,  // (Gamma_d)^k
  FM_DDW = 57, // D_i D_j W / W, then the exponents of R_ij's sums; then
  FM_DB = 57,  //   d_j beta^i, 3 i + j
  FM_TB = 66,  // second derivatives of the shift in the right-hand side of Gamt^i (sums)
  FM_SLOTS = 69
};

// The right-hand side of z4c_rhs_point (sc_z4c.cu): out(f, value) for every
// field.  Returns false, the values undefined, where a block is out of range.
//
// The code is kept short on purpose.  Written out in full (21,800 instructions
// a cell, 350 KB) it ran at 0.5 instructions per clock and SM: every warp waited
// for instruction-cache misses, 0.92 ms for 262,144 cells against 0.50 ms in
// FP64.  So the tensors that several loops share live in shared memory, and
// the loops over tensor components are rolled: 0.327 ms, and 0.269 with the
// global loads issued a loop iteration or a section ahead.
// CONS: instead of the right-hand side the seven constraints of
// z4c_constraints_kernel, out(q, value), from the same Ricci tensor; with
// d_k gt_ij = Gamma_{i,jk} + Gamma_{j,ik} and At^ij's own derivatives,
//   M^i = gt^im (gt^jp d_j At_mp - Gamma^n_mj At_n^j) - At^id Gamma^j_dj - At^i_p (Gamma_d)^p
//         - 3 At^ij d_j W / W - 2/3 gt^ij d_j (Khat + 2 Theta)
template <bool CONS, int T, class KT, class OUT>
FXD bool z4c_rhs_fixed(const double* __restrict__ Y, const double* __restrict__ S, long fs, long o, const Z4cParams& P,
                       double eta, const FxScales& c, const FxMem<T>& mem, const KT& K, const OUT& out) {
#define FLD(f) Y[(long)(f) * fs + o]
#define D1(f, d) S[(long)(Q_D1 + 3 * (f) + (d)) * fs + o]
#define D2(sl, p) S[(long)(Q_D2 + 6 * (sl) + (p)) * fs + o]
  int bad = 0;
  // Global loads are issued well before their values are needed: with three
  // warps per scheduler, waiting for them took half of the kernel's time.
  struct X3 {
    double v[3];
  };
  struct X6 {
    double v[6];
  };
  auto get_d1 = [&](int f) { return X3{{D1(f, 0), D1(f, 1), D1(f, 2)}}; };
  auto get_d2 = [&](int sl) {
    return X6{{D2(sl, 0), D2(sl, 1), D2(sl, 2), D2(sl, 3), D2(sl, 4), D2(sl, 5)}};
  };
  auto scalar = [&](double x) { return fx_load<59, 1>(&x, bad); };

  const double W = FLD(ZW), Kh = FLD(ZK), Th = FLD(ZTH), al = FLD(ZAL);

  double xdg[18];
#pragma unroll
  for (int q = 0; q < 18; ++q) xdg[q] = D1(ZG + q / 3, q % 3);
  // metric, inverse metric, 1 / W
  FxBlk<6> gu;
  FxBlk<1> iW;
  int eG;
  {
    double x[6];
#pragma unroll
    for (int s = 0; s < 6; ++s) x[s] = FLD(ZG + s);
    const FxBlk<6> g = fx_load<59, 6>(x, bad);
    constexpr int cf[6][4] = {{3, 5, 4, 4}, {2, 4, 1, 5}, {1, 4, 2, 3}, {0, 5, 2, 2}, {1, 2, 0, 4}, {0, 3, 1, 1}};
    FxSum<6> m;
    m.e = 2 * g.e + 61;
#pragma unroll
    for (int s = 0; s < 6; ++s) {
      FxDot p, q;
      p.mac(g.v[cf[s][0]], g.v[cf[s][1]]);
      q.mac(g.v[cf[s][2]], g.v[cf[s][3]]);
      p.sub(q);
      m.m[s] = p.fin<61>();  // 58
    }
    const FxBlk<6> cof = fx_norm<59>(m);
    const double det = fx_double(fx_dot3(g.v, cof.v).fin<61>(), g.e + cof.e + 61);
    const double rdw = 1.0 / fmul(det, W, K);  // one division for 1/det and 1/W
    const FxBlk<1> idet = scalar(fmul(W, rdw, K));
    iW = scalar(fmul(det, rdw, K));
    gu = fx_norm<59>(fx_times<60>(cof, idet.v[0], idet.e));  // 58
    mem.put(FM_G, g);
    mem.put(FM_GI, gu);
    eG = g.e;
  }

  FxBlk<3> Gd;  // (Gamma_d)^k = gt^ij Gamma^k_ij
  double xdG[9];
  X3 xdW, xda;
  X6 xddW;
  int eGu, eR;
  {
    const FxBlk<6> gus = fx_plain(fx_times<59>(gu, c.s1.v, c.s1.e - 1));  // gt^ij s1 / 2
    // Christoffel symbols: Gamma_{k,ij} = s1 / 2 Gs[k][s(ij)] and Gamma^k_ij
    int eGs;
    {
      FxSum<18> dg;  // 57
      fx_load_raw<57, 18>(xdg, dg, bad);
      eGs = dg.e;
#define DG(i, j, d) dg.m[3 * sidx(i, j) + (d)]
#pragma unroll
      for (int k = 0; k < 3; ++k)
#pragma unroll
        for (int i = 0; i < 3; ++i)
#pragma unroll
          for (int j = i; j < 3; ++j)  // 58.6
            mem.st(FM_GS + 6 * k + sidx(i, j), fx_split(k == i   ? DG(i, i, j)
                                                        : k == j ? DG(j, j, i)
                                                        : i == j ? 2 * DG(i, k, i) - DG(i, i, k)
                                                                 : DG(j, k, i) + DG(i, k, j) - DG(i, j, k)));
#undef DG
    }
    int mag = 0;
#pragma unroll 1
    for (int s = 0; s < 6; ++s) {
      const FxP b[3] = {mem.ld(FM_GS + s), mem.ld(FM_GS + 6 + s), mem.ld(FM_GS + 12 + s)};
#pragma unroll
      for (int k = 0; k < 3; ++k) {
        const long long m = fx_row(gus, k, b).fin<61>();  // 58.2
        mag |= fx_mag(m);
        mem.stm(FM_GU + 6 * k + s, m);
      }
    }
    const int sh = fx_clz(mag) - 5;
    eGu = gus.e + eGs + 61 - sh;
    FxSum<3> gd;
    gd.e = gu.e + eGu + 63;
#pragma unroll
    for (int k = 0; k < 3; ++k) {
      FxP v[6];
#pragma unroll
      for (int s = 0; s < 6; ++s) {
        v[s] = fx_split(fx_shl(mem.ldm(FM_GU + 6 * k + s), sh));
        mem.st(FM_GU + 6 * k + s, v[s]);
      }
      gd.m[k] = fx_trace(gu.v, v).fin<63>();  // 58.2
    }
    Gd = fx_norm<59>(gd);
    mem.put(FM_GD, Gd);

    // Conformal part of the Ricci tensor.
    // gt^lm (2 Gamma^k_l(i Gamma_j)km + Gamma^k_im Gamma_klj) = T_ij + T_ji + t3,
    // U[k][l] = gt^lm Gamma_{J,km}, T_iJ = Gamma^k_li U[k][l], t3 = Gamma^J_im U[j][m] summed over J
    FxSum<6> a{}, b;
    const int eU = gus.e + eGs + 61;
#pragma unroll
    for (int s = 0; s < 6; ++s) mem.stm(FM_R + s, 0);
#pragma unroll
    for (int q = 0; q < 9; ++q) xdG[q] = D1(ZGAM + q / 3, q % 3);
    xdW = get_d1(ZW);
    xda = get_d1(ZAL);
    xddW = get_d2(0);
#pragma unroll 1
    for (int J = 0; J < 3; ++J) {
      FxP U[3][3];
      {
        FxP G[6];
#pragma unroll
        for (int s = 0; s < 6; ++s) G[s] = mem.ld(FM_GS + 6 * J + s);
#pragma unroll
        for (int k = 0; k < 3; ++k) {
          const FxP r[3] = {G[sidx(k, 0)], G[sidx(k, 1)], G[sidx(k, 2)]};
#pragma unroll
          for (int l = 0; l < 3; ++l) U[k][l] = fx_split(fx_row(gus, l, r).fin<61>());  // 58.2
        }
      }
#pragma unroll 1
      for (int i = 0; i < 3; ++i) {
        FxDot t;
#pragma unroll
        for (int k = 0; k < 3; ++k) {
          FxP r[3];
          mem.row(FM_GU + 6 * k, i, r);
          t.add(fx_dot3(r, U[k]));
        }
        const int s = FM_R + fx_slot(i, J);
        const long long m = t.fin<61>();  // 59.4, six of these at most in one sum, 61 with t3
        mem.stm(s, mem.ldm(s) + (i == J ? m + m : m));
      }
      FxP G[6];
#pragma unroll
      for (int s = 0; s < 6; ++s) G[s] = mem.ld(FM_GU + 6 * J + s);
#pragma unroll
      for (int i = 0; i < 3; ++i)
#pragma unroll
        for (int j = i; j < 3; ++j) {
          const FxP r[3] = {G[sidx(i, 0)], G[sidx(i, 1)], G[sidx(i, 2)]};
          a.m[sidx(i, j)] += fx_dot3(r, U[j]).fin<61>();
        }
    }
    a.e = eGu + eU + 61;
#pragma unroll
    for (int s = 0; s < 6; ++s) a.m[s] += mem.ldm(FM_R + s);
    // (Gamma_d)^k Gamma_(ij)k
    {
      const FxBlk<3> gds = fx_plain(fx_times<59>(Gd, c.s1.v, c.s1.e - 1));
      FxDot d[6];
#pragma unroll
      for (int i = 0; i < 3; ++i) {
        FxP G[6];
#pragma unroll
        for (int s = 0; s < 6; ++s) G[s] = mem.ld(FM_GS + 6 * i + s);
#pragma unroll
        for (int j = 0; j < 3; ++j) {
          const FxP r[3] = {G[sidx(j, 0)], G[sidx(j, 1)], G[sidx(j, 2)]};
          FxDot t = fx_dot3(gds.v, r);
          if (i == j) t.twice();
          d[sidx(i, j)].add(t);
        }
      }
      b.e = gds.e + eGs + 60;
#pragma unroll
      for (int s = 0; s < 6; ++s) b.m[s] = d[s].fin<61>();  // 59.2
      fx_add(a, b);
    }
    // gt_k(i d_j) Gamt^k
    {
      const FxBlk<9> dG = fx_load<59, 9>(xdG, bad);
      const FxBlk<6> gh = fx_plain(fx_times<59>(mem.template get<6>(FM_G, eG), c.s1.v, c.s1.e - 1));
      b.e = gh.e + dG.e + 61;
#pragma unroll
      for (int i = 0; i < 3; ++i)
#pragma unroll
        for (int j = i; j < 3; ++j) {
          FxDot d;
#pragma unroll
          for (int k = 0; k < 3; ++k) {
            d.mac(gh.v[sidx(k, i)], dG.v[3 * k + j]);
            if (i != j) d.mac(gh.v[sidx(k, j)], dG.v[3 * k + i]);
          }
          if (i == j) d.twice();
          b.m[sidx(i, j)] = d.fin<61>();  // 59.6
        }
      fx_add(a, b);
    }
    eR = a.e;
#pragma unroll
    for (int s = 0; s < 6; ++s) mem.stm(FM_R + s, a.m[s]);
  }

  // d_i W / W, d_i alpha, and gt^ij d_j W / W
  FxBlk<3> dWi, dal, gdWi;
  {
    const FxBlk<1> siW = fx_norm<59>(fx_times<60>(iW, c.s1.v, c.s1.e));
    dWi = fx_norm<59>(fx_times<60>(fx_load<59, 3>(xdW.v, bad), siW.v[0], siW.e));
    dal = fx_norm<59>(fx_times<60>(fx_load<59, 3>(xda.v, bad), c.s1.v, c.s1.e));
    FxSum<3> m;
    m.e = gu.e + dWi.e + 61;
#pragma unroll
    for (int k = 0; k < 3; ++k) m.m[k] = fx_row(gu, k, dWi.v).fin<61>();  // 58.6
    gdWi = fx_norm<59>(m);
  }
  X6 xh = get_d2(1);
  FxBlk<1> z;
  int eDDW;
  {
    // D_i D_j W / W
    FxDot p, q;
    p.mac(c.kP.v, iW.v[0]);
    q.mac(c.kM.v, iW.v[0]);
    const FxP kp = fx_split(p.fin<59>()), km = fx_split(q.fin<59>());
    const FxBlk<6> h = fx_load<59, 6>(xddW.v, bad, c.poff);
    FxSum<6> a, b;
    a.e = h.e + c.kP.e + iW.e + 118;
    b.e = eGu + dWi.e + 60;
#pragma unroll
    for (int s = 0; s < 6; ++s) {
      FxDot u, v;
      u.mac(h.v[s], fx_pure(s) ? kp : km);
      a.m[s] = u.fin<59>();  // 59
#pragma unroll
      for (int k = 0; k < 3; ++k) v.mac(mem.ld(FM_GU + 6 * k + s), dWi.v[k]);
      b.m[s] = -v.fin<60>();  // 59.6
    }
    fx_add(a, b);
    const FxBlk<6> DDW = fx_norm_any(a);
    mem.put(FM_DDW, DDW);
    eDDW = DDW.e;
    // R^W_ij = D_i D_j W / W + gt_ij (D^l D_l W / W - 2 |dW|^2 / W^2)
    FxSum<1> x, t;
    x.m[0] = fx_trace(gu.v, DDW.v).fin<63>();  // 58.2
    x.e = gu.e + DDW.e + 63;
    t.m[0] = -fx_dot3(gdWi.v, dWi.v).fin<61>();  // 58.6
    t.e = gdWi.e + dWi.e + 62;
    fx_add(x, t);
    z = fx_norm_any(x);
  }
  // gt^ij times the scales of second derivatives
  FxBlk<6> guk;
  {
    FxSum<6> m;
    m.e = gu.e + c.kP.e + 60;
#pragma unroll
    for (int s = 0; s < 6; ++s) {
      FxDot d;
      d.mac(gu.v[s], fx_pure(s) ? c.kP.v : c.kM.v);
      m.m[s] = d.fin<60>();  // 58
    }
    guk = fx_norm<59>(m);
  }
  double xbe[18];
#pragma unroll
  for (int q = 0; q < 18; ++q) xbe[q] = D2(8 + q / 6, q % 6);
  int em = -1 << 20;
#pragma unroll 1
  for (int s = 0; s < 6; ++s) {
    // -1/2 gt^lm d_l d_m gt_ij and the terms in W
    const FxBlk<6> h = fx_load<59, 6>(xh.v, bad, c.poff);
    xh = get_d2(2 + s);  // the last one is alpha's
    long long m = mem.ldm(FM_R + s);
    int e = eR;
    fx_add1(m, e, -fx_trace(guk.v, h.v).fin<61>(), guk.e + h.e + 60);  // 60.2
    FxDot p;
    p.mac(mem.ld(FM_G + s), z.v[0]);
    fx_add1(m, e, p.fin<59>(), eG + z.e + 59);                // 59
    fx_add1(m, e, fx_join(mem.ld(FM_DDW + s)), eDDW);         // 59, 62.7 in all
    mem.stm(FM_R + s, m);
    mem.stm(FM_DDW + s, e);
    em = em > e ? em : e;
  }
  if constexpr (CONS) {
    FxSum<6> a;
    a.e = em;
#pragma unroll
    for (int s = 0; s < 6; ++s) a.m[s] = fx_shr(mem.ldm(FM_R + s), em - (int)mem.ldm(FM_DDW + s));
    const FxBlk<6> R = fx_norm_any(a);
    const double trR = fx_double(fx_trace(gu.v, R.v).fin<63>(), gu.e + R.e + 63);
    double x[6], xg[3], xd[18], xk[3];
#pragma unroll
    for (int s = 0; s < 6; ++s) x[s] = FLD(ZA + s);
#pragma unroll
    for (int q = 0; q < 18; ++q) xd[q] = D1(ZA + q / 3, q % 3);
#pragma unroll
    for (int i = 0; i < 3; ++i) {
      xg[i] = FLD(ZGAM + i);
      xk[i] = fma(2.0, D1(ZTH, i), D1(ZK, i));
    }
    const FxBlk<6> A = fx_load<59, 6>(x, bad);
    FxSum<9> m;
    m.e = gu.e + A.e + 61;
#pragma unroll
    for (int q = 0; q < 9; ++q) {
      const FxP b[3] = {A.v[sidx(0, q % 3)], A.v[sidx(1, q % 3)], A.v[sidx(2, q % 3)]};
      m.m[q] = fx_row(gu, q / 3, b).fin<61>();  // 58.6
    }
    const FxBlk<9> Am = fx_norm<59>(m);  // At^i_j, 3 i + j
    FxSum<6> u;
    u.e = gu.e + Am.e + 61;
#pragma unroll
    for (int i = 0; i < 3; ++i)
#pragma unroll
      for (int j = i; j < 3; ++j) u.m[sidx(i, j)] = fx_row(gu, j, Am.v + 3 * i).fin<61>();
    const FxBlk<6> Auu = fx_norm<59>(u);
    const double AA = fx_double(fx_trace(A.v, Auu.v).fin<63>(), A.e + Auu.e + 63), Kt = fma(2.0, Th, Kh);
    out(0, fma(fmul(W, W, K), trR, fma(fmul(2.0 / 3.0, Kt, K), Kt, -AA)));
    const FxBlk<18> dA = fx_load<59, 18>(xd, bad);
    const FxBlk<6> gs = fx_norm<59>(fx_times<60>(gu, c.s1.v, c.s1.e));
    const FxBlk<3> dd = fx_norm<59>(fx_times<60>(fx_load<59, 3>(xk, bad), c.ts1.v, c.ts1.e + 1));
    FxSum<3> t, b, d;
    t.e = eGu;
    b.e = gs.e + dA.e + 62;
    d.e = eGu + Am.e + 62;
#pragma unroll
    for (int i = 0; i < 3; ++i) {
      FxDot p, q;
      t.m[i] = 0;
#pragma unroll
      for (int j = 0; j < 3; ++j) {
#pragma unroll
        for (int k = 0; k < 3; ++k) {
          p.mac(gs.v[sidx(j, k)], dA.v[3 * sidx(i, k) + j]);
          q.mac(mem.ld(FM_GU + 6 * k + sidx(i, j)), Am.v[3 * j + k]);
        }
        t.m[i] += fx_join(mem.ld(FM_GU + 6 * j + sidx(i, j)));  // Gamma^j_ij, 60.6
      }
      b.m[i] = p.fin<62>();   // 59.2
      d.m[i] = -q.fin<62>();  // 59.2
    }
    fx_add(b, d);
    const FxBlk<3> bn = fx_norm_any(b), tn = fx_norm_any(t);
    FxSum<3> M, v;
    M.e = gu.e + bn.e + 61;
#pragma unroll
    for (int i = 0; i < 3; ++i) M.m[i] = fx_row(gu, i, bn.v).fin<61>();  // 58.6
    auto less = [&](const FxBlk<6>& a6, const FxBlk<3>& w, int times) {
      v.e = a6.e + w.e + 61;
#pragma unroll
      for (int i = 0; i < 3; ++i) v.m[i] = -times * fx_row(a6, i, w.v).fin<61>();
      fx_add(M, v);
    };
    less(Auu, tn, 1);
    less(Auu, dWi, 3);  // 60.2
    less(gu, dd, 1);
    v.e = Am.e + Gd.e + 61;
#pragma unroll
    for (int i = 0; i < 3; ++i) v.m[i] = -fx_dot3(Am.v + 3 * i, Gd.v).fin<61>();
    fx_add(M, v);
    fx_load_raw<59, 3>(xg, t, bad);
    v.e = Gd.e;
#pragma unroll
    for (int i = 0; i < 3; ++i) v.m[i] = -fx_join(Gd.v[i]);
    fx_add(t, v);
#pragma unroll
    for (int i = 0; i < 3; ++i) {
      out(1 + i, fx_double(M.m[i], M.e));
      out(4 + i, fx_double(t.m[i], t.e));
    }
    return !bad;
  } else {
    // second derivatives of the shift: gt^jk d_j d_k beta^i + 1/3 gt^ij d_j d_k beta^k
    int eTB;
    {
      const FxBlk<18> h = fx_load<59, 18>(xbe, bad, c.poff);
      FxSum<3> dv, sB, sL;
      dv.e = h.e + c.kP3.e + 61;
#pragma unroll
      for (int j = 0; j < 3; ++j) {
        FxDot d;
#pragma unroll
        for (int k = 0; k < 3; ++k) d.mac(h.v[6 * k + sidx(j, k)], j == k ? c.kP3.v : c.kM3.v);
        dv.m[j] = d.fin<61>();  // 58.6
      }
      const FxBlk<3> ddivb = fx_norm<59>(dv);  // 1/3 d_j d_k beta^k
      sL.e = gu.e + ddivb.e + 61;
      sB.e = guk.e + h.e + 61;
#pragma unroll
      for (int i = 0; i < 3; ++i) {
        sL.m[i] = fx_row(gu, i, ddivb.v).fin<61>();        // 58.6
        sB.m[i] = fx_trace(guk.v, h.v + 6 * i).fin<61>();  // 60.2
      }
      fx_add(sB, sL);
      eTB = sB.e;
#pragma unroll
      for (int i = 0; i < 3; ++i) mem.stm(FM_TB + i, sB.m[i]);  // 60.6
    }
    double xA[6], xdb[9];
#pragma unroll
    for (int s = 0; s < 6; ++s) xA[s] = FLD(ZA + s);
#pragma unroll
    for (int q = 0; q < 9; ++q) xdb[q] = D1(ZB + q / 3, q % 3);
    const FxBlk<1> fal = scalar(al);
    double trR, trDDa;
    int eTF;
    {
      FxBlk<6> R, DDa;
      FxSum<6> a, b, w;
      a.e = em;
#pragma unroll
      for (int s = 0; s < 6; ++s) a.m[s] = fx_shr(mem.ldm(FM_R + s), em - (int)mem.ldm(FM_DDW + s));
      R = fx_norm_any(a);
      // D_i D_j alpha with Gamma^k_ij - (delta^k_i d_j W + delta^k_j d_i W - gt_ij gt^kl d_l W) / W
      FxSum<1> zz;
      zz.m[0] = fx_dot3(gdWi.v, dal.v).fin<61>();
      zz.e = gdWi.e + dal.e + 61;
      const FxBlk<1> za = fx_norm<59>(zz);
      const FxBlk<6> h = fx_load<59, 6>(xh.v, bad, c.poff);
      a.e = h.e + c.kP.e + 59;
      b.e = eGu + dal.e + 60;
      w.e = dWi.e + dal.e + 60;
#pragma unroll
      for (int i = 0; i < 3; ++i)
#pragma unroll
        for (int j = i; j < 3; ++j) {
          const int s = sidx(i, j);
          FxDot p, q, u;
          p.mac(h.v[s], fx_pure(s) ? c.kP.v : c.kM.v);
          a.m[s] = p.fin<59>();  // 59
#pragma unroll
          for (int k = 0; k < 3; ++k) q.mac(mem.ld(FM_GU + 6 * k + s), dal.v[k]);
          b.m[s] = -q.fin<60>();  // 59.6
          u.mac(dWi.v[j], dal.v[i]);
          u.mac(dWi.v[i], dal.v[j]);
          w.m[s] = u.fin<60>();  // 59
        }
      fx_add(a, b);
      fx_add(a, w);
      const FxBlk<6> g = mem.template get<6>(FM_G, eG);
      b = fx_times<60>(g, za.v[0], za.e);  // 58
#pragma unroll
      for (int s = 0; s < 6; ++s) b.m[s] = -b.m[s];
      fx_add(a, b);  // 61
      DDa = fx_norm_any(a);
      trR = fx_double(fx_trace(gu.v, R.v).fin<63>(), gu.e + R.e + 63);
      trDDa = fx_double(fx_trace(gu.v, DDa.v).fin<63>(), gu.e + DDa.e + 63);
      // the trace-free part of alpha R_ij - D_i D_j alpha
      const FxBlk<1> zt = scalar(fmul(-1.0 / 3.0, fma(al, trR, -trDDa), K));
      a = fx_times<59>(R, fal.v[0], fal.e);
      b = fx_times<59>(g, zt.v[0], zt.e);
      fx_add(a, b);
      b.e = DDa.e;
#pragma unroll
      for (int s = 0; s < 6; ++s) b.m[s] = -fx_join(DDa.v[s]);
      fx_add(a, b);
      const FxBlk<6> tf = fx_norm_any(a);  // from 60.6
      mem.put(FM_TF, tf);
      eTF = tf.e;
    }
    const double W2 = fmul(W, W, K), Kt = fma(2.0, Th, Kh);

    const X3 xK = get_d1(ZK), xT = get_d1(ZTH);
    const double be[3] = {FLD(ZB), FLD(ZB + 1), FLD(ZB + 2)};
    const double gam[3] = {FLD(ZGAM), FLD(ZGAM + 1), FLD(ZGAM + 2)};
    // At with raised indices: Am[3 i + j] = At^i_j, Auu = At^ij
    double AA;
    int eA, eAU, eAB;
    {
      const FxBlk<6> A = fx_load<59, 6>(xA, bad);
      FxSum<9> m, kt;
      m.e = gu.e + A.e + 61;
#pragma unroll
      for (int q = 0; q < 9; ++q) {
        const FxP b[3] = {A.v[sidx(0, q % 3)], A.v[sidx(1, q % 3)], A.v[sidx(2, q % 3)]};
        m.m[q] = fx_row(gu, q / 3, b).fin<61>();  // 58.6
      }
      const FxBlk<9> Am = fx_norm<59>(m);
      FxSum<6> u;
      u.e = gu.e + Am.e + 61;
#pragma unroll
      for (int i = 0; i < 3; ++i)
#pragma unroll
        for (int j = i; j < 3; ++j) u.m[sidx(i, j)] = fx_row(gu, j, Am.v + 3 * i).fin<61>();
      const FxBlk<6> Auu = fx_norm<59>(u);
      AA = fx_double(fx_trace(A.v, Auu.v).fin<63>(), A.e + Auu.e + 63);
      // (Kt delta^k_i - 2 At^k_i) At_kj
      const FxBlk<1> fKt = scalar(Kt);
      m.e = Am.e + 1;
      kt.e = fKt.e;
#pragma unroll
      for (int q = 0; q < 9; ++q) {
        m.m[q] = -fx_join(Am.v[q]);
        kt.m[q] = q % 4 == 0 ? fx_join(fKt.v[0]) : 0;
      }
      fx_add(m, kt);
      const FxBlk<9> ak = fx_norm_any(m);
      u.e = ak.e + A.e + 61;
#pragma unroll
      for (int i = 0; i < 3; ++i)
#pragma unroll
        for (int j = i; j < 3; ++j) {
          FxDot d;
#pragma unroll
          for (int k = 0; k < 3; ++k) d.mac(ak.v[3 * k + i], A.v[sidx(k, j)]);
          u.m[sidx(i, j)] = d.fin<61>();  // 58.6
        }
      const FxBlk<6> ab = fx_norm<59>(u);
      mem.put(FM_A, A);
      mem.put(FM_AU, Auu);
      mem.put(FM_AB, ab);
      eA = A.e;
      eAU = Auu.e;
      eAB = ab.e;
    }

    // d_j beta^i, its trace, and -2/3 of that
    FxP p23, m23;
    double divb;
    int eDB;
    {
      const FxBlk<9> db = fx_norm<59>(fx_times<60>(fx_load<59, 9>(xdb, bad), c.s1.v, c.s1.e));
      const long long t = fx_join(db.v[0]) + fx_join(db.v[4]) + fx_join(db.v[8]);  // 60.6
      divb = fx_double(t, db.e);
      FxDot d;
      d.mac(fx_split(t), c.twothird.v);
      const long long u = d.fin<59>();  // 60, the units of db
      p23 = fx_split(u);
      m23 = fx_split(-u);
      mem.put(FM_DB, db);
      eDB = db.e;
    }
    // beta^i s1, for the advection terms
    const FxBlk<3> bes = fx_norm<59>(fx_times<60>(fx_load<59, 3>(be, bad), c.s1.v, c.s1.e));
    // The loops from here on finish one field after the other; next holds the
    // coming field's first derivatives and what out needs of it.
    struct Next {
      X3 d;
      typename OUT::Pre p;
    };
    auto get = [&](int f) { return Next{get_d1(f), out.load(f)}; };
    Next next = get(ZGAM);
    auto adv = [&](const X3& x, long long& m, int& e) {  // beta^i d_i f
      const FxBlk<3> d = fx_load<59, 3>(x.v, bad);
      m = fx_dot3(bes.v, d.v).fin<61>();  // 58.6
      e = bes.e + d.e + 61;
    };

    // Gamt^i
    {
      double x[3];
#pragma unroll
      for (int j = 0; j < 3; ++j) x[j] = fma(2.0, xK.v[j], xT.v[j]);  // d_j (2 Khat + Theta)
      const FxBlk<3> dd = fx_norm<59>(fx_times<60>(fx_load<59, 3>(x, bad), c.ts1.v, c.ts1.e));
      const FxBlk<6> Auu = mem.template get<6>(FM_AU, eAU);
      const FxBlk<1> k2 = scalar(fmul(-2.0 * P.kappa1, al, K));
#pragma unroll 1
      for (int i = 0; i < 3; ++i) {
        const Next now = next;
        next = get(i < 2 ? ZGAM + 1 + i : ZG);
        const double gami = i == 0 ? gam[0] : i == 1 ? gam[1] : gam[2];
        FxP v[6], r[3], ra[3];
#pragma unroll
        for (int s = 0; s < 6; ++s) v[s] = mem.ld(FM_GU + 6 * i + s);
        mem.row(FM_GI, i, r);
        mem.row(FM_AU, i, ra);
        FxSum<1> br, t;
        br.m[0] = fx_trace(v, Auu.v).fin<62>();  // Gamt^i_jk At^jk, 59.2
        br.e = eGu + Auu.e + 62;
        t.m[0] = -3 * fx_dot3(ra, dWi.v).fin<61>();  // 60.2
        t.e = Auu.e + dWi.e + 61;
        fx_add(br, t);
        t.m[0] = -fx_dot3(r, dd.v).fin<61>();  // 58.6
        t.e = gu.e + dd.e + 61;
        fx_add(br, t);
        const FxBlk<1> b = fx_norm_any(br);
        long long m;
        int e;
        adv(now.d, m, e);
        fx_add1(m, e, fx_times<59>(b, fal.v[0], 0).m[0], b.e + fal.e + 60);       // 2 alpha (...), 59
        fx_add1(m, e, -fx_dot3(ra, dal.v).fin<61>(), Auu.e + dal.e + 62);         // -2 At^ij d_j alpha, 58.6
        fx_add1(m, e, mem.ldm(FM_TB + i), eTB);                                   // 60.6
        const FxP gd = mem.ld(FM_GD + i);
        FxDot p;  // 2/3 (Gamma_d)^i div beta - (Gamma_d)^j d_j beta^i
        p.mac(gd, p23);
        const FxP w[3] = {mem.ld(FM_DB + 3 * i), mem.ld(FM_DB + 3 * i + 1), mem.ld(FM_DB + 3 * i + 2)};
        p.sub(fx_dot3(Gd.v, w));
        fx_add1(m, e, p.fin<60>(), Gd.e + eDB + 60);  // 60.4
        // -2 kappa1 alpha (Gamt^i - (Gamma_d)^i)
        FxSum<1> gm, gc;
        fx_load_raw<59, 1>(&gami, gm, bad);
        gc.m[0] = -fx_join(gd);
        gc.e = Gd.e;
        fx_add(gm, gc);
        const FxBlk<1> gn = fx_norm_any(gm);
        fx_add1(m, e, fx_times<60>(gn, k2.v[0], 0).m[0], gn.e + k2.e + 60);  // 58, 62 in all
        out(ZGAM + i, fx_double(m, e), now.p);
      }
    }
    // gt_ij and At_ij
    {
      const FxBlk<1> fW2 = scalar(W2);
#pragma unroll 1
      for (int s = 0; s < 6; ++s) {
        const int i = fx_slot_i(s), j = fx_slot_j(s);
        Next now = next;
        next = get(ZA + s);
        FxP ri[3], rj[3];
        const FxP di[3] = {mem.ld(FM_DB + i), mem.ld(FM_DB + 3 + i), mem.ld(FM_DB + 6 + i)};
        const FxP dj[3] = {mem.ld(FM_DB + j), mem.ld(FM_DB + 3 + j), mem.ld(FM_DB + 6 + j)};
        const FxP A = mem.ld(FM_A + s);
        long long m;
        int e;
        FxDot l, p, q, w;
        mem.row(FM_G, i, ri);
        mem.row(FM_G, j, rj);
        l = fx_dot3(ri, dj);
        l.add(fx_dot3(rj, di));
        l.mac(mem.ld(FM_G + s), m23);
        adv(now.d, m, e);
        fx_add1(m, e, l.fin<60>(), eG + eDB + 60);  // 61
        p.mac(fal.v[0], A);
        fx_add1(m, e, -p.fin<60>(), fal.e + eA + 61);  // 58
        out(ZG + s, fx_double(m, e), now.p);
        now = next;
        next = get(s < 5 ? ZG + 1 + s : ZW);
        mem.row(FM_A, i, ri);
        mem.row(FM_A, j, rj);
        l = fx_dot3(ri, dj);
        l.add(fx_dot3(rj, di));
        l.mac(A, m23);
        adv(now.d, m, e);
        fx_add1(m, e, l.fin<60>(), eA + eDB + 60);  // 61
        q.mac(fal.v[0], mem.ld(FM_AB + s));
        fx_add1(m, e, q.fin<59>(), fal.e + eAB + 59);  // 59
        w.mac(fW2.v[0], mem.ld(FM_TF + s));
        fx_add1(m, e, w.fin<59>(), fW2.e + eTF + 59);  // 59
        out(ZA + s, fx_double(m, e), now.p);
      }
    }
    // W, Khat, Theta, alpha and beta^i: the scalar parts in FP64
    {
      const double third = 1.0 / 3.0, twothird = 2.0 / 3.0;
      auto put = [&](int q, double v) {
        mem.stm(FM_GU + q, fx_shl((long long)fx_dhi(v), 32) | fx_dlo(v));
      };
      put(0, fmul(fmul(third, W, K), fma(al, Kt, -divb), K));
      put(1, fma(al, fma(fmul(third, Kt, K), Kt, AA), fma(fmul(al, P.kappa1 * (1.0 - P.kappa2), K), Th, fmul(-W2, trDDa, K))));
      put(2, fma(fmul(0.5, al, K), fma(fmul(twothird, Kt, K), Kt, fma(W2, trR, -AA)),
                 fmul(fmul(-al, P.kappa1 * (2.0 + P.kappa2), K), Th, K)));
      put(3, fmul(fmul(-2.0, al, K), Kh, K));
#pragma unroll
      for (int i = 0; i < 3; ++i) put(4 + i, fma(0.75, gam[i], fmul(-eta, be[i], K)));
#pragma unroll 1
      for (int q = 0; q < 7; ++q) {
        const int f = q < 2 ? 7 * q : q + 15;
        const Next now = next;
        next = get(q < 1 ? ZK : q < 6 ? q + 16 : ZB + 2);
        long long m;
        int e;
        adv(now.d, m, e);
        const long long v = mem.ldm(FM_GU + q);
        out(f, fadd(fx_make((int)(v >> 32), (int)v), fx_double(m, e), K), now.p);
      }
    }
    return !bad;
  }
#undef FLD
#undef D1
#undef D2
}

}  // namespace sc
