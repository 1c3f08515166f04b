// sc_z4c.cu -- Z4c right-hand side (Sec. III.A, vacuum, puncture gauge with
// constant eta), Kreiss-Oliger dissipation (Sec. III.C, r = 4) and the fused
// RK4 stage update, plus the constraint evaluation.
//
// Two passes per stage, both over the interior tiles of a level:
//   1. the derivative pass computes the centred first derivatives of every
//      field, the second derivatives of W, gt_ij, alpha and beta^i, and the
//      KO sum sum_d delta_d^6 u, and stores them in a scratch array indexed
//      like the level array: scratch[q * fs + cell].  The stored values are
//      the stencils' integer-weight sums, without their 1/h and 1/h^2
//      factors (see Z4cUnits): a multiplication issues at the slower of
//      the two FP64 rates, and the consumers fold the factors into FMA
//      constants they evaluate anyway.
//   2. z4c_stage_kernel: one thread per cell reads the 22 fields and their
//      derivatives, evaluates the right-hand side, adds dissipation and
//      performs the RK4 stage update.
// FP64 is the scarce resource on this GPU (the FP64 pipe issues 1/64 of the
// FP32 rate), so the stencil sums (sc_fixed.cuh) and the tensor sums that use
// their operands many times (sc_z4c_point.cuh) are formed in integers; the FP64
// forms beside them are for the cells whose values the integers do not take.
#include "sc_device.cuh"
#include "sc_z4c_point.cuh"

namespace sc {
namespace {

constexpr int kThreads = 256;

// slot of field f among the fields with second derivatives, -1 if none
__host__ __device__ inline int d2_slot(int f) {
  if (f == ZW) return 0;
  if (f >= ZG && f < ZG + 6) return 1 + (f - ZG);
  if (f == ZAL) return 7;
  if (f >= ZB && f < ZB + 3) return 8 + (f - ZB);
  return -1;
}

// One-kernel form of the derivative pass (4th order): one thread per (cell,
// field), mixed derivatives from the direct 16-point product stencil.
// Stored scales as the two-kernel form: 12 h d_i u, 12 h^2 d_i^2 u,
// 144 h^2 d_i d_j u, and the raw Kreiss-Oliger sum.
__global__ void __launch_bounds__(kThreads) z4c_derivs_kernel(const double* __restrict__ Y, double* __restrict__ S,
                                                             long fs, int sy_, int sz_,
                                                             const Tile* __restrict__ tiles, int ntiles) {
  const long st[3] = {1, (long)sy_, (long)sz_};
  for (int t = blockIdx.x; t < ntiles; t += gridDim.x) {
    const Tile T = tiles[t];
    const int n = T.nx * T.ny * T.nz;
    for (int q = threadIdx.x; q < n * kNZ4c; q += blockDim.x) {
      const int f = q / n;
      const int c = q - f * n;
      const int i = c % T.nx;
      const int j = (c / T.nx) % T.ny;
      const int k = c / (T.nx * T.ny);
      const long o = (T.z0 + k) * st[2] + (T.y0 + j) * st[1] + (T.x0 + i);
      const double* u = Y + (long)f * fs + o;
      const double u0 = u[0];
      double p1[3], p2[3], P3 = 0.0;
#pragma unroll
      for (int d = 0; d < 3; ++d) {
        const long s = st[d];
        const double a1 = u[-s], b1 = u[s], a2 = u[-2 * s], b2 = u[2 * s];
        p1[d] = a1 + b1;
        p2[d] = a2 + b2;
        P3 += u[-3 * s] + u[3 * s];
        // 12 h u' = u_-2 - 8 u_-1 + 8 u_1 - u_2
        S[(long)(Q_D1 + 3 * f + d) * fs + o] = fma(8.0, b1 - a1, a2 - b2);
      }
      // Kreiss-Oliger: sum_d (u_-3 - 6 u_-2 + 15 u_-1 - 20 u_0 + 15 u_1 - 6 u_2 + u_3)
      const double P1 = p1[0] + p1[1] + p1[2], P2 = p2[0] + p2[1] + p2[2];
      S[(long)(Q_KO + f) * fs + o] = fma(15.0, P1, fma(-6.0, P2, fma(-60.0, u0, P3)));
      const int sl = d2_slot(f);
      if (sl < 0) continue;
      double* d2 = S + (long)(Q_D2 + 6 * sl) * fs + o;
      // pure: 12 h^2 u'' = -u_-2 + 16 u_-1 - 30 u_0 + 16 u_1 - u_2
      d2[0 * fs] = fma(-30.0, u0, fma(16.0, p1[0], -p2[0]));
      d2[3 * fs] = fma(-30.0, u0, fma(16.0, p1[1], -p2[1]));
      d2[5 * fs] = fma(-30.0, u0, fma(16.0, p1[2], -p2[2]));
      // mixed: 144 h^2 d_i d_j u, the product of the two first-derivative stencils
      const int pa[3] = {0, 0, 1}, pb[3] = {1, 2, 2}, slot[3] = {1, 2, 4};
#pragma unroll
      for (int m = 0; m < 3; ++m) {
        const long sa = st[pa[m]], sb = st[pb[m]];
        double D[4];
        const int offs[4] = {-2, -1, 1, 2};
#pragma unroll
        for (int r = 0; r < 4; ++r) {
          const double* v = u + offs[r] * sb;
          D[r] = fma(8.0, v[sa] - v[-sa], v[-2 * sa] - v[2 * sa]);
        }
        d2[slot[m] * fs] = fma(8.0, D[2] - D[1], D[0] - D[3]);
      }
    }
  }
}


// ---------------------------------------------------------------------------
// Evolution form of the derivative pass, in two kernels.  The mixed second
// derivatives are the product of two first-derivative stencils, so
//   d_x d_y u = D_y (D_x u),  d_x d_z u = D_z (D_x u),  d_y d_z u = D_z (D_y u)
// exactly (the same 16-point stencil, summed in another order).  The first
// kernel stores D_x u and D_y u of the 11 fields with second derivatives on
// row segments covering the interior and its 2-cell extension in y and z
// (D_x) or in z (D_y); the second kernel computes everything else per
// interior cell and differentiates the stored first derivatives for the
// mixed terms: 4 FP64 operations per mixed derivative instead of 16.

// field of Hessian slot s (W, gt x6, alpha, beta x3): slots 0..6 -> fields 0..6, 7..10 -> 18..21
__device__ __forceinline__ int d2_field(int s) { return s <= 6 ? s : s + 11; }

// Centred first derivative as the integer-weight sum, lo[m - 1] = v_-m, hi[m - 1] = v_m:
// 4th order 8 (v_1 - v_-1) - (v_2 - v_-2) (= 12 h u'), 8th order
// 672 d1 - 168 d2 + 32 d3 - 3 d4 (= 840 h u'), dm = v_m - v_-m, in FP64.
template <int ORD, class KT>
__device__ __forceinline__ double dfirst_fp64(const double* lo, const double* hi, const KT& K) {
  if (ORD == 4) return fma(8.0, hi[0], fma(-8.0, lo[0], fsub(lo[1], hi[1], K)));
  return fma(672.0, fsub(hi[0], lo[0], K),
             fma(-168.0, fsub(hi[1], lo[1], K),
                 fma(32.0, fsub(hi[2], lo[2], K), fmul(-3.0, fsub(hi[3], lo[3], K), K))));
}

// The same in aligned integers (sc_fixed.cuh), or in FP64 where the values do not allow that.
template <int ORD, class KT>
__device__ __forceinline__ double dfirst(const double* lo, const double* hi, const KT& K) {
  using F = FxSums<ORD>;
  const int E1 = max(fx_exp(lo[0]), fx_exp(hi[0])), E2 = max(fx_exp(lo[1]), fx_exp(hi[1]));
  int E = max(E1, E2);
#pragma unroll
  for (int m = 2; m < ORD / 2; ++m) E = max(E, max(fx_exp(lo[m]), fx_exp(hi[m])));
  if (aligned_ok(E) && (ORD == 4 || E - E1 <= F::kExcess1 << 20 || E - E2 <= F::kExcess2 << 20)) return F::first(lo, hi, E);
  unsigned any = 0;
#pragma unroll
  for (int m = 0; m < ORD / 2; ++m) any |= zero_bits(lo[m]) | zero_bits(hi[m]);
  if (any == 0) return 0.0;
  return dfirst_fp64<ORD>(lo, hi, K);
}

template <int ORD, class KT = FmaK>
__global__ void __launch_bounds__(128) z4c_dxy_kernel(const double* __restrict__ Y, double* __restrict__ S, long fs,
                                                     int sy_, const RowSeg* __restrict__ segs, int nsegs, KT K) {
  constexpr int R = ORD / 2;
  const long sy = sy_;
  for (int sgi = blockIdx.x; sgi < nsegs; sgi += gridDim.x) {
    const RowSeg sg = segs[sgi];
    for (int q = threadIdx.x; q < sg.n * 11; q += blockDim.x) {
      const int slot = q / sg.n;
      const long o = sg.off + (q - slot * sg.n);
      const int f = d2_field(slot);
      const double* u = Y + (long)f * fs + o;
      double lo[R], hi[R];
      if (sg.which & 1) {
#pragma unroll
        for (int m = 1; m <= R; ++m) {
          lo[m - 1] = u[-m];
          hi[m - 1] = u[m];
        }
        S[(long)(Q_D1 + 3 * f + 0) * fs + o] = dfirst<ORD>(lo, hi, K);
      }
      if (sg.which & 2) {
#pragma unroll
        for (int m = 1; m <= R; ++m) {
          lo[m - 1] = u[-m * sy];
          hi[m - 1] = u[m * sy];
        }
        S[(long)(Q_D1 + 3 * f + 1) * fs + o] = dfirst<ORD>(lo, hi, K);
      }
    }
  }
}

// The sums of one cell that need u at the cell and its neighbours along the
// three axes (lo[d][m - 1] = u at -m along d), in FP64: D_d of the axes in
// dmask, the Kreiss-Oliger sum and, for d2 != null, the pure second
// derivatives.  The form of the cells that aligned_ok refuses.
template <int ORD, class KT>
__device__ __forceinline__ void cell_sums_fp64(double u0, const double (*lo)[ORD == 4 ? 3 : 4],
                                               const double (*hi)[ORD == 4 ? 3 : 4], double* d1, double* ko,
                                               double* d2, const KT& K) {
  double P[3] = {0.0, 0.0, 0.0};
#pragma unroll
  for (int d = 0; d < 3; ++d) {
    double p[4] = {0.0, 0.0, 0.0, 0.0};
#pragma unroll
    for (int m = 0; m < (ORD == 4 ? 3 : 4); ++m) p[m] = fadd(lo[d][m], hi[d][m], K);
    d1[d] = dfirst_fp64<ORD>(lo[d], hi[d], K);
    if (ORD == 4) d2[d] = fma(16.0, p[0], fma(-30.0, u0, -p[1]));
    else d2[d] = fma(-14350.0, u0, fma(8064.0, p[0], fma(-1008.0, p[1], fma(128.0, p[2], fmul(-9.0, p[3], K)))));
#pragma unroll
    for (int m = 0; m < 3; ++m) P[m] = d == 0 ? p[m] : fadd(P[m], p[m], K);
  }
  *ko = fma(15.0, P[0], fma(-6.0, P[1], fma(-60.0, u0, P[2])));
}

// One block per (tile, field): a thread per (x, y) column walks z with the
// packed values at z-W..z+W in registers (W = max(R, 3), R = ORD/2 the derivative
// radius, 3 the Kreiss-Oliger radius) and puts its centre value, and up to two
// of the tile's halo cells, into a shared plane, so that a value is unpacked once
// or twice instead of 19 (25) times.  Tiles: at most kDerivCols columns, 32 wide,
// 32 high; a plane then holds at most 38 x 14 (40 x 16) values.  At 4th order D_x
// and D_y along z are windows in registers too; at 8th order these would spill,
// and are read again (L1).  Integer ALU 45%, latency of 16 warps: 262,144 cells with
// the row pass before it, 0.251 ms with a thread per column and no sharing, 0.209
// so (0.200 with one alignment for a cell's whole star, whose error in a derivative was
// relative to the values along the other axes too); 110,592 cells 0.119 and 0.111; 8th order, 262,144
// cells, 0.347 and 0.357 (0.329).  With the mixed derivatives in FP64 instead: 0.211 and
// 0.444 (star alignment); with three or four blocks per SM and reads in place of the
// windows: 0.219 and 0.238.
template <int ORD, class KT = FmaK>
__global__ void __launch_bounds__(kDerivCols, 2)
    z4c_derivs_split_kernel(const double* __restrict__ Y, double* __restrict__ S, long fs, int sy_, int sz_,
                            const Tile* __restrict__ tiles, int ntiles, KT K) {
  using F = FxSums<ORD>;
  constexpr int R = ORD / 2;
  constexpr int WR = R > 3 ? R : 3;
  constexpr int NW = 2 * WR + 1;
  constexpr int ND = 2 * R + 1;
  constexpr bool kWindows = ORD == 4;
  __shared__ long long planes[2][plane_values(WR)];
  const long sy = sy_, sz = sz_;
  int buf = 0;
  for (int item = blockIdx.x; item < ntiles * kNZ4c; item += gridDim.x) {
    const int t = item / kNZ4c, f = item - t * kNZ4c;
    const Tile T = tiles[t];
    const int ncol = T.nx * T.ny, pitch = T.nx + 2 * WR;
    const double* base = Y + (long)f * fs + (long)T.z0 * sz + (long)T.y0 * sy + T.x0;
    const bool active = (int)threadIdx.x < ncol;
    const int i = threadIdx.x % T.nx, j = threadIdx.x / T.nx;
    const int own = (j + WR) * pitch + i + WR;
    const double* u = base + (long)j * sy + i;
    const long o0 = (long)T.z0 * sz + (long)(T.y0 + j) * sy + (T.x0 + i);
    int hs[2];
    const double* hp[2];
#pragma unroll
    for (int r = 0; r < 2; ++r) {
      long off;
      halo_cell<WR>(T, threadIdx.x + r * kDerivCols, sy, &hs[r], &off);
      hp[r] = base;
      if (hs[r] >= 0) hp[r] += off;
    }
    const int sl = d2_slot(f);
    const double* Dx = S + (long)(Q_D1 + 3 * f + 0) * fs + o0;
    const double* Dy = S + (long)(Q_D1 + 3 * f + 1) * fs + o0;
    long long w[NW];       // packed u at z-WR..z+WR
    double wx[ND], wy[ND];  // kWindows: D_x, D_y at z-R..z+R (Hessian fields)
    double hv[2] = {hs[0] >= 0 ? *hp[0] : 0.0, hs[1] >= 0 ? *hp[1] : 0.0};
    double un = 0.0;
    if (active) {
#pragma unroll
      for (int m = 0; m < NW - 1; ++m) w[m] = fx_pack(u[(m - WR) * sz]);
      un = u[WR * sz];
      if (kWindows && sl >= 0) {
#pragma unroll
        for (int m = 0; m < ND - 1; ++m) {
          wx[m] = Dx[(m - R) * sz];
          wy[m] = Dy[(m - R) * sz];
        }
      }
    }
#pragma unroll 1
    for (int k = 0; k < T.nz; ++k, buf ^= 1) {
      long long* pl = planes[buf];
      if (active) pl[own] = w[WR];
      const bool more = k + 1 < T.nz;
#pragma unroll
      for (int r = 0; r < 2; ++r)
        if (hs[r] >= 0) {
          pl[hs[r]] = fx_pack(hv[r]);
          if (more) hv[r] = hp[r][(k + 1) * sz];
        }
      // (the two planes alternate, also from one item to the next: a plane is
      // written again only after every thread has passed the next barrier)
      __syncthreads();
      if (!active) continue;
      w[NW - 1] = fx_pack(un);
      if (more) un = u[(k + 1 + WR) * sz];
      const long o = o0 + k * sz;
      if (kWindows && sl >= 0) {
        wx[ND - 1] = Dx[(k + R) * sz];
        wy[ND - 1] = Dy[(k + R) * sz];
      }
      auto at = [&](int dim, int m) {
        return dim == 0 ? pl[own + m] : dim == 1 ? pl[own + m * pitch] : w[WR + m];
      };
      // Each axis has an alignment of its own; one whose first derivative would lose by
      // that (its values far below u0 or those at +-3), and one of zeros, sends the cell to FP64.
      int Ed[3];
      bool ok = true;
#pragma unroll
      for (int dim = 0; dim < 3; ++dim) {
        const int E1 = max(fx_pexp(at(dim, -1)), fx_pexp(at(dim, 1)));
        const int E2 = max(fx_pexp(at(dim, -2)), fx_pexp(at(dim, 2)));
        int E = max(fx_pexp(w[WR]), max(E1, E2));
#pragma unroll
        for (int m = 3; m <= WR; ++m) E = max(E, max(fx_pexp(at(dim, -m)), fx_pexp(at(dim, m))));
        Ed[dim] = E;
        ok = ok && packed_ok(E) && (E - E1 <= F::kExcess1 || E - E2 <= F::kExcess2);
      }
      double* d1 = S + (long)(Q_D1 + 3 * f) * fs + o;
      double* d2 = S + (long)(Q_D2 + 6 * sl) * fs + o;
      double* ko = S + (long)(Q_KO + f) * fs + o;
      if (ok) {
        const int E = max(max(Ed[0], Ed[1]), Ed[2]);
        typename F::Ko sum;
#pragma unroll
        for (int dim = 0; dim < 3; ++dim) {
          long long l[WR], h[WR];
#pragma unroll
          for (int m = 0; m < WR; ++m) {
            l[m] = at(dim, -m - 1);
            h[m] = at(dim, m + 1);
          }
          const typename F::Axis A(l, h, w[WR], Ed[dim]);
          const int Ef = packed_field(Ed[dim]);
          // D_x, D_y of the Hessian fields are there already (z4c_dxy_kernel)
          if (sl < 0 || dim == 2) d1[dim * fs] = A.first(Ef);
          if (sl >= 0) d2[(dim == 0 ? 0 : dim == 1 ? 3 : 5) * fs] = A.second(Ef);
          sum.add(A, Ed[dim], E);
        }
        *ko = sum.get(w[WR], E);
      } else {
        const double* v = u + k * sz;
        double fl[3][ORD == 4 ? 3 : 4], fh[3][ORD == 4 ? 3 : 4], e1[3], e2[3], eko;
        const long st[3] = {1, sy, sz};
        unsigned any = zero_bits(v[0]);
#pragma unroll
        for (int dim = 0; dim < 3; ++dim)
#pragma unroll
          for (int m = 1; m <= WR; ++m) {
            fl[dim][m - 1] = v[-m * st[dim]];
            fh[dim][m - 1] = v[m * st[dim]];
            any |= zero_bits(fl[dim][m - 1]) | zero_bits(fh[dim][m - 1]);
          }
        if (any) {
          cell_sums_fp64<ORD>(v[0], fl, fh, e1, &eko, e2, K);
        } else {
          eko = 0.0;
#pragma unroll
          for (int dim = 0; dim < 3; ++dim) e1[dim] = e2[dim] = 0.0;
        }
        *ko = eko;
#pragma unroll
        for (int dim = 0; dim < 3; ++dim) {
          if (sl < 0 || dim == 2) d1[dim * fs] = e1[dim];
          if (sl >= 0) d2[(dim == 0 ? 0 : dim == 1 ? 3 : 5) * fs] = e2[dim];
        }
      }
      if (sl >= 0) {
        // mixed: the first-derivative stencil applied to the stored D_x (along y and z) and D_y (along z)
        auto mixed = [&](const double* d, long st) {
          double ml[R], mh[R];
#pragma unroll
          for (int m = 1; m <= R; ++m) {
            ml[m - 1] = d[-m * st];
            mh[m - 1] = d[m * st];
          }
          return dfirst<ORD>(ml, mh, K);
        };
        d2[1 * fs] = mixed(Dx + k * sz, sy);
        if (kWindows) {
          auto window = [&](double* v) {
            double ml[R], mh[R];
#pragma unroll
            for (int m = 1; m <= R; ++m) {
              ml[m - 1] = v[R - m];
              mh[m - 1] = v[R + m];
            }
#pragma unroll
            for (int m = 0; m < ND - 1; ++m) v[m] = v[m + 1];
            return dfirst<ORD>(ml, mh, K);
          };
          d2[2 * fs] = window(wx);
          d2[4 * fs] = window(wy);
        } else {
          d2[2 * fs] = mixed(Dx + k * sz, sz);
          d2[4 * fs] = mixed(Dy + k * sz, sz);
        }
      }
#pragma unroll
      for (int m = 0; m < NW - 1; ++m) w[m] = w[m + 1];
    }
  }
}

// Dissipation and the stage update of one field at one cell.
template <int FORM, class KT>
struct StageUpdate {
  const StageArgs& a;
  const double* S;
  long o;
  double ko;
  KT K;
  struct Pre {
    double ko, yn, k1, k2, k3;
  };
  __device__ __forceinline__ Pre load(int f) const {
    const long fo = (long)f * a.fs + o;
    Pre p;
    p.ko = S[(long)(Q_KO + f) * a.fs + o];
    if (FORM != kStageNone) p.yn = a.yn[fo];
    if (FORM == kStageRk4 || FORM == kStageTwo) p.k1 = a.k1[fo];
    if (FORM == kStageRk4) {
      p.k2 = a.k2[fo];
      p.k3 = a.k3[fo];
    }
    return p;
  }
  __device__ __forceinline__ void operator()(int f, double rhs, const Pre& p) const {
    const long fo = (long)f * a.fs + o;
    const double kv = fma(ko, p.ko, rhs);
    a.k[fo] = kv;
    if (FORM == kStageSingle) {
      a.out[fo] = fma(a.cdt, kv, p.yn);
    } else if (FORM == kStageRk4) {
      const double s = fadd(fma(2.0, p.k3, fma(2.0, p.k2, p.k1)), kv, K);
      a.out[fo] = fma(a.cdt, s, p.yn);
    } else if (FORM == kStageTwo) {
      a.out[fo] = fma(a.cdt, kv, fma(a.c1dt, p.k1, p.yn));
    }
  }
};

// FORM: the stage update of StageArgs (kStageSingle, kStageRk4, kStageTwo,
// kStageNone), fixed at compile time.  A block takes the up to 64 cells of a
// run, consecutive over the rows of a box, so that every lane has a cell whatever
// the extents (tiles of 32 x 2 cells left 38% of the lanes idle at 20 or 40 cells
// a row, 25% at 48), and the 152 SMs share the 125 runs of a 20^3 level.  BPS (a
// choice of sc_autotune): 2 leaves 255 registers a thread, 3 has six blocks of 168
// registers per SM.
// Bound by the FP64 pipe, 72% of its rate with BPS 3 (of 11,793 instructions a cell
// 564 are FP64, each 64 cycles of a scheduler's pipe), and by latency on small levels.
// 262,144 cells: 0.501 ms in FP64 throughout, 0.329 with BPS 3, 0.361 with 2; 110,592
// cells: 0.290, 0.150, 0.161; 8,000 cells: 0.041, 0.035, 0.035.  More of the sums in integers
// (second derivatives contracted with gt^ij too: 512 FP64 instructions) ran in 0.349.
template <int FORM, int BPS, class KT = FmaK>
__global__ void __launch_bounds__(kRunCells, 2 * BPS)
    z4c_stage_kernel(StageArgs a, const double* __restrict__ S, Z4cParams P, const CellRun* __restrict__ runs, int nruns,
                     const __grid_constant__ Z4cUnits c, KT K) {
  __shared__ long long slots[FM_SLOTS * kRunCells];
  __shared__ short exps[FM_SLOTS * kRunCells];
  const FxMem<kRunCells> mem{slots + threadIdx.x, exps + threadIdx.x};
  const double ko = P.ko_sigma / (64.0 * a.h);  // (as a kernel argument: 7% slower)
  for (int u = blockIdx.x; u < nruns; u += gridDim.x) {
    const CellRun R = runs[u];
    if ((int)threadIdx.x >= R.n) continue;
    const int q = R.first + threadIdx.x, row = q / R.nx, z = row / R.ny;
    const long o = R.off + (long)z * a.sz + (long)(row - z * R.ny) * a.sy + (q - row * R.nx);
    z4c_rhs_point<Connection>(a.Y, S, a.fs, o, P, a.eta ? a.eta[o] : P.eta, c, mem, K,
                              StageUpdate<FORM, KT>{a, S, o, ko, K});
  }
}

// Constraints at the interior cells of one box (z4c_constraints_point):
// out[c * out_stride + cell], cells numbered x-fastest within the box.  One thread
// per cell, 64 cells a block, so that an 11,000-cell box reaches every SM.
__global__ void __launch_bounds__(kRunCells, 4)
    z4c_constraints_kernel(const double* __restrict__ Y, const double* __restrict__ S, double* __restrict__ out, long fs,
                           int sy, int sz, const __grid_constant__ Z4cUnits c, long out_stride, int bx, int by, int bz,
                           int nbx, int nby, int nbz, FmaK K) {
  __shared__ long long slots[FM_SLOTS * kRunCells];
  __shared__ short exps[FM_SLOTS * kRunCells];
  const FxMem<kRunCells> mem{slots + threadIdx.x, exps + threadIdx.x};
  const long cells = (long)nbx * nby * nbz;
  for (long cell = (long)blockIdx.x * kRunCells + threadIdx.x; cell < cells; cell += (long)gridDim.x * kRunCells) {
    const int x = (int)(cell % nbx), y = (int)(cell / nbx % nby), z = (int)(cell / ((long)nbx * nby));
    const long o = (long)(bz + z) * sz + (long)(by + y) * sy + bx + x;
    z4c_constraints_point<Connection>(Y, S, fs, o, c, mem, K, [&](int q, double v) { out[q * out_stride + cell] = v; });
  }
}

// Persistent grids: each Z4c kernel is launched with (SMs x resident blocks
// per SM) blocks at most, looping over its tiles, so a level's work is spread
// evenly over the whole GPU instead of leaving a partial last wave.
struct GridCaps {
  int ready = 0;
  int stage[4] = {608, 608, 608, 912};  // by warps per scheduler of the build (2 or 3)
  int derivs[2] = {456, 304}, dxy = 2432;  // derivs: 4th, 8th order
};
GridCaps g_caps[64];

inline const GridCaps& caps() {
  int dev = 0;
  cudaGetDevice(&dev);
  return g_caps[dev & 63];
}

}  // namespace

cudaError_t z4c_init_launch_config() {
  int dev = 0, nsm = 0, occ = 0;
  cudaError_t e = cudaGetDevice(&dev);
  if (e != cudaSuccess) return e;
  GridCaps& c = g_caps[dev & 63];
  if (c.ready) return cudaSuccess;
  if ((e = cudaDeviceGetAttribute(&nsm, cudaDevAttrMultiProcessorCount, dev)) != cudaSuccess) return e;
  if ((e = cudaOccupancyMaxActiveBlocksPerMultiprocessor(&occ, z4c_stage_kernel<kStageSingle, 2>, kRunCells, 0)) !=
      cudaSuccess)
    return e;
  c.stage[2] = nsm * (occ > 0 ? occ : 1);
  if ((e = cudaOccupancyMaxActiveBlocksPerMultiprocessor(&occ, z4c_stage_kernel<kStageSingle, 3>, kRunCells, 0)) !=
      cudaSuccess)
    return e;
  c.stage[3] = nsm * (occ > 0 ? occ : 1);
  if ((e = cudaOccupancyMaxActiveBlocksPerMultiprocessor(&occ, z4c_derivs_split_kernel<4>, kDerivCols, 0)) != cudaSuccess)
    return e;
  c.derivs[0] = nsm * (occ > 0 ? occ : 1);
  if ((e = cudaOccupancyMaxActiveBlocksPerMultiprocessor(&occ, z4c_derivs_split_kernel<8>, kDerivCols, 0)) != cudaSuccess)
    return e;
  c.derivs[1] = nsm * (occ > 0 ? occ : 1);
  if ((e = cudaOccupancyMaxActiveBlocksPerMultiprocessor(&occ, z4c_dxy_kernel<8>, 128, 0)) != cudaSuccess) return e;
  c.dxy = nsm * (occ > 0 ? occ : 1);
  c.ready = 1;
  return cudaSuccess;
}

cudaError_t launch_z4c_derivs(const double* Y, double* scratch, long fs, int sy, int sz, const Tile* tiles,
                              int ntiles, cudaStream_t s) {
  if (ntiles == 0) return cudaSuccess;
  const int grid = ntiles < sm_count() * 16 ? ntiles : sm_count() * 16;
  z4c_derivs_kernel<<<grid, kThreads, 0, s>>>(Y, scratch, fs, sy, sz, tiles, ntiles);
  return cudaGetLastError();
}

namespace {

template <class KT>
void launch_dxy(const double* Y, double* scratch, long fs, int sy, const RowSeg* segs, int nsegs, int grid,
                cudaStream_t s, int order, const KT& K) {
  if (order == 8) z4c_dxy_kernel<8, KT><<<grid, 128, 0, s>>>(Y, scratch, fs, sy, segs, nsegs, K);
  else z4c_dxy_kernel<4, KT><<<grid, 128, 0, s>>>(Y, scratch, fs, sy, segs, nsegs, K);
}

template <class KT>
void launch_derivs(const double* Y, double* scratch, long fs, int sy, int sz, const Tile* tiles, int ntiles, int grid,
                   cudaStream_t s, int order, const KT& K) {
  if (order == 8) z4c_derivs_split_kernel<8, KT><<<grid, kDerivCols, 0, s>>>(Y, scratch, fs, sy, sz, tiles, ntiles, K);
  else z4c_derivs_split_kernel<4, KT><<<grid, kDerivCols, 0, s>>>(Y, scratch, fs, sy, sz, tiles, ntiles, K);
}

}  // namespace

cudaError_t launch_z4c_dxy(const double* Y, double* scratch, long fs, int sy, const RowSeg* segs, int nsegs,
                           cudaStream_t s, int order, bool op_class) {
  if (nsegs == 0) return cudaSuccess;
  const int grid = nsegs < caps().dxy ? nsegs : caps().dxy;
  if (op_class) launch_dxy(Y, scratch, fs, sy, segs, nsegs, grid, s, order, PlainK{});
  else launch_dxy(Y, scratch, fs, sy, segs, nsegs, grid, s, order, FmaK{1.0, -1.0, -0.0});
  return cudaGetLastError();
}

cudaError_t launch_z4c_derivs_split(const double* Y, double* scratch, long fs, int sy, int sz, const Tile* tiles,
                                    int ntiles, cudaStream_t s, int order, bool op_class) {
  if (ntiles == 0) return cudaSuccess;
  const long items = (long)ntiles * kNZ4c;
  const int cap = caps().derivs[order == 8];
  const int grid = items < cap ? (int)items : cap;
  if (op_class) launch_derivs(Y, scratch, fs, sy, sz, tiles, ntiles, grid, s, order, PlainK{});
  else launch_derivs(Y, scratch, fs, sy, sz, tiles, ntiles, grid, s, order, FmaK{1.0, -1.0, -0.0});
  return cudaGetLastError();
}

namespace {

template <int BPS>
void launch_stage_bps(const StageArgs& a, const double* scratch, const Z4cParams& p, const CellRun* runs, int nruns,
                      int grid, cudaStream_t s, const FmaK& K, bool op_class) {
  const Z4cUnits c = z4c_units(a.order, a.h);
  if (op_class)
    z4c_stage_kernel<kStageSingle, BPS, PlainK><<<grid, kRunCells, 0, s>>>(a, scratch, p, runs, nruns, c, PlainK{});
  else if (a.form == kStageRk4) z4c_stage_kernel<kStageRk4, BPS><<<grid, kRunCells, 0, s>>>(a, scratch, p, runs, nruns, c, K);
  else if (a.form == kStageTwo) z4c_stage_kernel<kStageTwo, BPS><<<grid, kRunCells, 0, s>>>(a, scratch, p, runs, nruns, c, K);
  else if (a.form == kStageNone)
    z4c_stage_kernel<kStageNone, BPS><<<grid, kRunCells, 0, s>>>(a, scratch, p, runs, nruns, c, K);
  else z4c_stage_kernel<kStageSingle, BPS><<<grid, kRunCells, 0, s>>>(a, scratch, p, runs, nruns, c, K);
}

}  // namespace

cudaError_t launch_z4c_stage(const StageArgs& a, const double* scratch, const Z4cParams& p, const CellRun* runs,
                             int nruns, cudaStream_t s, int bps, bool op_class) {
  if (nruns == 0) return cudaSuccess;
  if (bps != 2 && bps != 3) return cudaErrorInvalidValue;
  if (op_class && a.form != kStageSingle) return cudaErrorInvalidValue;
  // persistent grid: the resident blocks
  const int grid = nruns < caps().stage[bps] ? nruns : caps().stage[bps];
  const FmaK K{1.0, -1.0, -0.0};
  if (bps == 2) launch_stage_bps<2>(a, scratch, p, runs, nruns, grid, s, K, op_class);
  else launch_stage_bps<3>(a, scratch, p, runs, nruns, grid, s, K, op_class);
  return cudaGetLastError();
}

cudaError_t launch_z4c_constraints(const double* Y, const double* scratch, double* out, long fs, int sy, int sz,
                                   int order, double h, long out_stride, const int* box_lo, const int* box_n,
                                   cudaStream_t s) {
  const long blocks = ((long)box_n[0] * box_n[1] * box_n[2] + kRunCells - 1) / kRunCells;
  const int grid = (int)(blocks < sm_count() * 16L ? blocks : sm_count() * 16L);
  z4c_constraints_kernel<<<grid, kRunCells, 0, s>>>(Y, scratch, out, fs, sy, sz, z4c_units(order, h), out_stride,
                                                    box_lo[0], box_lo[1], box_lo[2], box_n[0], box_n[1], box_n[2],
                                                    FmaK{1.0, -1.0, -0.0});
  return cudaGetLastError();
}

}  // namespace sc
