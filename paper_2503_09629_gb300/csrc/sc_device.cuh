// sc_device.cuh -- bodies of the refinement-boundary, ghost-copy and wave
// stage kernels as device functions over an explicit worker range.
//
// Each body distributes its work over `nb` workers (thread blocks) of which
// this block is number `bid`, with the block's threads as lanes.  The
// stand-alone kernels call them with (blockIdx.x, gridDim.x); the persistent
// coarse-step kernel calls the same functions, phase after phase, with its
// own block range, so both forms execute identical arithmetic per value.
#pragma once

#include "sc_fixed.cuh"

namespace sc {

// Prolongation sums.  Values are v * 2^e with |v| < 2^60.2 (59 bits at a node,
// grown by less than 1.3 per axis: the weights' magnitudes sum to 10568 / 8192).
// A position's six nodes are aligned to their largest exponent and the weights are
// integers over 2^13, so a sum is exact to the last place of that alignment (2^-58
// of the largest node, rounded down; three axes: 2^-54 of the largest of 216 nodes at
// most) and depends on the six values alone.  Nodes that hold an infinity, a NaN or a value
// near the ends of the exponent range carry kNodeFp64, which spreads to every
// sum they enter; such a position is computed in FP64.
constexpr int kNodeFp64 = 0x7fff;
__device__ __forceinline__ void prolong_node(double d, long long* v, int* e) {
  const long long bits = __double_as_longlong(d), s = bits >> 63;
  const int t = (int)(bits >> 52) & 0x7ff;
  const long long m = (bits & 0xfffffffffffffll) | 0x10000000000000ll;
  const bool zero = (bits << 1) == 0;
  *v = zero ? 0 : ((m << 6) ^ s) - s;
  *e = zero || (unsigned)(t - 120) <= 1880u ? t : kNodeFp64;
}
__device__ __forceinline__ long long prolong_align(long long v, int n) {
  long long r;
  asm("shr.s64 %0, %1, %2;" : "=l"(r) : "l"(v), "r"(n));
  return r;
}
// weight * 2^13 of node m for parity 0 (-1/4 from cell c, nodes c-3..c+2); parity 1 mirrored
__device__ __forceinline__ constexpr int prolong_weight(int m) {
  constexpr int w[6] = {63, -495, 2310, 6930, -693, 77};
  return w[m];
}
__device__ __forceinline__ void prolong_one(const long long* v, const int* e, int parity, long long* r, int* E) {
  int em = 0;
#pragma unroll
  for (int m = 0; m < 6; ++m) em = max(em, e[m]);
  FxWide a;
#pragma unroll
  for (int m = 0; m < 6; ++m)
    a.add(parity ? prolong_weight(5 - m) : prolong_weight(m), prolong_align(v[m], em - e[m]));
  *r = a.get<13>();
  *E = em;
}
// One value in FP64 chains: x sums over six nodes from zero, then y sums of those, then z sums.
static __device__ __noinline__ double prolong_fp64(const double* p, long psy, long psz, const double* wx, const double* wy,
                                            const double* wz) {
  double sz = 0.0;
#pragma unroll 1
  for (int kz = 0; kz < kPN; ++kz) {
    double sy = 0.0;
#pragma unroll 1
    for (int ky = 0; ky < kPN; ++ky) {
      const double* row = p + (long)kz * psz + (long)ky * psy;
      double sx = 0.0;
#pragma unroll
      for (int kx = 0; kx < kPN; ++kx) sx = fma(wx[kx], row[kx], sx);
      sy = fma(wy[ky], sx, sy);
    }
    sz = fma(wz[kz], sy, sz);
  }
  return sz;
}

// Sec. II step 2, per-cell form: tensor-product quintic Lagrange prolongation
// of y_n and the stage vectors the dense output reads (the first nvec of yn,
// k1..k4) from 6x6x6 parent cells to refinement-boundary ghost cells
// [first, ncells); results go to store[(v * F + f) * ncells + cell].  The sums of
// the tile form below, so both give identical results.
__device__ __forceinline__ void amr_prolong_cells_body(const double* __restrict__ yn, const double* __restrict__ k1,
                                                       const double* __restrict__ k2, const double* __restrict__ k3,
                                                       const double* __restrict__ k4, long pfs, int psy, int psz,
                                                       const AmrCell* __restrict__ cells, int first, int ncells,
                                                       double* __restrict__ store, int F, const Weights& w, int nvec,
                                                       int bid, int nb) {
  const int nc = ncells - first;
  const long total = (long)nc * F;
  for (long idx = bid * (long)blockDim.x + threadIdx.x; idx < total; idx += (long)nb * blockDim.x) {
    const int a = first + (int)(idx % nc);
    const int f = (int)(idx / nc);
    const AmrCell c = cells[a];
    const int px = c.parity & 1, py = (c.parity >> 1) & 1, pz = (c.parity >> 2) & 1;
    const double* src[5] = {yn, k1, k2, k3, k4};
#pragma unroll 1
    for (int v = 0; v < nvec; ++v) {
      const double* p = src[v] + (long)f * pfs + c.pbase;
      long long z[kPN], y[kPN], x[kPN], r;
      int ez[kPN], ey[kPN], ex[kPN], e;
#pragma unroll
      for (int kz = 0; kz < kPN; ++kz) {
#pragma unroll
        for (int ky = 0; ky < kPN; ++ky) {
          const double* row = p + (long)kz * psz + (long)ky * psy;
#pragma unroll
          for (int kx = 0; kx < kPN; ++kx) prolong_node(__ldg(row + kx), &x[kx], &ex[kx]);
          prolong_one(x, ex, px, &y[ky], &ey[ky]);
        }
        prolong_one(y, ey, py, &z[kz], &ez[kz]);
      }
      prolong_one(z, ez, pz, &r, &e);
      store[((long)v * F + f) * ncells + a] =
          e == kNodeFp64 ? prolong_fp64(p, psy, psz, w.prolong[px], w.prolong[py], w.prolong[pz]) : fx_back<6, 0>(r, e << 20);
    }
  }
}

// Offset of the first stencil node of fine position i along one axis from
// the first node of a tile's parent region, for a tile whose first fine
// position has parity p0 (parity 0: the fine centre sits at -1/4 parent cell
// and uses nodes c-3..c+2; parity 1: +1/4 and c-2..c+3).
__device__ __forceinline__ int tile_node_offset(int p0, int i) { return ((p0 + i) >> 1) + ((p0 + i) & 1) - p0; }

// Shared memory (in doubles) the tile-separable prolongation needs per group of
// 128 threads: the parent region (at most 10 x 10 x 8 nodes), the x sums (at
// most 8 x 10 x 8) and the y sums (at most 8 x 8 x 8), and an exponent of two
// bytes for each of them.
constexpr int kTileRegion = 800, kTileXSums = 640, kTileYSums = 512;
constexpr int kTileValues = kTileRegion + kTileXSums + kTileYSums;
constexpr int kProlongSmemPerGroup = kTileValues + kTileValues / 4;

// The two fine positions of parent cell c of a line (parities 0 and 1, at -1/4
// and +1/4) from the seven nodes their stencils cover: nodes n0..n0 + 6 of the
// line's N (those outside it belong to a position that the tile does not have).
// Each position has its own alignment (prolong_one), so that its value does not
// depend on the tile it is in.
__device__ __forceinline__ void prolong_pair(const long long* __restrict__ v, const short* __restrict__ ve, int n0,
                                             int N, int stride, long long* lo, long long* hi, int* elo, int* ehi) {
  long long x[7];
  int e[7], mid = 0;
#pragma unroll
  for (int m = 0; m < 7; ++m) {
    // (n0 is at least -1 and n0 + 5 at most N - 1)
    const int n = (m == 0 ? max(n0, 0) : m == 6 ? min(n0 + 6, N - 1) : n0 + m) * stride;
    x[m] = v[n];
    e[m] = ve[n];
    if (m > 0 && m < 6) mid = max(mid, e[m]);
  }
  const int E0 = max(e[0], mid), E1 = max(mid, e[6]);
  FxWide a, b;
  a.add(prolong_weight(0), prolong_align(x[0], E0 - e[0]));
  b.add(prolong_weight(0), prolong_align(x[6], E1 - e[6]));
  long long y[5];
#pragma unroll
  for (int m = 1; m < 6; ++m) {
    y[m - 1] = prolong_align(x[m], E0 - e[m]);
    a.add(prolong_weight(m), y[m - 1]);
  }
  if (E0 != E1) {
#pragma unroll
    for (int m = 1; m < 6; ++m) y[m - 1] = prolong_align(x[m], E1 - e[m]);
  }
#pragma unroll
  for (int m = 1; m < 6; ++m) b.add(prolong_weight(6 - m), y[m - 1]);
  *lo = a.get<13>();
  *hi = b.get<13>();
  *elo = E0;
  *ehi = E1;
}
// q / d by a multiplication, exact for q (d - 1) < 65536.
struct SmallDiv {
  unsigned m;
  __device__ __forceinline__ explicit SmallDiv(int d) : m((65535u + (unsigned)d) / (unsigned)d) {}
  __device__ __forceinline__ int operator()(int q) const { return (int)((unsigned)q * m >> 16); }
};
// A tile's lines along one axis: lines * pairs work items (at most 500), line l's
// nodes at lay(l, &dst) + n * stride, its fine positions written by out(dst, i, v, e).
template <class LAY, class OUT>
__device__ __forceinline__ void prolong_axis(const long long* v, const short* ve, int t, int lines, int p0, int ext,
                                             int N, int stride, const LAY& lay, const OUT& out) {
  const int items = lines * (((p0 + ext - 1) >> 1) + 1);
  const SmallDiv by_lines(lines);
  for (int q = t; q < items; q += 128) {
    const int c = by_lines(q), l = q - c * lines, i = 2 * c - p0;
    int dst;
    const int b = lay(l, &dst);
    long long lo, hi;
    int elo, ehi;
    prolong_pair(v + b, ve + b, c - p0, N, stride, &lo, &hi, &elo, &ehi);
    if (i >= 0) out(dst, i, lo, elo);
    if (i + 1 < ext) out(dst, i + 1, hi, ehi);
  }
}

// Separable form of the same interpolation for the slab tiles of a ghost
// shell: one group of 128 threads per (tile, vector, field) stages the
// tile's parent region in shared memory and interpolates along x, then y,
// then z.  Along the thin axis of a slab tile (the ghost width) the sums shrink
// 7-8 nodes to 3-4 values, so a ghost value costs 20-40 multiplications instead
// of the 216 + 42 of the per-cell form.  The sums are integers (prolong_pair), two
// fine positions of a parent cell at a time: in FP64 chains the kernel was bound
// by that pipe, 82% of its rate.  Now integer issue: 684,504 ghost cells of two
// fields and five vectors, 0.443 ms in FP64, 0.343 with run-time divisions for the
// work items' places, 0.281 so; 46,872 ghost cells 0.054, 0.039, 0.033.
// ngrp groups of 128 threads (threads beyond them idle); sm: ngrp *
// kProlongSmemPerGroup doubles.  Every thread of the block must call this
// function (it synchronises the block).
__device__ __forceinline__ void amr_prolong_tiles_body(const double* __restrict__ yn, const double* __restrict__ k1,
                                                       const double* __restrict__ k2, const double* __restrict__ k3,
                                                       const double* __restrict__ k4, long pfs, int psy, int psz,
                                                       const AmrTile* __restrict__ tiles, int ntiles,
                                                       const int32_t* __restrict__ slots, int ncells,
                                                       double* __restrict__ store, int F, const Weights& w, int nvec,
                                                       int bid, int nb, double* sm, int ngrp) {
  const int grp = threadIdx.x >> 7, t = threadIdx.x & 127;
  long long* iR = reinterpret_cast<long long*>(sm + grp * kProlongSmemPerGroup);
  long long* iX = iR + kTileRegion;
  long long* iY = iX + kTileXSums;
  short* eR = reinterpret_cast<short*>(iR + kTileValues);
  short* eX = eR + kTileRegion;
  short* eY = eX + kTileXSums;
  const int combos = nvec * F;
  const int ngroups = (combos + ngrp - 1) / ngrp;
  const long items = (long)ntiles * ngroups;
  for (long item = bid; item < items; item += nb) {
    const int b = (int)(item / ngroups);
    const int combo = (int)(item % ngroups) * ngrp + grp;
    const bool active = grp < ngrp && combo < combos;
    const AmrTile T = tiles[b];
    const int ex = T.ext[0], ey = T.ext[1], ez = T.ext[2];
    const int px = T.par & 1, py = (T.par >> 1) & 1, pz = (T.par >> 2) & 1;
    const int Nx = tile_node_offset(px, ex - 1) + kPN, Ny = tile_node_offset(py, ey - 1) + kPN;
    const int Nz = tile_node_offset(pz, ez - 1) + kPN;
    const int v = active ? combo / F : 0, f = active ? combo % F : 0;
    const double* base = (v == 0 ? yn : v == 1 ? k1 : v == 2 ? k2 : v == 3 ? k3 : k4) + (long)f * pfs + T.pbase;
    const SmallDiv by_x(Nx), by_y(Ny), by_e(ex);
    if (active)
      for (int q = t; q < Nx * Ny * Nz; q += 128) {
        const int r = by_x(q), x = q - r * Nx, z = by_y(r);
        int e;
        prolong_node(__ldg(base + (long)z * psz + (long)(r - z * Ny) * psy + x), iR + q, &e);  // [z][y][x]
        eR[q] = (short)e;
      }
    __syncthreads();
    if (active)
      prolong_axis(iR, eR, t, Ny * Nz, px, ex, Nx, 1,
                   [&](int l, int* dst) {
                     *dst = l * ex;  // [z][y][i]
                     return l * Nx;
                   },
                   [&](int dst, int i, long long x, int e) {
                     iX[dst + i] = x;
                     eX[dst + i] = (short)e;
                   });
    __syncthreads();
    if (active)
      prolong_axis(iX, eX, t, ex * Nz, py, ey, Ny, ex,
                   [&](int l, int* dst) {
                     const int z = by_e(l), i = l - z * ex;
                     *dst = z * ey * ex + i;  // [z][j][i]
                     return z * Ny * ex + i;
                   },
                   [&](int dst, int j, long long x, int e) {
                     iY[dst + j * ex] = x;
                     eY[dst + j * ex] = (short)e;
                   });
    __syncthreads();
    if (active)
      prolong_axis(iY, eY, t, ex * ey, pz, ez, Nz, ex * ey,
                   [&](int l, int* dst) {
                     *dst = l;
                     return l;
                   },
                   [&](int dst, int k, long long x, int e) {
                     const int slot = slots[T.slot_base + k * ex * ey + dst];
                     if (slot < 0) return;
                     double d;
                     if (e == kNodeFp64) {
                       const int j = by_e(dst), i = dst - j * ex;
                       d = prolong_fp64(base + (long)tile_node_offset(pz, k) * psz +
                                            (long)tile_node_offset(py, j) * psy + tile_node_offset(px, i),
                                        psy, psz, w.prolong[(px + i) & 1], w.prolong[(py + j) & 1],
                                        w.prolong[(pz + k) & 1]);
                     } else {
                       d = fx_back<6, 0>(x, e << 20);
                     }
                     store[((long)v * F + f) * ncells + slot] = d;
                   });
    __syncthreads();
  }
}

// Sec. II steps 3/5: ghost value = P[y_n] + sum_j c_j P[k_j] over the nk
// prolonged stage vectors in the store (4 for RK4, 3 for RK3, 2 for RK2, 0
// for a plain prolonged value); the coefficients encode dense output (Eqs.
// denseoutput1/2) and the Taylor stage formulas (Eqs. Y1-Y4) for one stage of
// one fine substep.
__device__ __forceinline__ void amr_apply_body(double* __restrict__ vec, long fs, int F,
                                               const AmrCell* __restrict__ cells, int ncells,
                                               const double* __restrict__ store, double c1, double c2, double c3,
                                               double c4, int nk, int bid, int nb) {
  const long total = (long)ncells * F;
  for (long idx = bid * (long)blockDim.x + threadIdx.x; idx < total; idx += (long)nb * blockDim.x) {
    const int a = (int)(idx % ncells);
    const int f = (int)(idx / ncells);
    const long n = ncells;
    const double* s = store + (long)f * n + a;
    const long vs = (long)F * n;
    double v = s[0];
    if (nk > 0) v = fma(c1, s[vs], v);
    if (nk > 1) v = fma(c2, s[2 * vs], v);
    if (nk > 2) v = fma(c3, s[3 * vs], v);
    if (nk > 3) v = fma(c4, s[4 * vs], v);
    vec[(long)f * fs + cells[a].dst] = v;
  }
}

// Periodic images: ghost cell <- the wrapped interior cell (pairs: x =
// destination offset, y = source offset).
__device__ __forceinline__ void periodic_copy_body(double* __restrict__ vec, long fs, int F,
                                                   const int2* __restrict__ pairs, int npairs, int bid, int nb) {
  const long total = (long)npairs * F;
  for (long idx = bid * (long)blockDim.x + threadIdx.x; idx < total; idx += (long)nb * blockDim.x) {
    const int a = (int)(idx % npairs);
    const int f = (int)(idx / npairs);
    const int2 p = pairs[a];
    vec[(long)f * fs + p.x] = vec[(long)f * fs + p.y];
  }
}

// Sec. II step 7, per-cell form: every parent cell whose eight children are
// fine interior cells takes the tensor-product quintic interpolant of the
// 6x6x6 fine cells centred on it.
__device__ __forceinline__ void restrict_cells_body(double* __restrict__ parent, long pfs,
                                                    const double* __restrict__ fine, long ffs, int fsy, int fsz,
                                                    const RestrictCell* __restrict__ cells, int ncells, int F,
                                                    const Weights& w, int bid, int nb) {
  const long total = (long)ncells * F;
  for (long idx = bid * (long)blockDim.x + threadIdx.x; idx < total; idx += (long)nb * blockDim.x) {
    const int a = (int)(idx % ncells);
    const int f = (int)(idx / ncells);
    const RestrictCell c = cells[a];
    const double* p = fine + (long)f * ffs + c.fbase;
    double sz = 0.0;
#pragma unroll
    for (int kz = 0; kz < kRN; ++kz) {
      double sy = 0.0;
#pragma unroll
      for (int ky = 0; ky < kRN; ++ky) {
        const double* row = p + (long)kz * fsz + (long)ky * fsy;
        double sx = 0.0;
#pragma unroll
        for (int kx = 0; kx < kRN; ++kx) sx = fma(w.restrict_w[kx], __ldg(row + kx), sx);
        sy = fma(w.restrict_w[ky], sx, sy);
      }
      sz = fma(w.restrict_w[kz], sy, sz);
    }
    parent[(long)f * pfs + c.dst] = sz;
  }
}

// Shared-memory doubles the block-separable restriction needs per group.
constexpr int kRestrictSmemPerGroup = 1728 + 576 + 192;

// Separable form of the same restriction for 4x4x4 parent blocks: one group
// of 64 threads per (block, field) stages the 12x12x12 fine region in shared
// memory and sums along x, then y, then z (78 FMAs per parent cell instead of
// 216).  Each parent value is the same chain of fused multiply-adds as in the
// per-cell form (x sums, then y, then z, each from zero in stencil order), so
// both give identical results.  ngrp groups of 64 threads (threads beyond
// them idle); sm: ngrp * kRestrictSmemPerGroup doubles.  Every thread of the
// block must call this function (it synchronises the block).
__device__ __forceinline__ void restrict_blocks_body(double* __restrict__ parent, long pfs, int psy, int psz,
                                                     const double* __restrict__ fine, long ffs, int fsy, int fsz,
                                                     const RestrictBlock* __restrict__ blocks, int nblocks, int F,
                                                     const Weights& w, int bid, int nb, double* sm, int ngrp) {
  const int grp = threadIdx.x >> 6, t = threadIdx.x & 63;
  double* sF = sm + grp * 1728;
  double* sX = sm + ngrp * 1728 + grp * 576;
  double* sY = sm + ngrp * 2304 + grp * 192;
  const long items = (long)nblocks * F;
  const long chunks = (items + ngrp - 1) / ngrp;
  for (long it = bid; it < chunks; it += nb) {
    const long item = it * ngrp + grp;
    const bool active = grp < ngrp && item < items;
    const int b = active ? (int)(item / F) : 0, f = active ? (int)(item % F) : 0;
    const RestrictBlock B = blocks[b];
    if (active) {
      const double* src = fine + (long)f * ffs + B.fbase;
      for (int q = t; q < 1728; q += 64) {
        const int z = q / 144, y = (q / 12) % 12, x = q % 12;
        sF[q] = __ldg(src + (long)z * fsz + (long)y * fsy + x);
      }
    }
    __syncthreads();
    if (active) {  // x: row (z, y) of the fine region, parent px
      for (int q = t; q < 576; q += 64) {
        const int z = q / 48, y = (q / 4) % 12, px = q % 4;
        const double* row = &sF[(z * 12 + y) * 12 + 2 * px];
        double sx = 0.0;
#pragma unroll
        for (int m = 0; m < kRN; ++m) sx = fma(w.restrict_w[m], row[m], sx);
        sX[q] = sx;  // [z][y][px]
      }
    }
    __syncthreads();
    if (active) {  // y: fine z, parent (py, px)
      for (int q = t; q < 192; q += 64) {
        const int z = q / 16, py = (q / 4) % 4, px = q % 4;
        double sy = 0.0;
#pragma unroll
        for (int m = 0; m < kRN; ++m) sy = fma(w.restrict_w[m], sX[(z * 12 + 2 * py + m) * 4 + px], sy);
        sY[q] = sy;  // [z][py][px]
      }
    }
    __syncthreads();
    if (active && ((B.mask >> t) & 1ull)) {  // z: parent cell t = px + 4 py + 16 pz
      const int pz = t >> 4, py = (t >> 2) & 3, px = t & 3;
      double sz = 0.0;
#pragma unroll
      for (int m = 0; m < kRN; ++m) sz = fma(w.restrict_w[m], sY[((2 * pz + m) * 4 + py) * 4 + px], sz);
      parent[(long)f * pfs + B.pbase + (long)pz * psz + (long)py * psy + px] = sz;
    }
    __syncthreads();
  }
}

// The halo cells of a plane of a tile that a thread brings into shared memory,
// W columns and rows wide on each side without the corners: the shared-memory
// place (rows of nx + 2 W; -1: none) and the offset from the tile's first cell.
template <int W>
__device__ __forceinline__ void halo_cell(const Tile& T, int h, long sy, int* place, long* off) {
  *place = -1;
  *off = 0;
  if (h >= 2 * W * (T.nx + T.ny)) return;
  int x, y;
  if (h < 2 * W * T.ny) {
    y = h / (2 * W);
    x = h - y * (2 * W);
    x = x < W ? x - W : T.nx + x - W;
  } else {
    h -= 2 * W * T.ny;
    y = h / T.nx;
    x = h - y * T.nx;
    y = y < W ? y - W : T.ny + y - W;
  }
  *place = (y + W) * (T.nx + 2 * W) + x + W;
  *off = (long)y * sy + x;
}
// Values of a plane with its halo (tiles of at most kDerivCols columns, 32 wide, 32 high).
__host__ __device__ constexpr int plane_values(int W) { return (32 + 2 * W) * (8 + 2 * W); }

// Scalar-wave stage (Sec. IV.A): k_i = f(Y_i) with the centred Laplacian (4th
// or 8th order), then the stage update of StageArgs (Eqs. rk2-rk5 for RK4,
// the last-stage combinations of RK3/RK2, or k only).  One tile per worker at a
// time, a thread per column: it walks z with the packed values of u at z-R..z+R
// in registers and shares the plane's through shared memory (planes: 2 *
// plane_values(R)), so a value is unpacked once or twice instead of 13 (25)
// times; the Laplacian is summed in aligned integers (sc_fixed.cuh), or in FP64
// where the values do not allow that.  256 threads; every thread of the block must
// call this function (it synchronises the block).
template <int ORD>
__device__ __forceinline__ void wave_stage_body(const StageArgs& a, const Tile* __restrict__ tiles, int ntiles,
                                                const FmaK& K, int bid, int nb, long long* planes) {
  using F = FxSums<ORD>;
  constexpr int R = ORD / 2, NW = 2 * R + 1;
  const long sy = a.sy, sz = a.sz;
  int buf = 0;
  for (int t = bid; t < ntiles; t += nb) {
    const Tile T = tiles[t];
    const int pitch = T.nx + 2 * R;
    const bool active = (int)threadIdx.x < T.nx * T.ny;
    const int j = threadIdx.x / T.nx, i = threadIdx.x - j * T.nx, own = (j + R) * pitch + i + R;
    const long o0 = (long)T.z0 * sz + (long)T.y0 * sy + T.x0;
    int hs[2];
    long ho[2];
    double hv[2];
    halo_cell<R>(T, threadIdx.x, sy, &hs[0], &ho[0]);
    halo_cell<R>(T, threadIdx.x + kDerivCols, sy, &hs[1], &ho[1]);
#pragma unroll
    for (int r = 0; r < 2; ++r) hv[r] = hs[r] >= 0 ? a.Y[o0 + ho[r]] : 0.0;
    const double* u = a.Y + o0 + (long)j * sy + i;
    long long w[NW];
    double un = 0.0;
    if (active) {
#pragma unroll
      for (int m = 0; m < NW - 1; ++m) w[m] = fx_pack(u[(m - R) * sz]);
      un = u[R * sz];
    }
#pragma unroll 1
    for (int k = 0; k < T.nz; ++k, buf ^= 1) {
      long long* pl = planes + buf * plane_values(R);
      const bool more = k + 1 < T.nz;
      const long o = o0 + k * sz + (long)j * sy + i;
      double ku = 0.0, yu = 0.0, yp = 0.0, k1u = 0.0, k1p = 0.0, k2u = 0.0, k2p = 0.0, k3u = 0.0, k3p = 0.0;
      if (active) {
        pl[own] = w[R];
        ku = a.Y[a.fs + o];  // d_t u = Pi
        if (a.form != kStageNone) {
          yu = a.yn[o];
          yp = a.yn[a.fs + o];
        }
        if (a.form == kStageRk4 || a.form == kStageTwo) {
          k1u = a.k1[o];
          k1p = a.k1[a.fs + o];
        }
        if (a.form == kStageRk4) {
          k2u = a.k2[o];
          k2p = a.k2[a.fs + o];
          k3u = a.k3[o];
          k3p = a.k3[a.fs + o];
        }
        w[NW - 1] = fx_pack(un);
        if (more) un = u[(k + 1 + R) * sz];
      }
#pragma unroll
      for (int r = 0; r < 2; ++r)
        if (hs[r] >= 0) {
          pl[hs[r]] = fx_pack(hv[r]);
          if (more) hv[r] = a.Y[o0 + ho[r] + (k + 1) * sz];
        }
      // (the planes alternate, also from one tile to the next: a plane is written
      // again only after every thread has passed the next barrier)
      __syncthreads();
      if (!active) continue;
      long long v[R][6];
      int Ei = fx_pexp(w[R]), E = 0;
#pragma unroll
      for (int m = 0; m < R; ++m) {
        v[m][0] = pl[own - (m + 1)];
        v[m][1] = pl[own + (m + 1)];
        v[m][2] = pl[own - (m + 1) * pitch];
        v[m][3] = pl[own + (m + 1) * pitch];
        v[m][4] = w[R - (m + 1)];
        v[m][5] = w[R + (m + 1)];
#pragma unroll
        for (int q = 0; q < 6; ++q) {
          if (m == 0) Ei = max(Ei, fx_pexp(v[m][q]));
          else E = max(E, fx_pexp(v[m][q]));
        }
      }
      E = max(E, Ei);
      double lap;
      if (packed_ok(E) && E - Ei <= F::kLaplacianExcess) {
        lap = F::laplacian(v, w[R], E);
      } else {
        const double* c = u + k * sz;
        double p[R][6];
        unsigned any = zero_bits(c[0]);
#pragma unroll
        for (int m = 1; m <= R; ++m) {
          const double q[6] = {c[-m], c[m], c[-m * sy], c[m * sy], c[-m * sz], c[m * sz]};
#pragma unroll
          for (int n = 0; n < 6; ++n) {
            p[m - 1][n] = q[n];
            any |= zero_bits(q[n]);
          }
        }
        lap = 0.0;
        if (any) {
          double s[4];
#pragma unroll
          for (int m = 0; m < R; ++m) s[m] = ((p[m][0] + p[m][1]) + (p[m][2] + p[m][3])) + (p[m][4] + p[m][5]);
          if (ORD == 4) lap = fma(-90.0, c[0], fma(16.0, s[0], -s[1]));
          else lap = fma(-43050.0, c[0], fma(8064.0, s[0], fma(-1008.0, s[1], fma(128.0, s[2], -9.0 * s[3]))));
        }
      }
      const double kp = fmul(lap, a.lap, K);  // d_t Pi = Laplacian u, its sum over 12 h^2 or 5040 h^2
      a.k[o] = ku;
      a.k[a.fs + o] = kp;
      if (a.form == kStageSingle) {
        a.out[o] = fma(a.cdt, ku, yu);
        a.out[a.fs + o] = fma(a.cdt, kp, yp);
      } else if (a.form == kStageRk4) {
        const double su = fadd(fma(2.0, k3u, fma(2.0, k2u, k1u)), ku, K);
        const double sp = fadd(fma(2.0, k3p, fma(2.0, k2p, k1p)), kp, K);
        a.out[o] = fma(a.cdt, su, yu);
        a.out[a.fs + o] = fma(a.cdt, sp, yp);
      } else if (a.form == kStageTwo) {
        a.out[o] = fma(a.cdt, ku, fma(a.c1dt, k1u, yu));
        a.out[a.fs + o] = fma(a.cdt, kp, fma(a.c1dt, k1p, yp));
      }
#pragma unroll
      for (int m = 0; m < NW - 1; ++m) w[m] = w[m + 1];
    }
  }
}

// Outgoing radiative condition on the outer ghost shell of a radiative
// level 0 (the boundary cells are evolved with their own right-hand side):
//   d_t u = -(x^i / r) d_i u - (u - u_inf) / r
// with 2nd-order differences, centred where both neighbours exist in the
// array and one-sided inwards on its outermost layer; u_inf = 1 for W,
// alpha and the diagonal of gt, 0 otherwise.
__device__ __forceinline__ void radiative_stage_body(const StageArgs& a, const int32_t* __restrict__ cells,
                                                     int ncells, int F, const Geom& g, int system, int bid, int nb) {
  const double inv2h = 1.0 / (2.0 * a.h);
  const long str[3] = {1, (long)a.sy, (long)a.sz};
  const long total = (long)ncells * F;
  for (long idx = bid * (long)blockDim.x + threadIdx.x; idx < total; idx += (long)nb * blockDim.x) {
    const int c = (int)(idx % ncells);
    const int f = (int)(idx / ncells);
    const long o = cells[c];
    const int ijk[3] = {(int)(o % g.pitch), (int)((o / g.pitch) % g.ext[1]), (int)(o / ((long)g.pitch * g.ext[1]))};
    double x[3];
    for (int d = 0; d < 3; ++d) x[d] = g.x0[d] + ijk[d] * g.h;
    const double r2 = x[0] * x[0] + x[1] * x[1] + x[2] * x[2];
    const double ir = rsqrt(r2);
    const double* p = a.Y + (long)f * a.fs;
    double adv = 0.0;
    for (int d = 0; d < 3; ++d) {
      const long s = str[d];
      double der;
      if (ijk[d] == 0) der = (-3.0 * p[o] + 4.0 * p[o + s] - p[o + 2 * s]) * inv2h;
      else if (ijk[d] == g.ext[d] - 1) der = (3.0 * p[o] - 4.0 * p[o - s] + p[o - 2 * s]) * inv2h;
      else der = (p[o + s] - p[o - s]) * inv2h;
      adv = fma(x[d], der, adv);
    }
    double uinf = 0.0;
    if (system == SC_Z4C && (f == ZW || f == ZAL || f == ZG + 0 || f == ZG + 3 || f == ZG + 5)) uinf = 1.0;
    const double kv = -(adv + (p[o] - uinf)) * ir;
    const long fo = (long)f * a.fs + o;
    a.k[fo] = kv;
    if (a.form == kStageSingle) {
      a.out[fo] = fma(a.cdt, kv, a.yn[fo]);
    } else if (a.form == kStageRk4) {
      const double s = fma(2.0, a.k3[fo], fma(2.0, a.k2[fo], a.k1[fo])) + kv;
      a.out[fo] = fma(a.cdt, s, a.yn[fo]);
    } else if (a.form == kStageTwo) {
      a.out[fo] = fma(a.cdt, kv, fma(a.c1dt, a.k1[fo], a.yn[fo]));
    }
  }
}

// Non-finite scan of the interior tiles of one level array: sets bit
// kStatusNonFinite of *flag when any value is NaN or infinite.
__device__ __forceinline__ void nonfinite_body(const double* __restrict__ vec, long fs, int F,
                                               const Tile* __restrict__ tiles, int ntiles, int sy, int sz, int* flag,
                                               int bid, int nb) {
  for (int t = bid; t < ntiles; t += nb) {
    const Tile T = tiles[t];
    const int n = T.nx * T.ny * T.nz;
    for (int q = threadIdx.x; q < n * F; q += blockDim.x) {
      const int f = q / n, c = q % n;
      const int i = c % T.nx, j = (c / T.nx) % T.ny, k = c / (T.nx * T.ny);
      const double v = vec[(long)f * fs + (long)(T.z0 + k) * sz + (long)(T.y0 + j) * sy + T.x0 + i];
      if (!isfinite(v)) atomicOr(flag, kStatusNonFinite);
    }
  }
}

}  // namespace sc
