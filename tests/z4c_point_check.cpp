// The Z4c right-hand side and constraints at random cells: sc_z4c_point.cuh,
// compiled for the host, against the same equations written out in 113-bit
// arithmetic.  Usage: z4c_point_check KIND PARAM AMP; prints for every output its number
// and the RMS error over the RMS value (over 1 where that is zero) of the integer sums and of the FP64 form,
// then how many cells the integers refused.
//   stretch r: metric, and all tensors with it, stretched along x, g_xx : g_yy = r
//   offdiag e: off-diagonal components of gt, At, their derivatives and d_j beta^i times e
//   shift   e: y and z components of beta and their derivatives times e
//   plane   e: data that vary along x only, diagonal tensors but for yz components times e
//   second  v: one second derivative of size v
//   first   v: one first derivative of size v
// AMP: size of the derivatives.
#include <cuda_runtime.h>

#include <cstdio>
#include <cstdlib>
#include <cstring>
#include <random>
#include <vector>

#include "sc_z4c_point.cuh"

#ifdef __x86_64__
typedef __float128 Q;
#else
typedef long double Q;  // 113 bits on aarch64
#endif

struct HostK {};
static inline double fadd(double a, double b, const HostK&) { return a + b; }
static inline double fsub(double a, double b, const HostK&) { return a - b; }
static inline double fmul(double a, double b, const HostK&) { return a * b; }

using namespace sc;

// the sums in FP64 only, and as they are (counting the cells that the integers refuse)
static int g_refused;
template <bool FP64>
struct Form {
  template <bool CONS, int T, class KT>
  static void sums(const double* Y, const double* S, long fs, long o, const Z4cUnits& c, const double* gu,
                   const FxMem<T>& mem, const KT& K) {
    if (!FP64 && z4c_connection_fixed<CONS, T, KT>(Y, S, fs, o, c, gu, mem, K)) return;
    g_refused += !FP64;
    InverseMetric t;
    std::memcpy(t.gu, gu, sizeof(t.gu));
    z4c_connection_fp64<CONS, T, KT>(Y, S, fs, o, c, t, mem, K);
  }
};
struct Out {
  double* r;
  struct Pre {};
  Pre load(int) const { return Pre(); }
  void operator()(int f, double v, Pre) const { r[f] = v; }
};

// the equations, index by index; out: 22 right-hand sides and 7 constraints
static void exact(const double* Y, const double* S, double h, const Z4cParams& P, double eta, Q* out) {
  const Q w = 12 * (Q)h;
  Q u[22], d[22][3], dd[11][3][3], g[3][3], gu[3][3], A[3][3], dg[3][3][3], ddg[3][3][3][3];
  for (int f = 0; f < 22; ++f) {
    u[f] = Y[f];
    for (int k = 0; k < 3; ++k) d[f][k] = (Q)S[Q_D1 + 3 * f + k] / w;
  }
  for (int s = 0; s < 11; ++s)
    for (int i = 0; i < 3; ++i)
      for (int j = 0; j < 3; ++j) dd[s][i][j] = (Q)S[Q_D2 + 6 * s + sidx(i, j)] / (i == j ? w * h : w * w);
  for (int i = 0; i < 3; ++i)
    for (int j = 0; j < 3; ++j) {
      g[i][j] = u[ZG + sidx(i, j)];
      A[i][j] = u[ZA + sidx(i, j)];
      for (int k = 0; k < 3; ++k) {
        dg[i][j][k] = d[ZG + sidx(i, j)][k];
        for (int l = 0; l < 3; ++l) ddg[i][j][k][l] = dd[1 + sidx(i, j)][k][l];
      }
    }
  Q det = 0;
  for (int i = 0; i < 3; ++i) {
    const int j = (i + 1) % 3, k = (i + 2) % 3;
    det += g[0][i] * (g[1][j] * g[2][k] - g[1][k] * g[2][j]);
  }
  for (int i = 0; i < 3; ++i)
    for (int j = 0; j < 3; ++j) {
      const int a = (i + 1) % 3, b = (i + 2) % 3, c = (j + 1) % 3, e = (j + 2) % 3;
      gu[j][i] = (g[a][c] * g[b][e] - g[a][e] * g[b][c]) / det;
    }
  const Q W = u[ZW], al = u[ZAL], Th = u[ZTH], Kh = u[ZK], Kt = Kh + 2 * Th;
  const Q *dW = d[ZW], *da = d[ZAL];
  Q Gl[3][3][3], Gu[3][3][3], Gd[3];
  for (int k = 0; k < 3; ++k)
    for (int i = 0; i < 3; ++i)
      for (int j = 0; j < 3; ++j) Gl[k][i][j] = (dg[j][k][i] + dg[i][k][j] - dg[i][j][k]) / 2;
  for (int k = 0; k < 3; ++k) {
    Gd[k] = 0;
    for (int i = 0; i < 3; ++i)
      for (int j = 0; j < 3; ++j) {
        Gu[k][i][j] = 0;
        for (int l = 0; l < 3; ++l) Gu[k][i][j] += gu[k][l] * Gl[l][i][j];
        Gd[k] += gu[i][j] * Gu[k][i][j];
      }
  }
  Q DDW[3][3], DDa[3][3], R[3][3], lapW = 0, WW = 0, Wa = 0;
  for (int i = 0; i < 3; ++i)
    for (int j = 0; j < 3; ++j) {
      WW += gu[i][j] * dW[i] * dW[j];
      Wa += gu[i][j] * dW[i] * da[j];
      DDW[i][j] = dd[0][i][j];
      for (int k = 0; k < 3; ++k) DDW[i][j] -= Gu[k][i][j] * dW[k];
      lapW += gu[i][j] * DDW[i][j];
    }
  Q trR = 0, trDDa = 0;
  for (int i = 0; i < 3; ++i)
    for (int j = 0; j < 3; ++j) {
      Q r = (DDW[i][j] + g[i][j] * lapW) / W - 2 * g[i][j] * WW / (W * W);
      for (int k = 0; k < 3; ++k) {
        r += (g[k][i] * d[ZGAM + k][j] + g[k][j] * d[ZGAM + k][i] + Gd[k] * (Gl[i][j][k] + Gl[j][i][k])) / 2;
        for (int l = 0; l < 3; ++l) {
          r -= gu[k][l] * ddg[i][j][k][l] / 2;
          for (int m = 0; m < 3; ++m)
            r += gu[l][m] * (Gu[k][l][i] * Gl[j][k][m] + Gu[k][l][j] * Gl[i][k][m] + Gu[k][i][m] * Gl[k][l][j]);
        }
      }
      R[i][j] = r;
      trR += gu[i][j] * r;
      DDa[i][j] = dd[7][i][j] + (dW[i] * da[j] + dW[j] * da[i] - g[i][j] * Wa) / W;
      for (int k = 0; k < 3; ++k) DDa[i][j] -= Gu[k][i][j] * da[k];
      trDDa += gu[i][j] * DDa[i][j];
    }
  Q Am[3][3], Auu[3][3], AA = 0, divb = 0;
  for (int i = 0; i < 3; ++i)
    for (int j = 0; j < 3; ++j) {
      Am[i][j] = 0;
      for (int k = 0; k < 3; ++k) Am[i][j] += gu[i][k] * A[k][j];
    }
  for (int i = 0; i < 3; ++i) {
    divb += d[ZB + i][i];
    for (int j = 0; j < 3; ++j) {
      Auu[i][j] = 0;
      for (int k = 0; k < 3; ++k) Auu[i][j] += Am[i][k] * gu[k][j];
      AA += A[i][j] * Auu[i][j];
    }
  }
  auto adv = [&](int f) { return u[ZB] * d[f][0] + u[ZB + 1] * d[f][1] + u[ZB + 2] * d[f][2]; };
  out[ZW] = W * (al * Kt - divb) / 3 + adv(ZW);
  for (int i = 0; i < 3; ++i)
    for (int j = i; j < 3; ++j) {
      const int s = sidx(i, j);
      Q lg = -2 * divb * g[i][j] / 3, la = -2 * divb * A[i][j] / 3, aa = 0;
      for (int k = 0; k < 3; ++k) {
        lg += g[k][i] * d[ZB + k][j] + g[k][j] * d[ZB + k][i];
        la += A[k][i] * d[ZB + k][j] + A[k][j] * d[ZB + k][i];
        aa += A[i][k] * Am[k][j];
      }
      const Q tf = al * R[i][j] - DDa[i][j] - g[i][j] * (al * trR - trDDa) / 3;
      out[ZG + s] = -2 * al * A[i][j] + lg + adv(ZG + s);
      out[ZA + s] = W * W * tf + al * (Kt * A[i][j] - 2 * aa) + la + adv(ZA + s);
    }
  out[ZK] = -W * W * trDDa + al * (AA + Kt * Kt / 3) + al * P.kappa1 * (1 - (Q)P.kappa2) * Th + adv(ZK);
  out[ZTH] = al * (W * W * trR - AA + 2 * Kt * Kt / 3) / 2 - al * P.kappa1 * (2 + (Q)P.kappa2) * Th + adv(ZTH);
  out[ZAL] = -2 * al * Kh + adv(ZAL);
  Q M[3];
  for (int i = 0; i < 3; ++i) {
    Q r = adv(ZGAM + i) + 2 * Gd[i] * divb / 3 - 2 * (Q)P.kappa1 * al * (u[ZGAM + i] - Gd[i]);
    M[i] = 0;
    for (int j = 0; j < 3; ++j) {
      r += -2 * Auu[i][j] * da[j] - 6 * al * Auu[i][j] * dW[j] / W - Gd[j] * d[ZB + i][j];
      r -= 2 * al * gu[i][j] * (2 * d[ZK][j] + d[ZTH][j]) / 3;
      M[i] -= 3 * Auu[i][j] * dW[j] / W + 2 * gu[i][j] * (d[ZK][j] + 2 * d[ZTH][j]) / 3;
      for (int k = 0; k < 3; ++k) {
        r += 2 * al * Gu[i][j][k] * Auu[j][k] + gu[j][k] * dd[8 + i][j][k] + gu[i][j] * dd[8 + k][j][k] / 3;
        M[i] += Gu[i][j][k] * Auu[j][k];
        for (int l = 0; l < 3; ++l) {  // d_j At^ij
          M[i] += gu[i][k] * gu[j][l] * d[ZA + sidx(k, l)][j];
          for (int m = 0; m < 3; ++m)
            for (int n = 0; n < 3; ++n)
              M[i] -= (gu[i][m] * gu[k][n] * gu[j][l] + gu[i][k] * gu[j][m] * gu[l][n]) * dg[m][n][j] * A[k][l];
        }
      }
    }
    out[ZGAM + i] = r;
    out[ZB + i] = (Q)0.75 * u[ZGAM + i] - (Q)eta * u[ZB + i] + adv(ZB + i);
  }
  out[22] = W * W * trR + 2 * Kt * Kt / 3 - AA;
  for (int i = 0; i < 3; ++i) {
    out[23 + i] = M[i];
    out[26 + i] = u[ZGAM + i] - Gd[i];
  }
}

int main(int argc, char** argv) {
  if (argc < 4) return 2;
  const char* kind = argv[1];
  const double par = atof(argv[2]), amp = atof(argv[3]), h = 0.1;
  const bool plane = !strcmp(kind, "plane");
  double ax[3] = {1, 1, 1}, off = 1, ish = 1;
  if (!strcmp(kind, "stretch")) ax[0] = std::sqrt(par);
  if (!strcmp(kind, "offdiag")) off = par;
  if (!strcmp(kind, "shift")) ish = par;
  const int si[6] = {0, 0, 0, 1, 1, 2}, sj[6] = {0, 1, 2, 1, 2, 2};
  const double s1 = 1.0 / (12.0 * h), s2p = 1.0 / (12.0 * h * h), s2m = s1 * s1;  // of the stored sums
  const Z4cUnits units = z4c_units(4, h);
  const Z4cParams P{0.02, 0.0, 2.0, 0.3};
  std::mt19937_64 rng(5);
  auto U = [&] { return 2.0 * ((rng() >> 11) * 0x1p-53) - 1.0; };
  constexpr int N = 29;
  double val[N] = {}, err[2][N] = {};
  int differ = 0;
  for (int it = 0; it < 2000; ++it) {
    // size of a field: covariant indices grow with the axis, contravariant ones shrink
    auto size = [&](int f) {
      const int s = f >= ZG && f < ZG + 6 ? f - ZG : f >= ZA && f < ZA + 6 ? f - ZA : -1;
      if (plane && s >= 0) return si[s] == sj[s] ? 1.0 : s == 4 ? par : 0.0;
      if (plane && f >= ZGAM && f < ZAL + 4 && f != ZGAM && f != ZTH && f != ZAL && f != ZB) return 0.0;
      if (s >= 0) return ax[si[s]] * ax[sj[s]] * (si[s] == sj[s] ? 1.0 : off);
      if (f >= ZGAM && f < ZGAM + 3) return 1 / ax[f - ZGAM];
      if (f >= ZB && f < ZB + 3) return (f == ZB ? 1.0 : ish) / ax[f - ZB];
      return 1.0;
    };
    std::vector<double> Y(22), S(154);
    for (int f = 0; f < 22; ++f) {
      const bool one = f == ZW || f == ZAL || f == ZG || f == ZG + 3 || f == ZG + 5;
      Y[f] = size(f) * ((one ? 1.0 : 0.0) + 0.1 * U());
      for (int k = 0; k < 3; ++k) {
        const double e = plane && k > 0 ? 0.0 : f >= ZB && f < ZB + 3 && f - ZB != k ? off : 1.0;
        S[Q_D1 + 3 * f + k] = amp * size(f) * ax[k] * e * U() / s1;
      }
    }
    const int field[11] = {0, 1, 2, 3, 4, 5, 6, ZAL, ZB, ZB + 1, ZB + 2};
    for (int s = 0; s < 11; ++s)
      for (int p = 0; p < 6; ++p)
        S[Q_D2 + 6 * s + p] = plane && p > 0 ? 0.0
                                             : amp * size(field[s]) * ax[si[p]] * ax[sj[p]] * U() / (fx_pure(p) ? s2p : s2m);
    if (!strcmp(kind, "second")) S[Q_D2 + 6 * (it % 11) + (it / 11) % 6] = par;
    if (!strcmp(kind, "first")) S[Q_D1 + it % 66] = par;
    long long m[FM_SLOTS];
    short e[FM_SLOTS];
    const FxMem<1> mem{m, e};
    double got[2][N];
    z4c_rhs_point<Form<false>, 1>(Y.data(), S.data(), 1L, 0L, P, 2.0, units, mem, HostK(), Out{got[0]});
    z4c_rhs_point<Form<true>, 1>(Y.data(), S.data(), 1L, 0L, P, 2.0, units, mem, HostK(), Out{got[1]});
    z4c_constraints_point<Form<false>, 1>(Y.data(), S.data(), 1L, 0L, units, mem, HostK(), [&](int q, double v) { got[0][22 + q] = v; });
    z4c_constraints_point<Form<true>, 1>(Y.data(), S.data(), 1L, 0L, units, mem, HostK(), [&](int q, double v) { got[1][22 + q] = v; });
    Q ref[N];
    exact(Y.data(), S.data(), h, P, 2.0, ref);
    for (int f = 0; f < N; ++f) {
      differ += std::isfinite(got[0][f]) != std::isfinite(got[1][f]);
      val[f] += (double)(ref[f] * ref[f]);
      for (int q = 0; q < 2; ++q) {
        const Q d = got[q][f] - ref[f];
        err[q][f] += (double)(d * d);
      }
    }
  }
  for (int f = 0; f < N; ++f)
    printf("%d %.3e %.3e\n", f, std::sqrt(err[0][f] / (val[f] == 0 ? 1 : val[f])), std::sqrt(err[1][f] / (val[f] == 0 ? 1 : val[f])));
  printf("refused %d\nfiniteness differs %d\n", g_refused, differ);
  return 0;
}
