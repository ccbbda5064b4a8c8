// Host check of the integer-pipe Roe flux (csrc/fv_roe.h, the source the GPU
// kernels run) against the same flux in long double, beside an FP64 evaluation.
//   roe_check CASES
// prints, per regime and dimension: name, faces not taken, the largest error
// and the rms error of the integer flux and of the FP64 evaluation (units of
// 2^-53 of the magnitudes that the flux sums), then "refused N of M" for states
// that must be left to FP64.
#include <cmath>
#include <cstdint>
#include <cstdio>
#include <cstdlib>
#include <limits>
#include <random>

#include "../../paper_2306_14011_gb300/csrc/fv_roe.h"

// F(Q_up) + k alpha r of the upwind one-wave form; sc: the magnitudes summed.
template <class T, int NT>
static void reference(const double *QL, const double *QR, double gamma1, double efix, T *F, T *sc) {
  const int E = NT + 2;
  const T g1 = gamma1;
  const double *Q[2] = {QL, QR};
  T u[2][3], p[2], s[2], H[2];
  for (int i = 0; i < 2; ++i) {
    T k = 0;
    for (int c = 0; c <= NT; ++c) {
      u[i][c] = (T)Q[i][1 + c] / (T)Q[i][0];
      k += (T)Q[i][1 + c] * u[i][c];
    }
    p[i] = g1 * ((T)Q[i][E] - k / 2);
    s[i] = std::sqrt((T)Q[i][0]);
    H[i] = ((T)Q[i][E] + p[i]) / (T)Q[i][0];
  }
  T ut[3], q2 = 0;
  for (int c = 0; c <= NT; ++c) {
    ut[c] = (s[0] * u[0][c] + s[1] * u[1][c]) / (s[0] + s[1]);
    q2 += ut[c] * ut[c];
  }
  const T Ht = (s[0] * H[0] + s[1] * H[1]) / (s[0] + s[1]), c = std::sqrt(g1 * (Ht - q2 / 2));
  const bool left = ut[0] >= 0;
  const T x = std::fabs(ut[0]) - c, d = (T)efix * c;
  T k = x < 0 ? x : (T)0;
  if (std::fabs(x) < d) k = (x - (x * x + d * d) / (2 * d)) / 2;
  const T rc = s[0] * s[1] * c, du = u[1][0] - u[0][0], dp = p[1] - p[0];
  const T g = k * (left ? dp - rc * du : dp + rc * du) / (2 * c * c);
  const T gm = std::fabs(k) * (p[0] + p[1] + rc * (std::fabs(u[0][0]) + std::fabs(u[1][0]))) / (2 * c * c);
  const int i = left ? 0 : 1;
  const T m = Q[i][1], un = std::fabs(ut[0]);
  F[0] = m + g;
  sc[0] = std::fabs(m) + gm;
  F[1] = m * u[i][0] + p[i] + g * (left ? x : -x);
  sc[1] = std::fabs(m * u[i][0]) + p[i] + gm * (un + c);
  for (int t = 1; t <= NT; ++t) {
    F[1 + t] = m * u[i][t] + g * ut[t];
    sc[1 + t] = std::fabs(m * u[i][t]) + gm * (std::fabs(u[0][t]) + std::fabs(u[1][t]));
  }
  F[E] = u[i][0] * ((T)Q[i][E] + p[i]) + g * (Ht - c * un);
  sc[E] = std::fabs(u[i][0]) * ((T)Q[i][E] + p[i]) + gm * (Ht + c * un);
}

static std::mt19937_64 rng(2024);
static double uni() { return std::uniform_real_distribution<double>(-1, 1)(rng); }

template <int NT>
static void regime(const char *name, long n, double mach, double jump, double tang, double scale, double gamma,
                   double efix) {
  constexpr int NV = NT + 3;
  const double g1 = gamma - 1;
  const fvk::RoeConst rc = fvk::roe_const(g1, efix);
  long refused = 0;
  double mx[2] = {0, 0}, sq[2] = {0, 0};
  for (long i = 0; i < n; ++i) {
    double Q[2][NV], v0[3];
    const double rho0 = scale * std::exp(uni()), p0 = scale * std::exp(uni()), c0 = std::sqrt(gamma * p0 / rho0);
    for (int c = 0; c <= NT; ++c) v0[c] = mach * c0 * uni() * (c ? tang : 1.0);
    for (int s = 0; s < 2; ++s) {
      const double rho = rho0 * std::exp(jump * uni()), p = p0 * std::exp(jump * uni());
      double k = 0;
      Q[s][0] = rho;
      for (int c = 0; c <= NT; ++c) {
        const double v = v0[c] + jump * c0 * uni() * (c ? tang : 1.0);
        Q[s][1 + c] = (i & 7) == 7 ? 0.0 * v : rho * v;  // momenta of either zero too
        k += Q[s][1 + c] * Q[s][1 + c] / rho;
      }
      Q[s][NT + 2] = p / g1 + k / 2;
    }
    if ((i & 15) == 8)
      for (int v = 0; v < NV; ++v) Q[1][v] = Q[0][v];  // equal states
    double G[NV], D[NV], ds[NV];
    long double F[NV], sc[NV];
    if (!fvk::roe_fixed<NT>(Q[0], Q[1], rc, G)) {
      ++refused;
      continue;
    }
    reference<long double, NT>(Q[0], Q[1], g1, efix, F, sc);
    reference<double, NT>(Q[0], Q[1], g1, efix, D, ds);
    for (int v = 0; v < NV; ++v) {
      if (sc[v] == 0) {
        if (G[v] != 0.0) mx[0] = INFINITY;
        continue;
      }
      const double e[2] = {(double)(std::fabs((long double)G[v] - F[v]) / sc[v]) * 0x1p53,
                           (double)(std::fabs((long double)D[v] - F[v]) / sc[v]) * 0x1p53};
      for (int q = 0; q < 2; ++q) {
        mx[q] = e[q] > mx[q] || e[q] != e[q] ? e[q] : mx[q];
        sq[q] += e[q] * e[q];
      }
    }
  }
  std::printf("%s %dD %ld %g %g %g %g\n", name, NT + 1, refused, mx[0], std::sqrt(sq[0] / (n * NV)), mx[1],
              std::sqrt(sq[1] / (n * NV)));
}

int main(int argc, char **argv) {
  const long n = argc > 1 ? std::atol(argv[1]) : 100000;
  regime<1>("transonic", n, 1.5, 0.05, 1, 1, 1.4, 0.1);
  regime<2>("transonic", n, 1.5, 0.05, 1, 1, 1.4, 0.1);
  regime<1>("jumps", n, 1.0, 0.7, 1, 1, 1.4, 0.1);
  regime<2>("low_mach", n, 1e-4, 1e-5, 1, 1, 1.4, 0.1);
  regime<1>("thin_shear", n, 0.5, 0.01, 1e-10, 1, 1.4, 0.1);
  regime<1>("tiny_units", n, 0.5, 0.05, 1, 1e-60, 1.4, 0.1);
  regime<2>("huge_units", n, 0.5, 0.05, 1, 1e60, 1.4, 0.1);
  regime<1>("monatomic_wide_fix", n, 1.0, 0.05, 1, 1, 5.0 / 3.0, 0.9);
  regime<1>("gamma_2.5_no_fix", n, 1.0, 0.05, 1, 1, 2.5, 0.0);
  regime<1>("gamma_1.01", n, 1.0, 0.05, 1, 1, 1.01, 0.1);

  // states left to FP64
  const fvk::RoeConst rc = fvk::roe_const(0.4, 0.1);
  const double inf = std::numeric_limits<double>::infinity(), nan = std::numeric_limits<double>::quiet_NaN();
  const double sub = 1e-310;
  const double base[4] = {1, 0.3, -0.2, 2};
  struct { int v; double x; } one[] = {{0, 0.0},  {0, -1.0}, {0, sub}, {0, inf}, {0, nan}, {1, inf},
                                       {1, nan}, {2, nan}, {3, 0.0}, {3, -1.0}, {3, sub}, {3, inf},  {3, nan},
                                       {1, 10.0}, {0, 1e-12}};
  long bad = 0, all = 0;
  for (auto &o : one)
    for (int s = 0; s < 2; ++s) {
      double Q[2][4], G[4];
      for (int v = 0; v < 4; ++v) Q[0][v] = Q[1][v] = base[v];
      Q[s][o.v] = o.x;
      ++all;
      bad += !fvk::roe_fixed<1>(Q[0], Q[1], rc, G);
    }
  std::printf("refused %ld of %ld\n", bad, all);
  return 0;
}
