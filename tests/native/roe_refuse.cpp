// Host check that the integer-pipe Roe flux (csrc/fv_roe.h) takes no face with a
// side of negative pressure.
//   roe_refuse CASES
// prints, per dimension and side: name, faces of negative pressure, faces of
// them that were taken.  Kinetic energy from just above the total energy to
// 1000 times it, in every direction, over the densities' and energies' range.
#include <cmath>
#include <cstdio>
#include <cstdlib>
#include <random>

#include "../../paper_2306_14011_gb300/csrc/fv_roe.h"

static std::mt19937_64 rng(7);
static double uni(double a, double b) { return std::uniform_real_distribution<double>(a, b)(rng); }

// A state of energy E whose kinetic energy is about `ratio` times it.
template <int NT>
static void state(double rho, double E, double ratio, double *Q) {
  double d[NT + 1], n = 0;
  for (int c = 0; c <= NT; ++c) {
    d[c] = uni(-1, 1) * (uni(0, 1) < 0.3 ? std::exp2(uni(-60, 0)) : 1.0) * (uni(0, 1) < 0.2 ? 0.0 : 1.0);
    n += d[c] * d[c];
  }
  if (n == 0) n = d[0] = 1;
  for (int c = 0; c <= NT; ++c) Q[1 + c] = d[c] / std::sqrt(n) * std::sqrt(2 * rho * E * ratio);
  Q[0] = rho;
  Q[NT + 2] = E;
}

template <int NT>
static bool negative(const double *Q) {
  long double k = 0;
  for (int c = 0; c <= NT; ++c) k += (long double)Q[1 + c] * Q[1 + c] / (2 * (long double)Q[0]);
  return Q[NT + 2] - k < -0x1p-50L * Q[NT + 2];  // beyond what the arithmetic's 56 bits can decide
}

template <int NT>
static void scan(const char *name, long n, int which) {  // 0: left, 1: right, 2: both and equal, 3: both
  static const double gammas[] = {1.01, 1.4, 5.0 / 3.0, 2.5};
  long found = 0, taken = 0;
  for (long i = 0; i < n; ++i) {
    double Q[2][NT + 3], G[NT + 3];
    const double rho = std::exp2(uni(-200, 200)), E = std::exp2(uni(-200, 200));
    for (int s = 0; s < 2; ++s) {
      const bool bad = which >= 2 || s == which;
      state<NT>(rho * std::exp(uni(-1, 1)), E * std::exp(uni(-1, 1)), bad ? 1 + std::exp2(uni(-40, 10)) : uni(0, 0.99), Q[s]);
    }
    if (which == 2)
      for (int v = 0; v < NT + 3; ++v) Q[1][v] = Q[0][v];
    if (!negative<NT>(Q[0]) && !negative<NT>(Q[1])) continue;
    ++found;
    taken += fvk::roe_fixed<NT>(Q[0], Q[1], fvk::roe_const(gammas[i & 3] - 1, 0.1), G);
  }
  std::printf("%s %dD %ld %ld\n", name, NT + 1, found, taken);
}

int main(int argc, char **argv) {
  const long n = argc > 1 ? std::atol(argv[1]) : 100000;
  const char *name[] = {"left", "right", "equal", "both"};
  for (int w = 0; w < 4; ++w) {
    scan<1>(name[w], n, w);
    scan<2>(name[w], n, w);
  }
  return 0;
}
