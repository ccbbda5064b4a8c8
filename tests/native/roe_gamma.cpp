// The regimes of roe_check.cpp at large ratios of specific heats, in the form for
// those:
//   roe_gamma CASES
// prints roe_check's lines (name, faces not taken, errors of the integer flux and
// of the FP64 evaluation).
#include "../../paper_2306_14011_gb300/csrc/fv_roe.h"

namespace fvk {
template <int NT>
bool roe_large_gamma(const double (&QL)[NT + 3], const double (&QR)[NT + 3], const RoeConst &rc, double (&G)[NT + 3]) {
  return roe_fixed<NT, true>(QL, QR, rc, G);
}
}  // namespace fvk

#define roe_fixed roe_large_gamma
#define main roe_check_main
#include "roe_check.cpp"
#undef main

int main(int argc, char **argv) {
  const long n = argc > 1 ? std::atol(argv[1]) : 100000;
  for (double gamma : {1.4, 2.99, 3.01, 4.0, 5.0, 7.0, 8.99, 9.01, 17.0, 40.0, 200.0})
    for (double mach : {0.01, 0.6, 1.5, 4.0}) {
      char name[40];
      std::snprintf(name, sizeof name, "gamma_%g_mach_%g", gamma, mach);
      regime<1>(name, n, mach, mach * 0.05, 1, 1, gamma, 0.1);
      regime<2>(name, n, mach, mach * 0.05, 1, 1, gamma, 0.1);
    }
  return 0;
}
