// Host check of the pieces of the integer-pipe arithmetic (csrc/fv_roe.h): prints
// "ok" or the first deviation.
#include <cinttypes>
#include <cmath>
#include <cstdio>
#include <cstdlib>
#include <cstring>
#include <limits>
#include <random>

#include "../../paper_2306_14011_gb300/csrc/fv_roe.h"

static bool shifts() {
  const uint64_t as[] = {0, 1, 0x7fffffffffffffffull, 0x8000000000000000ull, 0xffffffffffffffffull, 0xc000000000000001ull};
  for (uint64_t a : as)
    for (int s = -3; s < 300; ++s) {
      const __int128 wide = (__int128)(int64_t)a;
      const uint64_t want = s < 0 || s > 63 ? 0 : a >> s;
      const int64_t wants = (int64_t)(wide >> (s < 0 || s > 127 ? 127 : s));
      if (fvk::fx_shr(a, s) != want || fvk::fx_sar((int64_t)a, s) != wants) {
        std::printf("shift of %016" PRIx64 " by %d: %016" PRIx64 " %016" PRIx64 "\n", a, s, fvk::fx_shr(a, s),
                    (uint64_t)fvk::fx_sar((int64_t)a, s));
        return false;
      }
    }
  return true;
}

static std::mt19937_64 rng(11);

// A positive double with the exponent field e; its significand random, or within
// a few units of 1 or of 2.
static double with_field(int e) {
  uint64_t f = rng() & 0xfffffffffffffull;
  switch (rng() % 4) {
    case 0: f &= 7; break;
    case 1: f |= 0xffffffffffff8ull; break;
    case 2: f &= 0xffffffe000000ull; break;  // what an FP32 seed takes exactly
  }
  const uint64_t b = ((uint64_t)e << 52) | f;
  double x;
  std::memcpy(&x, &b, 8);
  return x;
}

// got against the exact value, 0.51 units in the exact value's last place.
static bool near(double got, long double want) {
  int e;
  std::frexp(want, &e);
  return std::fabs((long double)got - want) <= 0.51L * std::ldexp(1.0L, e - 53);
}
static bool fail(const char *what, double a, double b, double got, int bad) {
  std::printf("%s(%a, %a) = %a, bad %d\n", what, a, b, got, bad);
  return false;
}

static bool mul(double a, double b) {
  int bad = 0;
  const double got = fvk::fx_mul(a, b, bad);
  const long double want = (long double)a * b;
  const bool finite = std::isfinite(a) && std::isfinite(b);
  if (bad < 0) return !finite || std::fabs(want) >= 0x1p1023L || fail("mul refused", a, b, got, bad);
  if (!finite) return fail("mul", a, b, got, bad);
  if (!std::isnormal(a) || !std::isnormal(b) || std::fabs(want) < 0x1p-1022L)
    return got == 0.0 || fail("mul to zero", a, b, got, bad);
  if (std::fabs(want) == 0x1p-1022L && got == 0.0) return true;  // the exact product may be just below
  return near(got, want) || fail("mul", a, b, got, bad);
}
static bool rcp(double x, bool takes) {
  int bad = 0;
  const double got = fvk::fx_rcp64(x, bad);
  return takes ? (bad >= 0 && near(got, 1.0L / x)) || fail("rcp", x, 0, got, bad) : bad < 0 || fail("rcp takes", x, 0, got, bad);
}
static bool rsqrt(double x, bool takes) {
  int bad = 0;
  const double got = fvk::fx_rsqrt64(x, bad);
  return takes ? (bad >= 0 && near(got, 1.0L / std::sqrt((long double)x))) || fail("rsqrt", x, 0, got, bad)
               : bad < 0 || fail("rsqrt takes", x, 0, got, bad);
}

static bool operations(long n) {
  bool ok = true;
  const double inf = std::numeric_limits<double>::infinity(), nan = std::numeric_limits<double>::quiet_NaN();
  const double ends[] = {0.0, 5e-324, 0x1.fffffffffffffp-1023, 0x1p-1022, 0x1.8p-511, 1.0, 0x1.fffffffffffffp511,
                         0x1p1023, std::numeric_limits<double>::max(), inf, nan};
  for (double a : ends)
    for (double b : ends)
      for (int s = 0; s < 4; ++s) ok = ok && mul(s & 1 ? -a : a, s & 2 ? -b : b);
  for (long i = 0; i < n && ok; ++i) {
    const int ea = 1 + (int)(rng() % 2046), sum = 1020 + (int)(rng() % 2), eb = (int)(rng() % 2047);
    const double sign = rng() & 1 ? -1.0 : 1.0;
    ok = mul(sign * with_field(ea), with_field(eb)) && mul(with_field(ea), sign * with_field(1024));  // any; results of every size
    const int other = sum + 3 - ea;                                                                   // results next to 2^-1022
    if (other >= 1 && other <= 2046) ok = ok && mul(with_field(ea), with_field(other));
    if (3068 - ea <= 2046 && 3068 - ea >= 1) ok = ok && mul(with_field(ea), with_field(3068 - ea));   // ... and to 2^1023
  }
  for (int e = 0; e <= 2047 && ok; ++e)  // every exponent field, both parities
    for (int k = 0; k < 64 && ok; ++k) {
      const double x = with_field(e);
      ok = rcp(x, e >= 2 && e <= 2044) && rcp(-x, false) && rsqrt(x, e >= 1 && e <= 2046) && rsqrt(-x, false);
    }
  for (long i = 0; i < n && ok; ++i) ok = rcp(with_field(1023), true) && rsqrt(with_field(1022 + (i & 1)), true);
  return ok;
}

// The mass flux of faces next to the edge of the entropy fix, |u~_n - c~| = delta (1
// +- 2^-1 .. 2^-40), against long double: the magnitudes that it sums, m and k
// alpha with their terms, times 4 units of 2^-53 as for the whole flux.
static bool edge(double efix, double sign, double eps) {
  const long double g1 = 0.4;
  std::uniform_real_distribution<double> u01(0, 1);
  const fvk::RoeConst rc = fvk::roe_const(0.4, efix);
  double Q[2][4];
  const double rho = 1 + 0.2 * u01(rng), p[2] = {1.0, 1 + 0.1 * u01(rng)};
  const long double c = std::sqrt(1.4L * (p[0] + p[1]) / 2 / rho);  // equal densities and velocities
  const double u = (double)(c * (1 + (long double)sign * efix * (1 + eps)));
  for (int s = 0; s < 2; ++s) {
    Q[s][0] = rho;
    Q[s][1] = rho * u;
    Q[s][2] = 0;
    Q[s][3] = p[s] / 0.4 + 0.5 * rho * u * u;
  }
  // the same from the rounded states
  long double P[2], H = 0;
  const long double ul = (long double)Q[0][1] / rho;
  for (int s = 0; s < 2; ++s) {
    P[s] = g1 * (Q[s][3] - (long double)Q[s][1] * Q[s][1] / rho / 2);
    H += (Q[s][3] + P[s]) / rho / 2;
  }
  const long double ct = std::sqrt(g1 * (H - ul * ul / 2)), x = ul - ct, d = (long double)efix * ct;
  long double k = x < 0 ? x : 0;
  if (std::fabs(x) < d) k = -(d - x) * (d - x) / (4 * d);
  const long double want = Q[0][1] + k * (P[1] - P[0]) / (2 * ct * ct);
  const long double scale = Q[0][1] + (std::fabs(k) + ct) * (P[0] + P[1]) / (2 * ct * ct);
  double G[4];
  if (!fvk::roe_fixed<1>(Q[0], Q[1], rc, G) || std::fabs(G[0] - want) > 4 * 0x1p-53L * scale) {
    std::printf("fix %g at %g %g: %a, exact %La, off by %Lg units\n", efix, sign, eps, G[0], want,
                (G[0] - want) / scale * 0x1p53L);
    return false;
  }
  return true;
}
static bool edges() {
  for (double efix : {0.9, 0.3, 0.1, 1e-2, 1e-3, 1e-5, 1e-7, 1e-9})
    for (int b = 1; b <= 40; ++b)
      for (int s = 0; s < 64; ++s)
        if (double v = 1 + (s & 1 ? 1 : -1) * 1.5 * efix; v > 0.1 && !edge(efix, s & 1 ? 1 : -1, (s & 2 ? 1 : -1) * std::exp2(-b))) return false;
  return true;
}

// The van Leer slope: 0.53 units in the last place of the quotient, and s's own
// rounding (2^-53 of it); over a range no further from exact than FP64 operations.
static bool vanleer(long n) {
  std::uniform_real_distribution<double> u01(0, 1);
  for (int kind = 0; kind < 6; ++kind) {
    double sq[2] = {0, 0};
    for (long i = 0; i < n; ++i) {
      double a = u01(rng) + 1e-9, b = kind == 0 ? u01(rng) + 1e-9 : kind == 1 ? a * (1 + 1e-3 * u01(rng)) : kind == 2 ? a
                                      : a * std::exp2((kind == 3 ? -20 : kind == 4 ? -60 : -900) * u01(rng));
      if (i & 1) std::swap(a, b);
      if (i & 2) a = -a, b = -b;
      int bad = 0, e;
      const double s = a + b, got = fvk::fx_vanleer(a, b, s, bad);
      const long double want = 2.0L * a * b / ((long double)a + b);
      std::frexp(want, &e);
      const long double ulp = std::ldexp(1.0L, e - 53);
      if (bad < 0 || std::fabs(got - want) > 0.53L * ulp + 0x1p-53L * std::fabs(want)) return fail("vanleer", a, b, got, bad);
      const double fp64 = (2.0 * a * b) * (1.0 / s);
      sq[0] += (double)((got - want) / ulp) * (double)((got - want) / ulp);
      sq[1] += (double)((fp64 - want) / ulp) * (double)((fp64 - want) / ulp);
    }
    if (sq[0] > sq[1]) {
      std::printf("vanleer, kind %d: rms %g units, FP64 operations %g\n", kind, std::sqrt(sq[0] / n), std::sqrt(sq[1] / n));
      return false;
    }
  }
  // the ends of what it takes
  const double inf = std::numeric_limits<double>::infinity(), nan = std::numeric_limits<double>::quiet_NaN();
  const struct { double a, b; bool takes; } ends[] = {
      {0x1p-1021, 0x1p-1021, true}, {0x1p-1021, 0x1p1020, true}, {0x1p1020, 0x1.fp1020, true}, {0x1p-1022, 1, false},
      {5e-324, 1, false}, {0x1p1021, 0x1p1021, false}, {0x1p1023, 0x1p1023, false}, {inf, 1, false}, {1, inf, false},
      {nan, 1, false}, {1, nan, false}};
  for (auto &x : ends)
    for (int s = -1; s < 2; s += 2) {
      int bad = 0;
      const double got = fvk::fx_vanleer(s * x.a, s * x.b, s * x.a + s * x.b, bad);
      const long double want = s * x.a * (2.0L * x.b / ((long double)x.a + x.b));
      if (x.takes != (bad >= 0) || (x.takes && std::fabs(got - want) > 0x1p-51L * std::fabs(want)))
        return fail("vanleer end", s * x.a, s * x.b, got, bad);
    }
  return true;
}

int main() {
  if (!shifts() || !operations(1000000) || !edges() || !vanleer(300000)) return 1;
  std::printf("ok\n");
  return 0;
}
