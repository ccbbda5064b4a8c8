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

int main() {
  if (!shifts() || !operations(1000000)) return 1;
  std::printf("ok\n");
  return 0;
}
