// Host check of the pieces of the integer-pipe arithmetic (csrc/fv_roe.h): prints
// "ok" or the first deviation.
#include <cinttypes>
#include <cstdio>

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

int main() {
  if (!shifts()) return 1;
  std::printf("ok\n");
  return 0;
}
