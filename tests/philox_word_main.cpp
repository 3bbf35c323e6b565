// Host build of the single-word Philox4x32-10 (csrc/copes_internal.h): for each line "key c0"
// on stdin it prints the four words of counter (c0, 0, 0, tag 0), each from its own call.
#include <cstdio>

#include "../paper_2608_02391_gb300/csrc/copes_internal.h"

int main() {
  unsigned long long key;
  unsigned c0;
  while (std::scanf("%llu %u", &key, &c0) == 2) {
    uint32_t rk[20], row[20];
    copes::philox_round_keys((uint32_t)key, (uint32_t)(key >> 32), rk);
    copes::philox_word_keys(rk, COPES_TAG_NOISE, row);
    const uint64_t m = (uint64_t)copes::kPhiloxM0 * c0;
    for (int w = 0; w < 4; ++w) {
      const bool h = w & 2, odd = w & 1;
      std::printf("%u%c", copes::philox4x32_10_word((uint32_t)m, (uint32_t)(m >> 32), row, h, odd, row[h ? 18 : 16],
                                                    row[h ? 19 : 17]), w == 3 ? '\n' : ' ');
    }
  }
  return 0;
}
