// Host build of the folded keys for one other high word (csrc/copes_internal.h, HighKeys): for each line
// "key c0 c1 tag" on stdin it prints the words of counter (c0, c1, 0, tag).
#include <cstdio>

#include "../paper_2608_02391_gb300/csrc/copes_internal.h"

int main() {
  unsigned long long key;
  unsigned c0, c1, tag;
  while (std::scanf("%llu %u %u %u", &key, &c0, &c1, &tag) == 4) {
    uint32_t rk[20], u[20], x[4];
    copes::philox_round_keys((uint32_t)key, (uint32_t)(key >> 32), rk);
    copes::philox_folded_keys(rk, tag, u);
    const uint64_t m = (uint64_t)copes::kPhiloxM0 * c0;
    copes::philox4x32_10_folded((uint32_t)m, (uint32_t)(m >> 32), copes::HighKeys(u, rk, c1), x);
    std::printf("%u %u %u %u\n", x[0], x[1], x[2], x[3]);
  }
  return 0;
}
