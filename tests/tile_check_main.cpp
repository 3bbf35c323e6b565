// Host build of the kernels' tile checks (csrc/copes_internal.h): for each line "b e n_alloc
// part log_parts" on stdin it prints tile_in_arena and tile_in_whole_parts.
#include <cstdio>

#include "../paper_2608_02391_gb300/csrc/copes_internal.h"

int main() {
  unsigned long long b, e, n;
  unsigned part, log_parts;
  while (std::scanf("%llu %llu %llu %u %u", &b, &e, &n, &part, &log_parts) == 5)
    std::printf("%d %d\n", copes::tile_in_arena(b, e, n), copes::tile_in_whole_parts(b, e, n, part, log_parts));
  return 0;
}
