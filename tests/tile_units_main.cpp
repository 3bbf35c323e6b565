// Host build of the tile launches' cut into units (csrc/tile_units.h): for each line "n_tiles
// n_alloc elements aligned" on stdin (elements 0: no hint) it prints, for each call below, its
// units, log2 of the parts and the run: the noise ops in bf16 and fp32 (led by 1 for the ragged
// tiles' kernel), the copies, updates by 1, 4 and 32 noise vectors, and the backup mode's.
#include <cstdio>

#include "../paper_2608_02391_gb300/csrc/tile_units.h"

static void print(const copes::TileUnits &u) { std::printf("%u %u %u  ", u.n_units, u.log_parts, u.run); }

int main() {
  unsigned long long n_tiles, n_alloc, elements;
  int aligned;
  while (std::scanf("%llu %llu %llu %d", &n_tiles, &n_alloc, &elements, &aligned) == 4) {
    const copes::TileWork w = copes::tile_work(n_tiles, n_alloc, elements ? COPES_TILES_HINT(elements, aligned) : 0);
    for (bool fp32 : {false, true})
      for (auto op : {copes::NoiseOp::kPerturb, copes::NoiseOp::kPair, copes::NoiseOp::kTwoPairs, copes::NoiseOp::kInit}) {
        const copes::NoisePlan p = copes::plan_noise(w, n_alloc, op, fp32);
        std::printf("%d ", p.ragged);
        print(p.units);
      }
    for (int copies : {-1, 0, 1, 3}) print(copes::plan_copy(w, copies, false));
    for (int P : {1, 4, 32}) print(copes::plan_update(w, P));
    for (int part : {4096, 2048}) print(copes::plan_backup(w, part));
    std::printf("\n");
  }
  return 0;
}
