// How a launch over TILES is cut into units of work, one grid block each.  Host code without CUDA
// calls: the tests build it on its own.
#pragma once

#include <stdint.h>

#include <algorithm>

#include "../../include/copes.h"

namespace copes {

// With g = u >> log_parts, unit u covers part u - (g << log_parts) of the tiles
// [g run, (g + 1) run); adjacent tiles of a run are joined.
struct TileUnits {
  uint32_t n_units, log_parts, run;
};

constexpr uint32_t kRunMax = 30;           // a warp looks at a run's tiles and one on either side
constexpr uint64_t kDefaultTile = 16384;
constexpr uint64_t kUnitsAtOnce = 4 * 152;    // blocks per SM and SMs
constexpr uint64_t kShortLaunch = 2 * kUnitsAtOnce * kDefaultTile;

// What a launch knows of its tiles: how many there are, their mean length, and whether they
// begin at multiples of 4, with whole groups.
struct TileWork {
  uint64_t n_tiles, mean;
  bool aligned;
  uint64_t elements() const { return n_tiles * mean; }
};

// From a subspace's hint (copes_subspace.n_index over TILES).  Without one the tiles are taken
// for default ones, or for as long as the arena allows if that is less.
inline TileWork tile_work(uint64_t n_tiles, uint64_t n_alloc, uint64_t hint) {
  const uint64_t elements = hint >> 1;
  const bool known = elements && elements <= n_alloc;
  const uint64_t mean = known ? elements / n_tiles : std::min(n_alloc / n_tiles, kDefaultTile);
  return TileWork{n_tiles, std::min<uint64_t>(std::max<uint64_t>(mean, 1), COPES_TILE_MAX), !known || (hint & 1)};
}

// Units of about `unit` elements: tiles more than half as long again in 2^k parts, shorter ones
// in runs of whole tiles that hold no more.  Parts are whole steps of 1,024 elements, so the
// parts of a tile that is not a power of two of them differ by a step: a coarser cut is taken
// where its longest part times its waves of units is less.
inline TileUnits cut_tiles(const TileWork &w, uint64_t unit) {
  TileUnits u{0, 0, 1};
  while (2 * (w.mean >> u.log_parts) > 3 * unit && w.n_tiles << (u.log_parts + 1) <= 1u << 30) ++u.log_parts;
  const uint64_t steps = std::max<uint64_t>((w.mean + 512) / 1024, 1);
  auto cost = [&](uint32_t log) {
    return (((w.n_tiles << log) + kUnitsAtOnce - 1) / kUnitsAtOnce) * ((steps + (1u << log) - 1) >> log);
  };
  while (u.log_parts > 0 && cost(u.log_parts - 1) < cost(u.log_parts)) --u.log_parts;
  if (u.log_parts == 0) u.run = (uint32_t)std::min<uint64_t>(std::max<uint64_t>(unit / w.mean, 1), kRunMax);
  u.n_units = (uint32_t)(u.run > 1 ? (w.n_tiles + u.run - 1) / u.run : w.n_tiles << u.log_parts);
  return u;
}

// Whether the noise ops' kernels for default tiles serve these: tiles of 4,096 elements, or twice,
// four times ... as many, but for the last ones of their ranges, that begin with whole groups;
// or so long that few of their parts do not.
inline bool default_like(const TileWork &w) {
  uint64_t size = 4096;
  while (size < w.mean) size *= 2;
  return (w.aligned || size >= 4 * kDefaultTile) && 10 * w.mean > 9 * size;
}

// The noise ops over TILES, their kernel and its units.
// Elements per unit: few elements are spread over the SMs; many go in units as long as leaves the
// last wave short.  us, by units of 4,096 / 8,192 / 16,384:
// - default tiles, bf16 perturb, pair, two pairs: 4M 7.7 / 8.9 / 7.3, 8.4 / 9.3 / 8.3, 12.9 / 13.5 /
//   12.9; 15M 19.8 / 23.5 / 20.3, 22.7 / 24.7 / 23.8, 35.9 / 37.0 / 36.4; 134M 146 / 169 / 136,
//   172 / 184 / 164, 286 / 290 / 256.  8,192 elements have no form of their own.  The fp32 pair
//   and two pairs, whose stores are twice as long: 134M 232 / 238 / 242, 397 / 405 / 412.
// - other tiles (of 1,000): 1M 3.8 / 3.7 / 5.0, 4.2 / 4.2 / 5.8, 5.2 / 5.3 / 8.0; 11.1M 18.8 / 17.0 /
//   17.1, 21.6 / 20.0 / 21.1, 31.1 / 29.6 / 29.8; 134M 193 / 160 / 145, 225 / 191 / 177, 332 / 297 /
//   280; fp32 pair and two pairs 259 / 236 / 240, 394 / 398 / 405.
// - restores to 1 and 4 copies: 2M 3.8 / 3.1 / 3.3, 5.3 / 5.1 / 5.7; 134M 145 / 117 / 114, 237 / 232 / 234;
//   4 copies in fp32 386 / 392 / 398.  The partner copy is as the restore to one.
inline uint64_t small_unit(uint64_t elements) {
  return elements < 128u << 10 ? 1024 : (elements < 384u << 10 ? 2048 : 4096);
}

enum class NoiseOp { kPerturb, kPair, kTwoPairs, kInit };
struct NoisePlan {
  bool ragged;  // elem_ragged_kernel, else elem_tiles_kernel
  TileUnits units;
};

inline NoisePlan plan_noise(const TileWork &w, uint64_t n_alloc, NoiseOp op, bool fp32) {
  const uint64_t n = w.elements();
  if (n_alloc > 1ull << 34 || !default_like(w)) {
    uint64_t unit = small_unit(n);
    if (n >= 3u << 19 && !(fp32 && op == NoiseOp::kTwoPairs))
      unit = n < 6u << 20 || (fp32 && op == NoiseOp::kPair) ? 8192 : kDefaultTile;
    return NoisePlan{true, cut_tiles(w, unit)};
  }
  if (n < 128u << 10) return NoisePlan{false, cut_tiles(w, 1024)};
  const bool pairs = op == NoiseOp::kPair || op == NoiseOp::kTwoPairs;
  // parts of a tile with a cut group are whole spans only where they are as long as those
  const uint64_t short_launch = !w.aligned ? 3u << 20 : (op == NoiseOp::kInit ? 6u << 20 : kShortLaunch);
  return NoisePlan{false, cut_tiles(w, n < short_launch || (fp32 && pairs) ? 4096 : kDefaultTile)};
}

// Restores by the working copies beyond w that they write; the partner copy as -1.
inline TileUnits plan_copy(const TileWork &w, int copies, bool fp32) {
  const uint64_t n = w.elements();
  if (n < 3u << 19) return cut_tiles(w, small_unit(n));
  if (copies > 0) return cut_tiles(w, fp32 && copies == 3 ? 4096 : 8192);
  return cut_tiles(w, n < (copies < 0 ? 8u << 20 : 3u << 20) ? 8192 : kDefaultTile);
}

// log2 of the parts an update cuts the default tile into (units of other tiles are as long).  From
// four noise vectors on: up to 128 tiles, sixteenths (one group a thread).  Beyond, of the cuts
// that give each SM its four blocks, the one with the least ceil(parts / slots) (1 / 2^log +
// overhead / P), the overhead of a part being a fifth to a third of a tile's time for one
// noise vector: up to two waves of tiles the SM with the most parts sets the time (152 slots),
// beyond the last wave does (608), where parts have to gain 3%; four noise vectors beyond two
// waves take whole tiles.  A block a tile / eighths to 608 tiles, whole ones above / this, us:
// P = 16, 3M, 6M, 11.1M and 18M elements 84.6 / 51.2 / 49.2, 122.6 / 93.8 / 91.5, 196 / 176 /
// 155 and 306 / 272 / 266; P = 4, 8M 48.0 / 47.8 / 39.3; P = 64, 30M and 134M 1,900 / 1,670 /
// 1,574 and 7,820 / 7,066 / 6,867.
// Up to three noise vectors the update is bound by memory and by its blocks' starts: the cut with
// the least waves times its steps, a start counted as three of them; beyond a wave of whole
// tiles only for one noise vector, and where that gains a tenth.  Sixteenths to 192 tiles and whole
// ones above / this, P = 1: 1M, 2M, 4M and 11.1M elements 6.5 / 5.1, 9.4 / 7.5, 12.2 / 11.7 and 27.2 /
// 25.4; halves of 24M 44.0 / 46.8, and for P = 2 and 3 of 14.5M 36.2 / 38.2 and 47.1 / 49.7.
inline uint32_t update_log_parts(uint64_t n_tiles, int n_noise) {
  uint32_t best = 0;
  double best_cost = 1e30;
  if (n_noise <= 3) {
    for (uint32_t log = 0; log <= 4; ++log) {
      if (log && n_noise > 1 && n_tiles > kUnitsAtOnce) break;
      const double cost = (double)(((n_tiles << log) + kUnitsAtOnce - 1) / kUnitsAtOnce * ((16 >> log) + 3));
      if (cost < best_cost * (best == 0 && n_tiles > kUnitsAtOnce ? 0.9 : 1.0)) best = log, best_cost = cost;
    }
    return best;
  }
  if (n_tiles <= 128) return 4;
  const bool waves = n_tiles > 2 * kUnitsAtOnce;
  if (waves && n_noise == 4) return 0;
  const uint64_t slots = waves ? kUnitsAtOnce : 152;
  const double overhead = (waves ? 0.3 : 0.2) / n_noise;
  for (uint32_t log = 0; log <= (waves ? 2u : 3u); ++log) {
    if ((n_tiles << log) < kUnitsAtOnce) continue;
    const double cost = (double)(((n_tiles << log) + slots - 1) / slots) * (1.0 / (1 << log) + overhead);
    if (cost < best_cost * (waves && best == 0 ? 0.97 : 1.0)) best = log, best_cost = cost;
  }
  return best;
}

// The run of short tiles that leaves the SM with the most units the least to do, as the cut of
// default tiles: 11.1M elements in tiles of 1,000, P = 7 85 us in runs of 8, 77 in these.
inline void best_run(TileUnits &u, const TileWork &w, int n_noise) {
  uint64_t best = ~0ull;
  for (uint32_t run = 1; run <= kRunMax && run * w.mean <= kDefaultTile + 1024; ++run) {
    const uint64_t units = (w.n_tiles + run - 1) / run;
    if (units < kUnitsAtOnce) break;
    const uint64_t cost = (units + 151) / 152 * (run * w.mean + 3277 / n_noise);
    if (cost < best) best = cost, u.run = run, u.n_units = (uint32_t)units;
  }
}

// The same for the parts of long tiles: 11.1M elements in tiles of 24,000, P = 6 85.6 us cut as
// default tiles are, 74.1 in these.
inline void best_parts(TileUnits &u, const TileWork &w, int n_noise) {
  uint64_t best = ~0ull;
  const uint64_t steps = (w.mean + 512) / 1024;
  for (uint32_t log = 0; steps >> log >= 2; ++log) {
    const uint64_t units = w.n_tiles << log;
    if (units < kUnitsAtOnce) continue;
    const uint64_t cost = (units + 151) / 152 * (((steps + (1u << log) - 1) >> log) * 1024 + 3277 / n_noise);
    if (cost < best) best = cost, u.log_parts = log, u.n_units = (uint32_t)units;
  }
}

inline TileUnits plan_update(const TileWork &w, int n_noise) {
  const uint64_t defaults = std::max<uint64_t>(w.elements() / kDefaultTile, 1);
  TileUnits u = cut_tiles(w, kDefaultTile >> update_log_parts(defaults, n_noise));
  if (n_noise > 3 && defaults > 128 && defaults <= 2 * kUnitsAtOnce) {
    if (u.run > 1) best_run(u, w, n_noise);
    else best_parts(u, w, n_noise);
  }
  return u;
}

// The backup mode.
// Elements per unit: parts of `part` up to two waves of default tiles; short tiles in runs of up to
// as many as leave 500 units, since the host link takes whole lines (11.1M elements in tiles
// of 1,000, update, P = 1: 147 us, 174 in runs of 2).  Few elements are spread wide: the link's
// latency is hidden by threads.
inline TileUnits plan_backup(const TileWork &w, uint64_t part) {
  const uint64_t n = w.elements();
  if (w.mean < 8192) return cut_tiles(w, std::min(std::max<uint64_t>(n / 500, 1024), kDefaultTile));
  return cut_tiles(w, n < 1u << 20 ? 1024 : (n <= kShortLaunch ? part : kDefaultTile));
}

}  // namespace copes
