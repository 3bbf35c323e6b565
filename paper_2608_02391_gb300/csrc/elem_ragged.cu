// The elementwise noise ops over TILES of any length and place: tiles that are not whole parts of
// the default tile, that begin in the middle of a group, or whose counters pass 2^32.  (Default
// tiles have kernels of their own in es_kernels.cu, whose bounds are compile-time constants.
// In one kernel the two forms cost each other registers: the pair perturb of 15M elements in
// default tiles took 24.6 us instead of 22.1 with the cuts below beside them.)
#include "elem_ops.cuh"

namespace copes {

__device__ unsigned int g_ragged_error = 0;

__device__ __forceinline__ void ragged_flag(unsigned bit) { atomicOr(&g_ragged_error, bit); }

// The tiles a unit looks at: lane 1 + i of every warp holds tile i of the unit's run, and lanes 0
// and 1 + run the tiles before and after it.
__device__ __forceinline__ bool unit_lane(uint32_t unit, const ElemArgs &a, uint64_t &tile) {
  const uint32_t lane = threadIdx.x & 31u;
  tile = (uint64_t)(unit >> a.units.log_parts) * a.units.run + lane - 1;
  return lane <= a.units.run + 1 && tile < a.n_tiles;  // the tile before the first wraps
}

__device__ __forceinline__ ulonglong2 load_unit(uint32_t unit, const ElemArgs &a) {
  uint64_t t;
  if (!unit_lane(unit, a, t)) return make_ulonglong2(1, 0);  // no tile
  return __ldg(reinterpret_cast<const ulonglong2 *>(a.tiles) + t);
}

// The unit's first stretch of adjacent tiles from lane `from` on, as [b, e) with `from` past it;
// false when there is none.  v: load_unit's tile of the lane.  A tile outside the arena, or,
// for the pair, outside the partner buffer, is flagged and left out.
//
// Where one tile continues another, the cut between them is moved down to the next multiple of
// 64, if the lower tile reaches that far: both sides of the cut look at the same two tiles
// and move it alike.  So all stretches of a range of any begin are whole cache lines but its
// first and last, and no group of 4 is cut inside a range.  Measured on ranges that begin at
// an odd place (bf16, default tiles; cuts where they lie / moved): perturb and pair of 11.1M
// elements 20.5 / 16.7 and 22.8 / 20.9 us, two pairs 33.3 / 30.0.
template <int OP>
__device__ __forceinline__ bool unit_stretch(ulonglong2 v, uint32_t unit, const ElemArgs &a, uint32_t &from,
                                             uint64_t &b, uint64_t &e) {
  constexpr uint32_t kAll = 0xffffffffu;
  const uint32_t lane = threadIdx.x & 31u, run = a.units.run;
  bool ok = tile_in_arena(v.x, v.y, a.n_alloc);
  uint64_t t;
  if (!ok && threadIdx.x < 32 && unit_lane(unit, a, t)) ragged_flag(kErrTileRange);
  if (OP == kOpPerturbPair && ok && !(v.x >= a.partner_base && v.y - a.partner_base <= a.partner_len)) {
    if (threadIdx.x < 32) ragged_flag(kErrPartnerRange);
    ok = false;
  }
  const uint64_t before_b = __shfl_up_sync(kAll, v.x, 1), before_e = __shfl_up_sync(kAll, v.y, 1);
  const uint32_t valid = __ballot_sync(kAll, ok);
  const bool joins = ok && lane > 0 && (valid >> (lane - 1) & 1u) && before_e == v.x;
  const uint32_t joined = __ballot_sync(kAll, joins);  // the lane's tile continues the lane before's
  const uint64_t down = v.x & ~63ull, cut = joins && down >= before_b ? down : v.x;
  const uint32_t own = valid & (((1u << run) - 1u) << 1) & ~0u << from;
  if (!own) return false;
  const uint32_t i = __ffs(own) - 1;
  const uint32_t more = (joined & ((2u << run) - 1u)) >> (i + 1);
  const uint32_t j = i + __ffs(~more) - 1;  // the last tile of the run joined to tile i
  from = j + 1;
  b = __shfl_sync(kAll, cut, i);
  const uint64_t end = __shfl_sync(kAll, v.y, j), next = __shfl_sync(kAll, cut, (j + 1) & 31u);
  e = joined >> (j + 1) & 1u ? next : end;
  return true;
}

// The whole groups [lo, hi) (multiples of 4) by the block: steps from the multiple of 64 below
// lo, so that a warp's accesses are whole sectors; of G groups while more than half of one is
// left, then of G / 2, then one of single groups, so that little is generated for nobody.
template <int OP, typename WT, int G, typename Keys>
__device__ __forceinline__ void ragged_range(const ElemArgs &a, const Keys &keys, const WideTable &tab, uint64_t lo,
                                             uint64_t hi) {
  constexpr uint32_t kStep = 4u * kThreads * G;
  const uint64_t base = lo & ~63ull;
  const uint32_t skip = (uint32_t)(lo - base), n = (uint32_t)(hi - base);
  uint32_t at = 0;
  for (; at + kStep / 2 < n; at += kStep)
    elem_step<OP, WT, G, true>(a, keys, tab, base, at + 4u * threadIdx.x, skip, n);
  if (G > 2 && at + kStep / 4 < n) {
    elem_step<OP, WT, G / 2, true>(a, keys, tab, base, at + 4u * threadIdx.x, skip, n);
    at += kStep / 2;
  }
  const uint32_t off = at + 4u * threadIdx.x;
  if (off - skip < n - skip) elem_step<OP, WT, 1>(a, keys, tab, base, off);
}

// The elements [b, e): a group cut by either end by one thread, the whole groups by the block.
template <int OP, typename WT, int G, typename Keys>
__device__ __forceinline__ void ragged_stretch(const ElemArgs &a, const Keys &keys, const WideTable &tab, uint64_t b,
                                               uint64_t e) {
  const uint64_t lo = (b + 3) & ~3ull, hi = e & ~3ull;  // the whole groups, if lo < hi
  if (lo != b && threadIdx.x == kThreads - 1) elem_partial_group<OP, WT>(a, keys, tab, b, min(lo, e));
  if (hi != e && hi >= lo && threadIdx.x == kThreads - 33) elem_partial_group<OP, WT>(a, keys, tab, hi, e);
  if (lo < hi) ragged_range<OP, WT, G>(a, keys, tab, lo, hi);
}

// One unit a block, 4 blocks of 256 threads per SM.  Groups per thread step (bf16, 44.7M elements
// in tiles of 1,000, us): perturb 4 at 4 blocks 51.6, 2 at 5 blocks 55.2, 8 at 3 blocks 57.4;
// pair 62.9, 69 and 65.6; two pairs 2 at 4 blocks 98.5, 1 at 5 blocks 105, 4 at 2 blocks 110.
// HIGH: the form for arenas of more than 2^34 elements.
template <int OP>
constexpr int ragged_groups() { return OP == kOpPerturbTwoPairs ? 2 : 4; }

template <int OP, typename WT, bool HIGH>
__global__ void __launch_bounds__(kThreads, 4) elem_ragged_kernel(const __grid_constant__ ElemArgs a) {
  constexpr int G = ragged_groups<OP>();
  __shared__ __align__(128) float4 s_tab[WideTable::kFloat4s];
  ulonglong2 v = load_unit(blockIdx.x, a);  // on its way while the table is filled
  WideTable::fill(s_tab);
  __syncthreads();
  const WideTable tab(s_tab);
  uint32_t from = 1;
  uint64_t b, e;
  while (unit_stretch<OP>(v, blockIdx.x, a, from, b, e)) {
    if (a.units.log_parts) tile_part(a.units, blockIdx.x & ((1u << a.units.log_parts) - 1u), b, e);
    if constexpr (HIGH) {
      while (b < e) {  // one pass, two where the counters' high word changes
        const uint64_t end = min(e, ((b >> 34) + 1) << 34);
        ragged_stretch<OP, WT, G>(a, HighWord(a, (uint32_t)(b >> 34)), tab, b, end);
        b = end;
      }
    } else if (b < e) {
      ragged_stretch<OP, WT, G>(a, LowKeys{}, tab, b, e);
    }
    if (from > a.units.run) return;
    v = load_unit(blockIdx.x, a);  // again, rather than keep it through the stretch
  }
}

template <int OP, typename WT>
static cudaError_t launch_ragged_typed(const ElemArgs &a, cudaStream_t s) {
  if (a.n_alloc > 1ull << 34) elem_ragged_kernel<OP, WT, true><<<a.units.n_units, kThreads, 0, s>>>(a);
  else elem_ragged_kernel<OP, WT, false><<<a.units.n_units, kThreads, 0, s>>>(a);
  return cudaGetLastError();
}

template <int OP>
static cudaError_t launch_ragged_op(int dtype, const ElemArgs &a, cudaStream_t s) {
  return dtype == COPES_BF16 ? launch_ragged_typed<OP, __nv_bfloat16>(a, s) : launch_ragged_typed<OP, float>(a, s);
}

cudaError_t launch_elem_ragged(int op, int dtype, const ElemArgs &a, cudaStream_t s) {
  switch (op) {
    case kOpPerturb: return launch_ragged_op<kOpPerturb>(dtype, a, s);
    case kOpPerturbPair: return launch_ragged_op<kOpPerturbPair>(dtype, a, s);
    case kOpPerturbTwoPairs: return launch_ragged_op<kOpPerturbTwoPairs>(dtype, a, s);
    case kOpInit: return launch_ragged_op<kOpInit>(dtype, a, s);
    default: return cudaErrorInvalidValue;
  }
}

unsigned read_and_clear_ragged_errors() {
  unsigned v = 0, zero = 0;
  cudaMemcpyFromSymbol(&v, g_ragged_error, sizeof(v));
  if (v) cudaMemcpyToSymbol(g_ragged_error, &zero, sizeof(zero));
  return v;
}

}  // namespace copes
