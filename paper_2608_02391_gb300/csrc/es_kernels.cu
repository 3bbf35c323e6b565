// Elementwise ES kernels: perturb (Eq. 8), restore / context commit (Supp. A.8), the
// fused reward-weighted update (Eq. 6 / Eq. 13) and the synthetic initialiser, over
// TILES subspaces (vectorised, 4-element groups = one Philox counter) and INDICES
// subspaces (gather / scatter through a sorted int64 list).
#include <cuda_bf16.h>

#include "copes_device.cuh"
#include "copes_internal.h"
#include "elem_ops.cuh"
#include "es_common.cuh"

namespace copes {

__device__ unsigned int g_es_error = 0;

__device__ __forceinline__ void flag_error(unsigned bit) { atomicOr(&g_es_error, bit); }

// ------------------------------------------------------------ perturb / restore / init
template <int OP>
constexpr uint32_t op_tag() { return OP == kOpInit ? COPES_TAG_INIT : COPES_TAG_NOISE; }

// The two pairs' bf16 step by octets: G / 2 runs of two adjacent groups a thread, at
// b + off + 8 kThreads i, each with one 32-byte load and one 16-byte store a value where
// elem_step has two of half the size: fewer memory instructions in a launch bound by its issue
// slots.  2^28 elements take 510 us instead of 523 (518 with a product M0 q for each group,
// where the second is the first's plus M0).  The pair and the perturb (320 -> 311 and 258 -> 257
// us, but 8.01 -> 8.08 and 7.4 -> 8.4 of 4M elements) keep elem_step, as do elem_part's units
// (10.1 -> 11.0 us of 3M elements with octets).
template <int G>
__device__ __forceinline__ void two_pairs_octets(const ElemArgs &a, const WideTable &tab, uint64_t b, uint32_t off) {
  constexpr int OP = kOpPerturbTwoPairs, H = G / 2;
  const float *__restrict__ mt = a.master + b;
  float th[G][4];
#pragma unroll
  for (int i = 0; i < H; ++i) ld_stream_f8(mt + off + 8u * kThreads * i, th[2 * i], th[2 * i + 1]);
  uint32_t w[2 * G][4];
  const uint32_t q0 = (uint32_t)(b >> 2);
#pragma unroll
  for (int i = 0; i < H; ++i) {
    uint64_t m = (uint64_t)kPhiloxM0 * (q0 + ((off >> 2) + 2 * kThreads * i));
#pragma unroll
    for (int h = 0; h < 2; ++h, m += kPhiloxM0) {
      philox4x32_10_folded((uint32_t)m, (uint32_t)(m >> 32), a.fk, w[4 * i + 2 * h]);
      philox4x32_10_folded((uint32_t)m, (uint32_t)(m >> 32), a.fk_b, w[4 * i + 2 * h + 1]);
    }
  }
  unsigned long long e2[2 * G][2];
  normals_packed<2 * G>(w, tab, e2);
#pragma unroll
  for (int i = 0; i < H; ++i) {
    const uint64_t g = b + off + 8u * kThreads * i;
    float v[2][4][4];
#pragma unroll
    for (int h = 0; h < 2; ++h) group_values<OP>(a, &e2[2 * (2 * i + h)], th[2 * i + h], v[h]);
#pragma unroll
    for (int m = 0; m < 4; ++m)
      __stcs(reinterpret_cast<uint4 *>(reinterpret_cast<uint16_t *>(m == 0 ? a.w : a.copies.p[m - 1]) + g),
             make_uint4(pack_bf16x2(v[0][m][0], v[0][m][1]), pack_bf16x2(v[0][m][2], v[0][m][3]),
                        pack_bf16x2(v[1][m][0], v[1][m][1]), pack_bf16x2(v[1][m][2], v[1][m][3])));
  }
}

// Whether an octet at b starts on 32 bytes of theta and 16 of each buffer.  (The addresses
// themselves: the same answer from b and the bases, 524 us for 512 of 2^28 elements, is
// compiled to a slower loop.)
__device__ __forceinline__ bool octets_aligned(const ElemArgs &a, uint64_t b) {
  uintptr_t w = reinterpret_cast<uintptr_t>(reinterpret_cast<uint16_t *>(a.w) + b);
#pragma unroll
  for (int m = 0; m < 3; ++m) w |= reinterpret_cast<uintptr_t>(reinterpret_cast<uint16_t *>(a.copies.p[m]) + b);
  return ((reinterpret_cast<uintptr_t>(a.master + b) | w << 1 | b * 4) & 31) == 0;
}

// The default tile, with every bound a compile-time constant (a runtime bound spilled
// registers and cost the two-pairs perturb 5%).
constexpr uint32_t kElemSpan = 16384;

template <int OP, typename WT, int G>
__device__ __forceinline__ void elem_span(const ElemArgs &a, const WideTable &tab, uint64_t b, NextUnit &next) {
  constexpr uint32_t kStep = 4u * kThreads * G;
  static_assert(kElemSpan % kStep == 0, "a span is whole steps");
  if constexpr (OP == kOpPerturbTwoPairs && sizeof(WT) == 2) {
    if (octets_aligned(a, b)) {
      for (uint32_t at = 0; at < kElemSpan; at += kStep) {
        if (at == kElemSpan - kStep) next.ask();
        two_pairs_octets<G>(a, tab, b, at + 8u * threadIdx.x);
      }
      return;
    }
  }
  for (uint32_t at = 0; at < kElemSpan; at += kStep) {
    if (at == kElemSpan - kStep) next.ask();
    elem_step<OP, WT, G>(a, LowKeys{}, tab, b, at + 4u * threadIdx.x);
  }
}

// n elements from b, whole groups (b and n multiples of 4), counters below 2^32: steps of G
// groups while more than half of one is left, then of single groups, so that little is
// generated for nobody.
template <int OP, typename WT, int G>
__device__ __forceinline__ void elem_range(const ElemArgs &a, const WideTable &tab, uint64_t b, uint32_t n,
                                           NextUnit &next) {
  constexpr uint32_t kStep = 4u * kThreads * G;
  uint32_t at = 0;
  for (; at + kStep / 2 < n; at += kStep) {
    if (at + kStep + kStep / 2 >= n) next.ask();
    elem_step<OP, WT, G, true>(a, LowKeys{}, tab, b, at + 4u * threadIdx.x, 0, n);
  }
  for (uint32_t off = at + 4u * threadIdx.x; off < n; off += 4u * kThreads) elem_step<OP, WT, 1>(a, LowKeys{}, tab, b, off);
}

// A stretch of less than a group a thread.  Out of line for the sake of the forms above: beside it
// they are compiled to faster code than without it (two pairs of 4M elements 12.2 / 12.8 us).
template <int OP, typename WT>
__device__ __noinline__ void elem_small(const ElemArgs &a, const WideTable &tab, uint64_t b, uint32_t n) {
  for (uint32_t off = 4u * threadIdx.x; off < n; off += 4u * kThreads) elem_step<OP, WT, 1>(a, LowKeys{}, tab, b, off);
}

// The elements [b, e): the whole groups by the block, a group cut by either end by one thread
// (of the last warps, which have the least of a ragged tile).
template <int OP, typename WT, int G>
__device__ __forceinline__ void elem_stretch(const ElemArgs &a, const WideTable &tab, uint64_t b, uint64_t e,
                                             NextUnit &next) {
  const uint64_t lo = (b + 3) & ~3ull, hi = e & ~3ull;  // the whole groups, if lo < hi
  if (lo != b && threadIdx.x == kThreads - 1) elem_partial_group<OP, WT>(a, LowKeys{}, tab, b, min(lo, e));
  if (hi != e && hi >= lo && threadIdx.x == kThreads - 33) elem_partial_group<OP, WT>(a, LowKeys{}, tab, hi, e);
  if (lo >= hi) return;
  if (hi - lo < 4 * kThreads) elem_small<OP, WT>(a, tab, lo, (uint32_t)(hi - lo));
  else if (hi - lo == kElemSpan) elem_span<OP, WT, G>(a, tab, lo, next);
  else elem_range<OP, WT, G>(a, tab, lo, (uint32_t)(hi - lo), next);
}

// Groups per thread step, at 4 blocks of 256 threads per SM (64 registers).  Measured with
// 16,384-element tiles on 2^28 elements (bf16; probe): the two-pairs perturb 2 groups
// 0.509 ms, 1 group at 5 blocks 0.542 ms, 2 groups at 3 blocks 0.551 ms; the pair 4 groups
// 0.311 ms, 2 groups at 5 or 6 blocks 0.320 and 0.314 ms.  At 64 registers these kernels spill 20 to
// 84 bytes a thread (most for the bf16 two pairs): about one local load a step of 16 normals and
// 400 instructions, from L1; 3 blocks, which need none, are the slower.
template <int OP>
constexpr int elem_groups() { return OP == kOpPerturbTwoPairs ? 2 : 4; }

// A tile outside [partner_base, partner_base + partner_len) is skipped and flagged.
__device__ __forceinline__ bool partner_covers(const ElemArgs &a, uint64_t b, uint64_t e) {
  if (b >= a.partner_base && e - a.partner_base <= a.partner_len) return true;
  flag_error(kErrPartnerRange);
  return false;
}

// A unit of exactly kElemPart aligned elements whose counters are below 2^32 (a quarter of the
// default tile, say), every bound a compile-time constant; false when unit `unit` is not
// one.  Short launches are cut into such units: 4.5 us for a two-pairs perturb of 2^20
// elements against 5.1 us through the general path below.
constexpr uint32_t kElemPart = 4096;

template <int OP, typename WT, int G>
__device__ __forceinline__ bool elem_part(const ElemArgs &a, const WideTable &tab, uint32_t unit, NextUnit &next) {
  const uint32_t lp = a.units.log_parts;
  if (a.units.run != 1) return false;
  const ulonglong2 v = __ldg(reinterpret_cast<const ulonglong2 *>(a.tiles) + (unit >> lp));
  if (!tile_in_whole_parts(v.x, v.y, a.n_alloc, kElemPart, lp)) return false;
  if (OP == kOpPerturbPair && !(v.x >= a.partner_base && v.y - a.partner_base <= a.partner_len)) return false;
  next.ask();
  const uint64_t b = v.x + (unit - (unit >> lp << lp)) * kElemPart;
#pragma unroll
  for (uint32_t at = 0; at < kElemPart; at += 4u * kThreads * G)
    elem_step<OP, WT, G>(a, LowKeys{}, tab, b, at + 4u * threadIdx.x);
  return true;
}

template <int OP, typename WT, int G>
__global__ void __launch_bounds__(kThreads, 4) elem_tiles_kernel(const __grid_constant__ ElemArgs a) {
  __shared__ __align__(128) float4 s_tab[WideTable::kFloat4s];
  __shared__ UnitSmem s_unit;
  if (threadIdx.x == 0) units_init(s_unit);
  // worth it where the first units are much of the launch: 4M elements 8.03 -> 7.54 us (perturb)
  if (OP != kOpInit && threadIdx.x == kThreads - 1 && (a.units.log_parts || a.units.n_units <= kUnitsResident))
    prefetch_unit(a.units, a.tiles, a.n_alloc, a.master);
  WideTable::fill(s_tab);
  __syncthreads();
  const WideTable tab(s_tab);
  for_units(s_unit, a.units, flag_error, [&](uint32_t unit, NextUnit &next) {
    if (elem_part<OP, WT, G>(a, tab, unit, next)) return;
    for_unit(unit, a.units, a.tiles, a.n_tiles, a.n_alloc, flag_error,
             [&](uint64_t b, uint64_t e) { return OP != kOpPerturbPair || partner_covers(a, b, e); },
             [&](uint64_t b, uint64_t e) { elem_stretch<OP, WT, G>(a, tab, b, e, next); });
  });
}

// Restore / commit over TILES: v = theta, to every working copy.  G groups per thread step,
// their loads in flight together, at 3 blocks per SM (8 groups: 104-107% of the copy rate
// on 16,384-element tiles).  Without a prologue one block per unit is as good.
template <typename WT, int G>
__global__ void __launch_bounds__(kThreads, 3) restore_tiles_kernel(const __grid_constant__ ElemArgs a) {
  for_unit(blockIdx.x, a.units, a.tiles, a.n_tiles, a.n_alloc, flag_error, [](uint64_t, uint64_t) { return true; },
           [&](uint64_t b, uint64_t e) {
    // whole groups from a sector's start on (from an odd begin, 134M elements to four copies 274 ->
    // 236 us), and up to 15 elements before them and 3 behind one by one
    const uint64_t lo = (b + 15) & ~15ull, hi = e & ~3ull;
    const uint64_t edge = threadIdx.x < 16 ? b + threadIdx.x : hi + threadIdx.x - 16;
    const bool has_edge = threadIdx.x < 20 && edge < e && (threadIdx.x < 16 ? edge < lo : hi >= lo);
    const float edge_v = has_edge ? a.master[edge] : 0.0f;
    const float *__restrict__ mt = a.master + lo;
    const uint32_t n = lo < hi ? (uint32_t)(hi - lo) : 0u;
    for (uint32_t off = 4u * threadIdx.x; off < n; off += 4u * kThreads * G) {
      float4 th[G];
#pragma unroll
      for (int i = 0; i < G; ++i)
        if (off + 4u * kThreads * i < n) th[i] = ld_stream_f4(mt + off + 4u * kThreads * i);
#pragma unroll
      for (int i = 0; i < G; ++i) {
        const uint32_t o = off + 4u * kThreads * i;
        if (o >= n) continue;
        const float v[4] = {th[i].x, th[i].y, th[i].z, th[i].w};
        WStore<WT>::full(a.w, lo + o, v);
        store_copies_full<WT>(a.copies, lo + o, v);
      }
    }
    if (has_edge) {
      WStore<WT>::one(a.w, edge, edge_v);
      store_copies_one<WT>(a.copies, edge, edge_v);
    }
  });
}

// The partner member's perturb over TILES: w[g] = partner[g - partner_base], a copy of
// the working dtype's bits (the values kOpPerturbPair wrote), by whole 4-element groups (8 B
// bf16, 16 B fp32); partner_base is a multiple of 4, so both sides' groups are aligned.
template <typename WT>
struct Group4;
template <>
struct Group4<__nv_bfloat16> {
  using T = uint2;
};
template <>
struct Group4<float> {
  using T = uint4;
};

template <typename WT, int G>
__global__ void __launch_bounds__(kThreads) partner_tiles_kernel(const __grid_constant__ ElemArgs a) {
  for_unit(blockIdx.x, a.units, a.tiles, a.n_tiles, a.n_alloc, flag_error,
           [&](uint64_t b, uint64_t e) { return partner_covers(a, b, e); }, [&](uint64_t b, uint64_t e) {
    const uint64_t lo = (b + 3) & ~3ull, hi = e & ~3ull;  // the whole groups, if lo < hi
    const WT *__restrict__ src = reinterpret_cast<const WT *>(a.partner);
    WT *__restrict__ dst = reinterpret_cast<WT *>(a.w);
    const uint64_t edge = threadIdx.x < 4 ? b + threadIdx.x : hi + threadIdx.x - 4;
    if (threadIdx.x < 8 && edge < e && (threadIdx.x < 4 ? edge < lo : hi >= lo)) dst[edge] = src[edge - a.partner_base];
    if (lo >= hi) return;
    using V = typename Group4<WT>::T;
    const V *__restrict__ vs = reinterpret_cast<const V *>(src + (lo - a.partner_base));
    V *__restrict__ vd = reinterpret_cast<V *>(dst + lo);
    const uint32_t n = (uint32_t)(hi - lo) / 4;
    for (uint32_t i0 = threadIdx.x; i0 < n; i0 += kThreads * G) {
      V v[G];
#pragma unroll
      for (int k = 0; k < G; ++k)
        if (i0 + kThreads * k < n) v[k] = __ldcs(vs + i0 + kThreads * k);
#pragma unroll
      for (int k = 0; k < G; ++k)
        if (i0 + kThreads * k < n) __stcs(vd + i0 + kThreads * k, v[k]);
    }
  });
}

// Gather form: the block's segment of the sorted index list is staged into shared memory
// chunk by chunk (TMA bulk copies, double-buffered); each thread then handles its indices
// of the chunk: load theta[g], one Philox word's normal, store w[g] (and theta[g] for init).
// GATH: theta lives in the subspace's gathered copy at the index's list position p
// (a.gathered[p]) instead of master[g]; kOpGather / kOpScatter copy between the two.
template <int OP, typename WT, bool GATH>
__global__ void __launch_bounds__(kThreads) elem_index_kernel(const __grid_constant__ ElemArgs a) {
  constexpr bool kNoise = OP == kOpPerturb || OP == kOpPerturbPair || OP == kOpInit;
  __shared__ __align__(128) int64_t s_idx[2][kStageChunk];
  __shared__ __align__(128) float4 s_tab[kNoise ? SlimTable::kFloat4s : 1];
  __shared__ __align__(8) uint64_t s_bar[2];
  if (kNoise) {
    SlimTable::fill(s_tab);
    __syncthreads();
  }
  const SlimTable tab(s_tab);
  constexpr int U = kStageChunk / kThreads;
  const uint64_t s0 = (uint64_t)blockIdx.x * a.segment;
  const uint64_t s1 = min(s0 + a.segment, a.n_index);
  float *__restrict__ master = a.master;
  float *__restrict__ gath = a.gathered;
  staged_index_segment(a.index, s0, s1, s_idx, s_bar, [] { flag_error(kErrStageTimeout); },
                       [&](const int64_t *chunk, int cnt, uint64_t first) {
    int64_t g[U];
    float th[U];
    bool ok[U];
#pragma unroll
    for (int u = 0; u < U; ++u) {
      const int p = threadIdx.x + kThreads * u;
      ok[u] = p < cnt;
      g[u] = ok[u] ? chunk[p] : 0;
      if (ok[u] && (g[u] < 0 || (uint64_t)g[u] >= a.n_alloc)) {
        flag_error(kErrIndexRange);
        ok[u] = false;
      }
      if ((OP == kOpPerturbPair || OP == kOpPartner) && ok[u] &&
          ((uint64_t)g[u] < a.partner_base || (uint64_t)g[u] - a.partner_base >= a.partner_len)) {
        flag_error(kErrPartnerRange);
        ok[u] = false;
      }
      const bool from_gathered = GATH && OP != kOpGather;
      const bool reads_theta = OP != kOpInit && OP != kOpPartner;
      th[u] = (reads_theta && ok[u]) ? (from_gathered ? gath[first + p] : master[g[u]]) : 0.0f;
    }
#pragma unroll
    for (int u = 0; u < U; ++u) {
      if (!ok[u]) continue;
      if constexpr (OP == kOpGather) {
        gath[first + threadIdx.x + kThreads * u] = th[u];
        continue;
      } else if constexpr (OP == kOpScatter) {
        master[g[u]] = th[u];
        continue;
      } else if constexpr (OP == kOpPartner) {
        const uint64_t gi = (uint64_t)g[u];
        reinterpret_cast<WT *>(a.w)[gi] = reinterpret_cast<const WT *>(a.partner)[gi - a.partner_base];
        continue;
      } else {
        float v, vp = 0.0f;
        if (OP == kOpRestore) {
          v = th[u];
        } else {
          uint32_t x[4];
          const uint64_t q = (uint64_t)g[u] >> 2;
          philox4x32_10_rk((uint32_t)q, (uint32_t)(q >> 32), 0u, op_tag<OP>(), a.rk, x);
          const uint32_t sel = (uint32_t)g[u] & 3u;
          const uint32_t wd = sel == 0 ? x[0] : (sel == 1 ? x[1] : (sel == 2 ? x[2] : x[3]));
          const float eps = normal_from_word(wd, tab);
          v = __fmaf_rn(a.a, eps, OP == kOpInit ? a.b : th[u]);
          if (OP == kOpPerturbPair) vp = __fmaf_rn(-a.a, eps, th[u]);
        }
        if (OP == kOpInit) {
          if (GATH) gath[first + threadIdx.x + kThreads * u] = v;
          else master[g[u]] = v;
        }
        WStore<WT>::one(a.w, (uint64_t)g[u], v);
        if (writes_context<OP>()) store_copies_one<WT>(a.copies, (uint64_t)g[u], v);
        if (OP == kOpPerturbPair) WStore<WT>::one(a.partner, (uint64_t)g[u] - a.partner_base, vp);
      }
    }
  });
}

// Indices per block: whole staging chunks, as many as leave about 8 waves of 4 blocks on each of
// 152 SMs, at most kIndexSegment.
static uint32_t index_segment(uint64_t n_index) {
  const uint64_t chunks = n_index / (8 * 4 * 152) / kStageChunk;
  return (uint32_t)(chunks < 1 ? kStageChunk : (chunks >= kIndexSegment / kStageChunk ? kIndexSegment : chunks * kStageChunk));
}

template <int OP, typename WT>
static cudaError_t launch_elem_typed(int kind, ElemArgs &a, cudaStream_t s) {
  if constexpr (OP != kOpGather && OP != kOpScatter) {
    if (kind == COPES_SUBSPACE_TILES) {
      if (OP == kOpPerturbTwoPairs && a.copies.n != 3) return cudaErrorInvalidValue;
      if (a.n_tiles == 0) return cudaSuccess;
      const TileWork work = tile_work(a.n_tiles, a.n_alloc, a.tile_hint);
      if constexpr (OP == kOpPartner || OP == kOpRestore) {
        a.units = plan_copy(work, OP == kOpPartner ? -1 : a.copies.n, sizeof(WT) == 4);
      } else {
        const NoiseOp op = OP == kOpInit ? NoiseOp::kInit
                                         : (OP == kOpPerturbTwoPairs ? NoiseOp::kTwoPairs
                                                                     : (OP == kOpPerturbPair ? NoiseOp::kPair : NoiseOp::kPerturb));
        const NoisePlan plan = plan_noise(work, a.n_alloc, op, sizeof(WT) == 4);
        a.units = plan.units;
        if (plan.ragged) return launch_elem_ragged(OP, sizeof(WT) == 2 ? COPES_BF16 : COPES_FP32, a, s);
      }
      const unsigned grid = a.units.n_units;
      if constexpr (OP == kOpPartner) partner_tiles_kernel<WT, 8><<<grid, kThreads, 0, s>>>(a);
      else if constexpr (OP == kOpRestore) restore_tiles_kernel<WT, 8><<<grid, kThreads, 0, s>>>(a);
      else elem_tiles_kernel<OP, WT, elem_groups<OP>()><<<grid, kThreads, 0, s>>>(a);
      return cudaGetLastError();
    }
  }
  if constexpr (OP == kOpPerturbTwoPairs) {
    return cudaErrorInvalidValue;  // TILES only
  } else {
    constexpr bool kGatheredOnly = OP == kOpGather || OP == kOpScatter;
    if (kGatheredOnly && (kind != COPES_SUBSPACE_INDICES || !a.gathered)) return cudaErrorInvalidValue;
    if (a.n_index == 0) return cudaSuccess;
    a.segment = index_segment(a.n_index);
    const unsigned blocks = (unsigned)((a.n_index + a.segment - 1) / a.segment);
    if (kGatheredOnly || a.gathered) elem_index_kernel<OP, WT, true><<<blocks, kThreads, 0, s>>>(a);
    else elem_index_kernel<OP, WT, kGatheredOnly><<<blocks, kThreads, 0, s>>>(a);
    return cudaGetLastError();
  }
}

template <int OP>
static cudaError_t launch_elem_op(int kind, int dtype, ElemArgs &a, cudaStream_t s) {
  return dtype == COPES_BF16 ? launch_elem_typed<OP, __nv_bfloat16>(kind, a, s)
                             : launch_elem_typed<OP, float>(kind, a, s);
}

cudaError_t launch_elementwise(int op, int kind, int dtype, ElemArgs &a, cudaStream_t s) {
  switch (op) {
    case kOpPerturb: return launch_elem_op<kOpPerturb>(kind, dtype, a, s);
    case kOpRestore: return launch_elem_op<kOpRestore>(kind, dtype, a, s);
    case kOpGather: return launch_elem_op<kOpGather>(kind, dtype, a, s);
    case kOpScatter: return launch_elem_op<kOpScatter>(kind, dtype, a, s);
    case kOpPerturbPair: return launch_elem_op<kOpPerturbPair>(kind, dtype, a, s);
    case kOpPartner: return launch_elem_op<kOpPartner>(kind, dtype, a, s);
    case kOpPerturbTwoPairs: return launch_elem_op<kOpPerturbTwoPairs>(kind, dtype, a, s);
    default: return launch_elem_op<kOpInit>(kind, dtype, a, s);
  }
}

// ------------------------------------------------------------------------- update
// Every thread regenerates all P noise vectors for its G groups in registers
// (noise_sum_groups), acc = sum_j w_j eps_j (j ascending), and writes theta = fma(coef, acc,
// theta) and, with COMMIT, its rounding to the working copies.  All counters of [b, e) have
// the high word s.q_hi.
template <typename WT, int G, bool COMMIT, bool AHEAD>
__device__ __forceinline__ void update_step(const UpdateArgs &a, const UpdateSmem &s, uint64_t base, uint64_t b,
                                            uint64_t e) {
  float *__restrict__ master = a.master;
  if (AHEAD)
#pragma unroll
    for (int i = 0; i < G; ++i)
      if (base + 4ull * kThreads * i < e) prefetch_l2(master + base + 4ull * kThreads * i);
  float acc[G][4];
  noise_sum_groups<G>(base, a.n_noise, s, acc);
  // theta is read only now, after the noise loop, so it occupies no registers there
#pragma unroll
  for (int i = 0; i < G; ++i) {
    const uint64_t g4 = base + 4ull * kThreads * i;
    if (g4 >= e) continue;
    if (g4 >= b && g4 + 4 <= e) {
      const float4 t = ld_stream_f4(master + g4);
      float v[4] = {__fmaf_rn(a.coef, acc[i][0], t.x), __fmaf_rn(a.coef, acc[i][1], t.y),
                    __fmaf_rn(a.coef, acc[i][2], t.z), __fmaf_rn(a.coef, acc[i][3], t.w)};
      st_stream_f4(master + g4, make_float4(v[0], v[1], v[2], v[3]));
      if (COMMIT) {
        WStore<WT>::full(a.w, g4, v);
        store_copies_full<WT>(a.copies, g4, v);
      }
    } else {
#pragma unroll
      for (int k = 0; k < 4; ++k) {
        const uint64_t g = g4 + k;
        if (g >= b && g < e) {
          const float v = __fmaf_rn(a.coef, acc[i][k], master[g]);
          master[g] = v;
          if (COMMIT) {
            WStore<WT>::one(a.w, g, v);
            store_copies_one<WT>(a.copies, g, v);
          }
        }
      }
    }
  }
}

// Steps of G groups while they are whole for the block, then of single groups.
template <typename WT, int G, bool COMMIT, bool AHEAD>
__device__ __forceinline__ void update_range(const UpdateArgs &a, const UpdateSmem &s, uint64_t b, uint64_t e,
                                             NextUnit &next) {
  constexpr uint64_t kStep = 4ull * kThreads * G;
  uint64_t at = b & ~3ull;
  for (; at + kStep <= e; at += kStep) {
    if (at + 2 * kStep > e) next.ask();
    update_step<WT, G, COMMIT, AHEAD>(a, s, at + 4ull * threadIdx.x, b, e);
  }
  for (uint64_t base = at + 4ull * threadIdx.x; base < e; base += 4ull * kThreads)
    update_step<WT, 1, COMMIT, AHEAD>(a, s, base, b, e);
}

// update_range for exactly kUpdateSpan elements from an aligned b (the default tile size),
// with compile-time bounds and no edge tests: the same values bit for bit.
constexpr uint32_t kUpdateSpan = 16384;

template <typename WT, int G, bool COMMIT, bool AHEAD>
__device__ __forceinline__ void update_span(const UpdateArgs &a, const UpdateSmem &s, uint64_t b, NextUnit &next) {
  constexpr uint32_t kStep = 4u * kThreads * G;
  static_assert(kUpdateSpan % kStep == 0, "a full span is whole steps");
  float *__restrict__ mt = a.master + b;
  for (uint32_t at = 0; at < kUpdateSpan; at += kStep) {
    if (at == kUpdateSpan - kStep) next.ask();
    const uint32_t off = at + 4u * threadIdx.x;
    if (AHEAD)
#pragma unroll
      for (int i = 0; i < G; ++i) {
        const float *t = mt + off + 4u * kThreads * i;
        if (at == 0) prefetch_l2(t);
        if (at + kStep < kUpdateSpan) prefetch_l2(t + kStep);
      }
    float acc[G][4];
    noise_sum_groups<G>(b + off, a.n_noise, s, acc);
#pragma unroll
    for (int i = 0; i < G; ++i) {
      const uint32_t o = off + 4u * kThreads * i;
      const float4 t = ld_stream_f4(mt + o);
      float v[4] = {__fmaf_rn(a.coef, acc[i][0], t.x), __fmaf_rn(a.coef, acc[i][1], t.y),
                    __fmaf_rn(a.coef, acc[i][2], t.z), __fmaf_rn(a.coef, acc[i][3], t.w)};
      st_stream_f4(mt + o, make_float4(v[0], v[1], v[2], v[3]));
      if (COMMIT) {
        WStore<WT>::full(a.w, b + o, v);
        store_copies_full<WT>(a.copies, b + o, v);
      }
    }
  }
}

// Launch shape of the tile update: groups per thread and resident blocks per SM
// (registers: 65536 / (256 x blocks) a thread).  Cycles per warp-normal at P = 16: 2 groups at
// 4 blocks 33.1, at 5 blocks 32.9, at 3 blocks 33.2; 4 groups at 3 blocks 32.9; 1 group at 6
// blocks 34.3.  At 64 registers 48 to 56 bytes a thread spill, outside the noise loop: about one
// local load a step (a warp's 256 elements) whatever P; at 3 blocks none do and it is no faster.
constexpr int kUpdateGroups = 2;
constexpr int kUpdateBlocksPerSM = 4;

// AHEAD: theta is asked into L2 a step ahead of its noise, which costs no registers.  Few noise
// vectors do not hide its latency: 134M elements, P = 1, 2, 4 and 8 355 -> 327, 385 -> 329,
// 522 -> 498 and 946 -> 922 us.  With more it gains nothing (P = 16 1,776 / 1,782), and the form
// without it is the faster code.
constexpr int kAheadNoise = 8;

template <typename WT, int G, bool COMMIT, int BLOCKS, bool AHEAD>
__global__ void __launch_bounds__(kThreads, BLOCKS) update_tiles_kernel(const __grid_constant__ UpdateArgs a) {
  extern __shared__ __align__(128) char s_update[];
  __shared__ UnitSmem s_unit;
  if (threadIdx.x == 0) units_init(s_unit);
  UpdateSmem s = update_prologue(a, s_update);  // ends with __syncthreads
  for_units(s_unit, a.units, flag_error, [&](uint32_t unit, NextUnit &next) {
    for_unit(unit, a.units, a.tiles, a.n_tiles, a.n_alloc, flag_error, [](uint64_t, uint64_t) { return true; },
             [&](uint64_t b, uint64_t e) {
      while (b < e) {  // one pass, two where the counters' high word changes
        const uint64_t end = min(e, ((b >> 34) + 1) << 34);
        update_keys_for(a, s, b);
        if (end - b == kUpdateSpan && (b & 3ull) == 0) update_span<WT, G, COMMIT, AHEAD>(a, s, b, next);
        else update_range<WT, G, COMMIT, AHEAD>(a, s, b, end, next);
        b = end;
      }
    });
  });
}

// Gather form of the update: indices staged through shared memory as in
// elem_index_kernel; every index regenerates the P normals from its own Philox word.
// GATH: theta is read from and written to the gathered copy at the list position.
template <typename WT, bool COMMIT, bool GATH>
__global__ void __launch_bounds__(kThreads) update_index_kernel(const __grid_constant__ UpdateArgs a) {
  extern __shared__ __align__(128) char s_update[];
  __shared__ __align__(128) int64_t s_idx[2][kStageChunk];
  __shared__ __align__(8) uint64_t s_bar[2];
  const GatherSmem s = gather_prologue(a, s_update);  // ends with __syncthreads
  constexpr int U = 2;  // 1.40 ms for 16.8M indices at P = 32; 4 an unrolled step took 1.44 ms
  const uint64_t s0 = (uint64_t)blockIdx.x * a.segment;
  const uint64_t s1 = min(s0 + a.segment, a.n_index);
  float *__restrict__ master = a.master;
  float *__restrict__ gath = a.gathered;
  staged_index_segment(a.index, s0, s1, s_idx, s_bar, [] { flag_error(kErrStageTimeout); },
                       [&](const int64_t *chunk, int cnt, uint64_t first) {
    for (int p0 = threadIdx.x; p0 < cnt; p0 += kThreads * U) {
      int64_t g[U];
      float acc[U];
      bool ok[U];
#pragma unroll
      for (int u = 0; u < U; ++u) {
        const int p = p0 + kThreads * u;
        ok[u] = p < cnt;
        g[u] = ok[u] ? chunk[p] : 0;
        if (ok[u] && (g[u] < 0 || (uint64_t)g[u] >= a.n_alloc)) {
          flag_error(kErrIndexRange);
          ok[u] = false;
        }
      }
      gather_noise_sum(a, s, g, acc);
#pragma unroll
      for (int u = 0; u < U; ++u) {
        if (!ok[u]) continue;
        float *th = GATH ? &gath[first + p0 + kThreads * u] : &master[g[u]];
        const float v = __fmaf_rn(a.coef, acc[u], *th);
        *th = v;
        if (COMMIT) {
          WStore<WT>::one(a.w, (uint64_t)g[u], v);
          store_copies_one<WT>(a.copies, (uint64_t)g[u], v);
        }
      }
    }
  });
}

template <typename WT, bool COMMIT>
static cudaError_t launch_update_typed(int kind, UpdateArgs &a, cudaStream_t s) {
  if (kind == COPES_SUBSPACE_TILES) {
    if (a.n_tiles == 0) return cudaSuccess;
    a.units = plan_update(tile_work(a.n_tiles, a.n_alloc, a.tile_hint), a.n_noise);
    auto kernel = a.n_noise <= kAheadNoise
                      ? update_tiles_kernel<WT, kUpdateGroups, COMMIT, kUpdateBlocksPerSM, true>
                      : update_tiles_kernel<WT, kUpdateGroups, COMMIT, kUpdateBlocksPerSM, false>;
    kernel<<<a.units.n_units, kThreads, update_smem_bytes(a.n_noise), s>>>(a);
  } else {
    if (a.n_index == 0) return cudaSuccess;
    a.segment = index_segment(a.n_index);
    const unsigned blocks = (unsigned)((a.n_index + a.segment - 1) / a.segment);
    const uint32_t smem = gather_smem_bytes(a.n_noise);
    auto kernel = a.gathered ? update_index_kernel<WT, COMMIT, true> : update_index_kernel<WT, COMMIT, false>;
    const cudaError_t e = allow_smem((const void *)kernel, smem + 2 * kStageChunk * 8 + 64, gather_smem_bytes(COPES_MAX_NOISE));
    if (e != cudaSuccess) return e;
    kernel<<<blocks, kThreads, smem, s>>>(a);
  }
  return cudaGetLastError();
}

cudaError_t launch_update(int kind, int dtype, UpdateArgs &a, cudaStream_t s) {
  if (dtype == COPES_BF16)
    return a.fuse_commit ? launch_update_typed<__nv_bfloat16, true>(kind, a, s)
                         : launch_update_typed<__nv_bfloat16, false>(kind, a, s);
  return a.fuse_commit ? launch_update_typed<float, true>(kind, a, s)
                       : launch_update_typed<float, false>(kind, a, s);
}

// -------------------------------------------------------------------------- debug
__global__ void debug_philox_kernel(uint64_t seed, uint64_t q0, uint64_t n, uint32_t aux,
                                    uint32_t tag, uint32_t *out) {
  const uint64_t i = (uint64_t)blockIdx.x * blockDim.x + threadIdx.x;
  if (i >= n) return;
  const uint64_t q = q0 + i;
  uint32_t rk[20], x[4];
  philox_round_keys((uint32_t)seed, (uint32_t)(seed >> 32), rk);
  philox4x32_10_rk((uint32_t)q, (uint32_t)(q >> 32), aux, tag, rk, x);
  reinterpret_cast<uint4 *>(out)[i] = make_uint4(x[0], x[1], x[2], x[3]);
}

__global__ void __launch_bounds__(kThreads) debug_normals_kernel(uint64_t seed, uint32_t tag, uint64_t g0,
                                                                 uint64_t n, float *out) {
  __shared__ __align__(16) float4 s_tab[SlimTable::kFloat4s];
  SlimTable::fill(s_tab);
  __syncthreads();
  const SlimTable tab(s_tab);
  const uint64_t i = (uint64_t)blockIdx.x * blockDim.x + threadIdx.x;
  if (i >= n) return;
  uint32_t x[4];
  const uint64_t q = (g0 + i) >> 2;
  philox4x32_10((uint32_t)q, (uint32_t)(q >> 32), 0u, tag, (uint32_t)seed, (uint32_t)(seed >> 32), x);
  const uint32_t sel = (uint32_t)(g0 + i) & 3u;
  out[i] = normal_from_word(sel == 0 ? x[0] : (sel == 1 ? x[1] : (sel == 2 ? x[2] : x[3])), tab);
}

__global__ void __launch_bounds__(kThreads) debug_transform_kernel(const uint32_t *words, uint64_t n, float *out) {
  __shared__ __align__(16) float4 s_tab[SlimTable::kFloat4s];
  SlimTable::fill(s_tab);
  __syncthreads();
  const SlimTable tab(s_tab);
  const uint64_t i = (uint64_t)blockIdx.x * blockDim.x + threadIdx.x;
  if (i < n) out[i] = normal_from_word(words[i], tab);
}

static unsigned blocks_for(uint64_t n) { return (unsigned)((n + kThreads - 1) / kThreads); }

cudaError_t launch_debug_philox(uint64_t seed, uint64_t q0, uint64_t n, uint32_t aux,
                                uint32_t tag, uint32_t *out, cudaStream_t s) {
  if (n == 0) return cudaSuccess;
  debug_philox_kernel<<<blocks_for(n), kThreads, 0, s>>>(seed, q0, n, aux, tag, out);
  return cudaGetLastError();
}

cudaError_t launch_debug_normals(uint64_t seed, uint32_t tag, uint64_t g0, uint64_t n,
                                 float *out, cudaStream_t s) {
  if (n == 0) return cudaSuccess;
  debug_normals_kernel<<<blocks_for(n), kThreads, 0, s>>>(seed, tag, g0, n, out);
  return cudaGetLastError();
}

cudaError_t launch_debug_transform(const uint32_t *words, uint64_t n, float *out,
                                   cudaStream_t s) {
  if (n == 0) return cudaSuccess;
  debug_transform_kernel<<<blocks_for(n), kThreads, 0, s>>>(words, n, out);
  return cudaGetLastError();
}

unsigned read_and_clear_es_errors() {
  unsigned v = 0, zero = 0;
  cudaMemcpyFromSymbol(&v, g_es_error, sizeof(v));
  if (v) cudaMemcpyToSymbol(g_es_error, &zero, sizeof(zero));
  return v;
}

}  // namespace copes
