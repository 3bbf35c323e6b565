// Device pieces shared by the ES kernels of the tile / gather path (es_kernels.cu), of the
// partition-replay path (replay_kernels.cu) and of the backup mode (backup_kernels.cu): the
// scheduling of tile work, working-weight stores and the update's prologue.
#pragma once

#include <cuda_bf16.h>

#include "copes_device.cuh"
#include "copes_internal.h"

namespace copes {

// ------------------------------------------------------------------------ tile work
// The grid has one block per unit of tile work (TileUnits).  In the kernels with a prologue
// (key schedules, the table) a running block takes over units whose blocks have not started
// yet (cluster launch control): it asks for one while it works on its own, and ends when
// none is left.  So the prologue is paid once per resident block, and the hardware still
// hands the units out one by one, where a static loop over them leaves SMs idle at the end.
// Measured on a two-pairs perturb of 2^28 elements (probe): 0.532 ms static, 0.525 ms one
// unit per block, 0.509 ms taken over.
//
// A block asks at its unit's start, which hides the answer's latency, while more than three
// waves of units are left, and before the last step of its unit after that: asking early
// hands the last units to the blocks that start first, SM by SM, whatever their progress
// (910 units on 608 resident blocks then took 1.23 times as long).  A grid that is resident
// at once has nothing to take over and does not ask.
constexpr uint32_t kUnitsResident = 4 * 152;
constexpr uint32_t kUnitsLate = 3 * kUnitsResident;

struct UnitSmem {
  uint4 response;  // of the request: 16-byte aligned
  uint64_t bar;
};

// Before the kernel's first __syncthreads, by thread 0.
__device__ __forceinline__ void units_init(UnitSmem &s) {
  mbar_init(&s.bar, 1);
  mbar_fence_init();
}

// The request for a block that has not started; the answer completes s.bar's phase.
struct NextUnit {
  UnitSmem &s;
  bool asked;
  __device__ __forceinline__ void ask() {
    if (!asked && threadIdx.x == 0) {
      asm volatile("fence.proxy.async.shared::cta;" ::: "memory");  // the previous answer has been read
      asm volatile("mbarrier.arrive.expect_tx.shared::cta.b64 _, [%0], 16;" ::"r"(smem_addr(&s.bar)) : "memory");
      asm volatile(
          "clusterlaunchcontrol.try_cancel.async.shared::cta.mbarrier::complete_tx::bytes.b128 [%0], [%1];" ::"r"(
              smem_addr(&s.response)),
          "r"(smem_addr(&s.bar))
          : "memory");
    }
    asked = true;
  }
};

// The answer: true and the taken-over unit, or false when no block is left.
__device__ __forceinline__ bool unit_answer(const UnitSmem &s, uint32_t &unit) {
  uint32_t ok, x;
  asm volatile(
      "{\n .reg .b128 r;\n .reg .pred p;\n .reg .b32 y, z, w;\n"
      " ld.shared.b128 r, [%2];\n"
      " clusterlaunchcontrol.query_cancel.is_canceled.pred.b128 p, r;\n"
      " selp.u32 %0, 1, 0, p;\n mov.u32 %1, 0;\n"
      " @p clusterlaunchcontrol.query_cancel.get_first_ctaid.v4.b32.b128 {%1, y, z, w}, r;\n}"
      : "=r"(ok), "=r"(x)
      : "r"(smem_addr(&s.response))
      : "memory");
  unit = x;
  return ok != 0;
}

// Part `part` of the elements [b, e): as many steps as the others to within one, from the group of
// b on; the three elements that a cut group may leave over are the last one's.
__device__ __forceinline__ void tile_part(const TileUnits &u, uint32_t part, uint64_t &b, uint64_t &e) {
  constexpr uint32_t kStep = 4 * kThreads;
  const uint64_t lo = b & ~3ull;
  const uint32_t steps = max(((uint32_t)(e - lo) + kStep - 4) / kStep, 1u);  // of at most COPES_TILE_MAX + 66
  const uint64_t p0 = lo + (part * steps >> u.log_parts) * kStep;
  const uint64_t p1 = lo + ((part + 1) * steps >> u.log_parts) * kStep;
  b = min(max(b, p0), e);
  if (part + 1 != 1u << u.log_parts) e = max(b, min(e, p1));
}

// Runs body(b, e) for the stretches of one unit: the part of its tile, or its run of tiles with
// adjacent ones joined, so that short tiles do not cut the work into short stretches.  Each
// tile is checked first: one outside the arena is flagged and left out, and one for which
// the op's own check(b, e) is false.  The bounds are read again for the body (from L1)
// rather than kept, which would cost the body registers.
template <typename Flag, typename Check, typename Body>
__device__ __forceinline__ void for_unit(uint32_t unit, const TileUnits &u, const uint64_t *tiles, uint64_t n_tiles,
                                         uint64_t n_alloc, Flag flag, Check check, Body body) {
  const uint64_t first = (uint64_t)(unit >> u.log_parts) * u.run;
  const ulonglong2 *tab = reinterpret_cast<const ulonglong2 *>(tiles) + first;
  auto valid = [&](ulonglong2 v, bool reports) {
    if (!tile_in_arena(v.x, v.y, n_alloc)) {
      if (reports) flag(kErrTileRange);
      return false;
    }
    return check(v.x, v.y);
  };
  uint64_t b = 0, e = 0;
  uint32_t left = 0, joined = 0;  // bit i: tile i of the run is to do; it continues tile i - 1
  if (u.run == 1) {
    const ulonglong2 v = __ldg(tab);
    if (!valid(v, threadIdx.x == 0)) return;
    b = v.x, e = v.y;
    if (u.log_parts) tile_part(u, unit & ((1u << u.log_parts) - 1u), b, e);
  } else {
    // lane i looks at tile i of the run, at most 32
    const uint32_t lane = threadIdx.x & 31u;
    ulonglong2 v = make_ulonglong2(0, 0);
    bool ok = false;
    if (lane < (uint32_t)min((uint64_t)u.run, n_tiles - first)) {
      v = __ldg(tab + lane);
      ok = valid(v, threadIdx.x < 32);
    }
    const uint64_t before = __shfl_up_sync(0xffffffffu, v.y, 1);
    left = __ballot_sync(0xffffffffu, ok);
    joined = __ballot_sync(0xffffffffu, ok && lane > 0 && before == v.x) & (left << 1);
    if (!left) return;
  }
  do {
    if (u.run > 1) {
      const uint32_t i = __ffs(left) - 1;
      const uint32_t above = i == 31 ? 0u : joined >> (i + 1);
      const uint32_t j = i + __ffs(~above) - 1;  // the last tile joined to tile i
      left &= j == 31 ? 0u : ~0u << (j + 1);
      b = __ldg(&tab[i].x);
      e = __ldg(&tab[j].y);
    }
    body(b, e);
  } while (left);
}

// Starts the first unit's theta on its way to L2 (one thread), while the block fills its table.
__device__ __forceinline__ void prefetch_unit(const TileUnits &u, const uint64_t *tiles, uint64_t n_alloc,
                                              const float *theta) {
  const ulonglong2 v =
      __ldg(reinterpret_cast<const ulonglong2 *>(tiles) + (uint64_t)(blockIdx.x >> u.log_parts) * u.run);
  uint64_t b = v.x, e = v.y;
  if (!tile_in_arena(b, e, n_alloc)) return;
  if (u.log_parts) tile_part(u, blockIdx.x & ((1u << u.log_parts) - 1u), b, e);
  b &= ~3ull;  // 16-byte aligned; and whole 16 bytes
  const uint32_t bytes = (uint32_t)(e - b) * 4u & ~15u;
  if (e > b && bytes)
    asm volatile("cp.async.bulk.prefetch.L2.global [%0], %1;" ::"l"(theta + b), "r"(bytes) : "memory");
}

// Runs work(unit, next) for the block's unit and the units it takes over; all threads of the
// block take part, and no thread may leave early.  work may call next.ask() before the last
// step of its unit.
template <typename Flag, typename Work>
__device__ __forceinline__ void for_units(UnitSmem &s, const TileUnits &u, Flag flag, Work work) {
  uint32_t unit = blockIdx.x, phase = 0;
  const bool alone = u.n_units <= kUnitsResident;
  while (true) {
    NextUnit next{s, alone};
    if (unit + kUnitsLate < u.n_units) next.ask();
    work(unit, next);
    if (alone) return;
    next.ask();
    if (!mbar_wait_bounded(&s.bar, phase)) {
      if (threadIdx.x == 0) flag(kErrStageTimeout);
      mbar_wait_bounded(&s.bar, phase);  // the answer may still be written to this block's shared memory
      return;
    }
    phase ^= 1;
    const bool more = unit_answer(s, unit);
    __syncthreads();  // every thread has read the answer before the next one overwrites it
    if (!more) return;
  }
}

template <typename WT>
struct WStore;

template <>
struct WStore<__nv_bfloat16> {
  static __device__ __forceinline__ void full(void *w, uint64_t g, const float v[4]) {
    uint2 p;
    p.x = pack_bf16x2(v[0], v[1]);
    p.y = pack_bf16x2(v[2], v[3]);
    st_stream_u2(reinterpret_cast<uint16_t *>(w) + g, p);
  }
  static __device__ __forceinline__ void one(void *w, uint64_t g, float v) {
    reinterpret_cast<uint16_t *>(w)[g] = to_bf16_bits(v);
  }
};

template <>
struct WStore<float> {
  static __device__ __forceinline__ void full(void *w, uint64_t g, const float v[4]) {
    st_stream_f4(reinterpret_cast<float *>(w) + g, make_float4(v[0], v[1], v[2], v[3]));
  }
  static __device__ __forceinline__ void one(void *w, uint64_t g, float v) {
    reinterpret_cast<float *>(w)[g] = v;
  }
};

// The context's stores to the working copies beyond w (restore / commit / init and the
// update's fused commit).
template <typename WT>
__device__ __forceinline__ void store_copies_full(const WorkingCopies &c, uint64_t g, const float v[4]) {
#pragma unroll
  for (int i = 0; i < 3; ++i)
    if (i < c.n) WStore<WT>::full(c.p[i], g, v);
}

template <typename WT>
__device__ __forceinline__ void store_copies_one(const WorkingCopies &c, uint64_t g, float v) {
#pragma unroll
  for (int i = 0; i < 3; ++i)
    if (i < c.n) WStore<WT>::one(c.p[i], g, v);
}

// The weight of noise vector j: the members folded,
//   w_j = sum_{i : noise(i) = j} sign_i f_i  (member order, fp32).
__device__ __forceinline__ float noise_weight(const UpdateArgs &a, int j) {
  float acc = 0.0f;
  for (int m = a.noise_ptr[j]; m < a.noise_ptr[j + 1]; ++m) {
    const int i = a.noise_member[m];
    const float f = a.fitness[i];
    acc = __fadd_rn(acc, a.sign[i] > 0 ? f : -f);
  }
  return acc;
}

// Each noise vector's folded Philox keys for counters whose high word is q_hi (noise tag).
__device__ __forceinline__ void noise_keys_to_smem(const UpdateArgs &a, uint32_t q_hi, uint32_t (*s_fk)[20]) {
  for (int j = threadIdx.x; j < a.n_noise; j += blockDim.x) {
    uint32_t rk[20];
    philox_round_keys(a.seed_lo[j], a.seed_hi[j], rk);
    philox_folded_keys(rk, COPES_TAG_NOISE, s_fk[j], q_hi);
  }
}

// Shared memory of the tile updates (dynamic: 88 bytes per noise vector beside the table).
// s_fk[j] are the keys for q_hi, the high word of the counters of the tiles at hand.
struct UpdateSmem {
  uint32_t (*fk)[20];
  float2 *w;
  WideTable tab;
  uint32_t q_hi;
};

constexpr uint32_t kUpdateSmemBytes = WideTable::kFloat4s * 16;
__host__ __device__ constexpr uint32_t update_smem_bytes(int n_noise) {
  return kUpdateSmemBytes + (uint32_t)n_noise * (20 * 4 + 8);
}

// Fills it for counters below 2^32; ends with a __syncthreads.
__device__ __forceinline__ UpdateSmem update_prologue(const UpdateArgs &a, char *smem) {
  float4 *tab = reinterpret_cast<float4 *>(smem);
  uint32_t(*fk)[20] = reinterpret_cast<uint32_t (*)[20]>(smem + kUpdateSmemBytes);
  float2 *w = reinterpret_cast<float2 *>(smem + kUpdateSmemBytes + a.n_noise * 80);
  // the last warps fold the members, the first the keys, while the table is on its way
  WideTable::fill(tab, [&] {
    for (int j = kThreads - 1 - threadIdx.x; j < a.n_noise; j += blockDim.x) {
      const float wj = noise_weight(a, j);
      w[j] = make_float2(wj, wj);
    }
    noise_keys_to_smem(a, 0, fk);
  });
  __syncthreads();
  return UpdateSmem{fk, w, WideTable(tab), 0};
}

// The keys for the counters of the stretch starting at element b (block-uniform).
__device__ __forceinline__ void update_keys_for(const UpdateArgs &a, UpdateSmem &s, uint64_t b) {
  const uint32_t hi = (uint32_t)(b >> 34);
  if (hi == s.q_hi) return;
  __syncthreads();  // every thread is done with the old keys
  noise_keys_to_smem(a, hi, s.fk);
  __syncthreads();
  s.q_hi = hi;
}

// The update's noise sum for the G groups of one thread, the 4-element groups at
// base + 4 kThreads i, whose counters have the high word s.q_hi: acc[i][k] = sum_j w_j
// eps_j[g] over the P noise vectors, j ascending, each term one fp32 fma.  Per noise vector
// the G groups' Philox calls run first (folded, with each group's product M0 * q computed
// once for all noise vectors), then their transforms, then the accumulation, on packed
// fp32 pairs (the values of scalar steps, bit for bit).
template <int G>
__device__ __forceinline__ void noise_sum_groups(uint64_t base, int P, const UpdateSmem &s, float (&acc)[G][4]) {
  unsigned long long acc2[G][2];  // the accumulators of group i as pairs (2p, 2p + 1)
#pragma unroll
  for (int i = 0; i < G; ++i) acc2[i][0] = acc2[i][1] = 0ull;
  const uint32_t q_lo = (uint32_t)(base >> 2);  // counter of group 0
  uint32_t m0_lo[G], m0_hi[G];                  // M0 * counter of each group
#pragma unroll
  for (int i = 0; i < G; ++i) {
    const uint64_t m = (uint64_t)kPhiloxM0 * (q_lo + kThreads * i);
    m0_lo[i] = (uint32_t)m;
    m0_hi[i] = (uint32_t)(m >> 32);
  }
  for (int j = 0; j < P; ++j) {
    uint32_t k[20];
#pragma unroll
    for (int r = 0; r < 20; r += 4) {
      const uint4 v = *reinterpret_cast<const uint4 *>(s.fk[j] + r);
      k[r] = v.x, k[r + 1] = v.y, k[r + 2] = v.z, k[r + 3] = v.w;
    }
    const float2 wj = s.w[j];
    const unsigned long long w2 = pack_f32x2(wj.x, wj.y);
    uint32_t w[G][4];
#pragma unroll
    for (int i = 0; i < G; ++i) philox4x32_10_folded(m0_lo[i], m0_hi[i], k, w[i]);
    unsigned long long e2[G][2];
    normals_packed<G>(w, s.tab, e2);
#pragma unroll
    for (int i = 0; i < G; ++i)
#pragma unroll
      for (int p = 0; p < 2; ++p) acc2[i][p] = fma_f32x2(w2, e2[i][p], acc2[i][p]);
  }
#pragma unroll
  for (int i = 0; i < G; ++i) {
    unpack_f32x2(acc2[i][0], acc[i][0], acc[i][1]);
    unpack_f32x2(acc2[i][1], acc[i][2], acc[i][3]);
  }
}

// Shared memory of the gather updates (index lists and replay), whose elements may lie
// anywhere: each noise vector's keys (philox_word_keys) with its weight in their free slot.
struct GatherSmem {
  const uint32_t (*row)[20];
  WideTable tab;
  bool high;  // the arena has counters past 2^32
};

constexpr uint32_t gather_smem_bytes(int n_noise) { return kUpdateSmemBytes + (uint32_t)n_noise * 80; }

// Ends with a __syncthreads.
__device__ __forceinline__ GatherSmem gather_prologue(const UpdateArgs &a, char *smem) {
  float4 *tab = reinterpret_cast<float4 *>(smem);
  uint32_t(*row)[20] = reinterpret_cast<uint32_t (*)[20]>(smem + kUpdateSmemBytes);
  WideTable::fill(tab);
  for (int j = threadIdx.x; j < a.n_noise; j += blockDim.x) {
    uint32_t rk[20];
    philox_round_keys(a.seed_lo[j], a.seed_hi[j], rk);
    philox_word_keys(rk, COPES_TAG_NOISE, row[j]);
    row[j][15] = __float_as_uint(noise_weight(a, j));
  }
  __syncthreads();
  return GatherSmem{row, WideTable(tab), a.n_alloc > (1ull << 34)};
}

// sum_j w_j eps_j[g] for any counter (q, q_hi): q_hi only enters the folded keys u[2] and u[3]
// (philox_folded_keys), which are formed here for each element.  Out of line, so that it takes
// no registers from the form for counters below 2^32.
static __device__ __noinline__ float gather_noise_sum_high(const UpdateArgs &a, const GatherSmem &s, uint64_t g) {
  const uint64_t m = (uint64_t)kPhiloxM0 * (uint32_t)(g >> 2);
  const bool h = (uint32_t)g & 2u, odd = (uint32_t)g & 1u;
  float acc = 0.0f;
  for (int j = 0; j < a.n_noise; ++j) {
    uint32_t k[16];
#pragma unroll
    for (int r = 0; r < 16; r += 4) {
      const uint4 v = *reinterpret_cast<const uint4 *>(&s.row[j][r]);
      k[r] = v.x, k[r + 1] = v.y, k[r + 2] = v.z, k[r + 3] = v.w;
    }
    const uint64_t mk = (uint64_t)kPhiloxM0 * (a.seed_lo[j] ^ (uint32_t)(g >> 34));
    k[2] = (uint32_t)(mk >> 32) ^ (a.seed_hi[j] + kPhiloxW1);     // round key 3
    k[3] = (uint32_t)mk ^ (a.seed_hi[j] + 2u * kPhiloxW1);        // round key 5
    const uint2 last = *reinterpret_cast<const uint2 *>(&s.row[j][h ? 18 : 16]);
    const uint32_t wd = philox4x32_10_word((uint32_t)m, (uint32_t)(m >> 32), k, h, odd, last.x, last.y);
    acc = __fmaf_rn(__uint_as_float(k[15]), normal_from_word(wd, s.tab), acc);
  }
  return acc;
}

// acc[u] = sum_j w_j eps_j[g[u]] (j ascending, one fp32 fma a term) for a thread's U elements.
// An element takes one word of its Philox block, so the words are bound by the multiplies
// of a whole call: 15 and a half of 20 are left (philox4x32_10_word), the counter's product
// once for all noise vectors.  16.8M elements, P = 32: 1.73 -> 1.40 ms.
template <int U, typename Index>
__device__ __forceinline__ void gather_noise_sum(const UpdateArgs &a, const GatherSmem &s, const Index (&g)[U],
                                                 float (&acc)[U]) {
  static_assert(U % 2 == 0, "normals are paired");
  if (s.high) {
#pragma unroll
    for (int u = 0; u < U; ++u) acc[u] = gather_noise_sum_high(a, s, (uint64_t)g[u]);
    return;
  }
  uint32_t m0_lo[U], m0_hi[U];
#pragma unroll
  for (int u = 0; u < U; ++u) {
    const uint64_t m = (uint64_t)kPhiloxM0 * (uint32_t)((uint64_t)g[u] >> 2);
    m0_lo[u] = (uint32_t)m;
    m0_hi[u] = (uint32_t)(m >> 32);
    acc[u] = 0.0f;
  }
  for (int j = 0; j < a.n_noise; ++j) {
    uint32_t k[16];
#pragma unroll
    for (int r = 0; r < 16; r += 4) {
      const uint4 v = *reinterpret_cast<const uint4 *>(&s.row[j][r]);
      k[r] = v.x, k[r + 1] = v.y, k[r + 2] = v.z, k[r + 3] = v.w;
    }
    uint32_t wd[U];
#pragma unroll
    for (int u = 0; u < U; ++u) {
      const bool h = (uint32_t)g[u] & 2u, odd = (uint32_t)g[u] & 1u;
      const uint2 last = *reinterpret_cast<const uint2 *>(&s.row[j][h ? 18 : 16]);
      wd[u] = philox4x32_10_word(m0_lo[u], m0_hi[u], k, h, odd, last.x, last.y);
    }
    const float wj = __uint_as_float(k[15]);
#pragma unroll
    for (int u = 0; u < U; u += 2) {  // two normals as one packed pair (bit-identical to one at a time)
      float e0, e1;
      unpack_f32x2(normal_pair(wd[u], wd[u + 1], s.tab), e0, e1);
      acc[u] = __fmaf_rn(wj, e0, acc[u]);
      acc[u + 1] = __fmaf_rn(wj, e1, acc[u + 1]);
    }
  }
}

}  // namespace copes
