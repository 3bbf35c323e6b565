// Partition replay (Supp. A.8 "Partition Replay"; Eq. 7): the ES kernels over subspace k
// of the hash partition (K, seed) with membership recomputed from the partition seed, not
// read from a stored index list.  Each block takes 1 to 4 consecutive 16,384-element hash
// tiles; each warp streams through its 2,048-element stretch of every tile (replay_stream):
//  - it hashes 32 four-element groups at a time -- one Philox4x32-10 call per group at
//    counter (e >> 2, tensor id, TAG_PARTITION), bucket floor(x K / 2^32) per word, or,
//    when the subspace carries a membership mask built once per visit, reads their bits --
//    and appends the members of subspace k to its shared-memory buffer;
//  - whenever the buffer holds a full batch, the warp processes it one member per lane,
//    exactly as the gather kernels process an index list: perturb / restore / commit /
//    init, or the fused update regenerating the P normals of each element.
// Every element's arithmetic is that of the gather path, so the results are identical to
// those over the INDICES list of (K, seed, k).
#include <type_traits>

#include "es_common.cuh"

namespace copes {

__device__ unsigned int g_replay_error = 0;

__device__ __forceinline__ void replay_flag(unsigned bit) { atomicOr(&g_replay_error, bit); }

constexpr int kReplayTile = (int)kHashTile;  // elements per hash tile
constexpr int kReplayTilesPerBlock = 4;      // consecutive hash tiles per block, at most
static_assert(kReplayTile % 4 == 0 && kReplayTile <= 65536, "tile offsets fit 16 bits");
constexpr int kReplayWarpGroups = kReplayTile / 4 / (kThreads / 32);  // groups per warp per tile
constexpr int kReplayIters = kReplayWarpGroups / 32;                  // 32 groups per iteration

constexpr uint64_t kMaskWordsPerTile = kReplayTile / 32;  // membership mask: one bit per element

struct ReplayTile {
  uint64_t g0;        // global index of the tile's first element
  uint64_t q0;        // partition counter of the tile's first group (tensor-local e >> 2)
  uint32_t len;       // elements in the tile (0: skip the tile)
  uint32_t tensor_id;
};

// Hash tile `tile`: its tensor comes from the table's tile map; every thread reads the
// same entries (cached broadcasts), so the result is block-uniform.  A tile the table
// maps outside its tensor or past the arena is skipped and flagged.
__device__ __forceinline__ ReplayTile replay_tile(const ReplayArgs &r, uint64_t n_alloc, uint64_t tile) {
  ReplayTile t{};
  const uint32_t ti = r.tile_tensor[tile];
  if (ti >= (uint32_t)r.n_tensors) {
    if (threadIdx.x == 0) replay_flag(kErrPartition);
    return t;
  }
  const HashTensor T = r.table[ti];
  const uint64_t e0 = (tile - T.tile_begin) * (uint64_t)kReplayTile;
  if (tile < T.tile_begin || e0 >= T.numel) {
    if (threadIdx.x == 0) replay_flag(kErrPartition);
    return t;
  }
  const uint32_t len = (uint32_t)min((uint64_t)kReplayTile, T.numel - e0);
  const uint64_t g0 = T.offset + e0;
  if (g0 + len > n_alloc || (g0 & 3ull) != 0) {
    if (threadIdx.x == 0) replay_flag(kErrIndexRange);
    return t;
  }
  t.g0 = g0;
  t.q0 = e0 >> 2;
  t.len = len;
  t.tensor_id = T.tensor_id;
  return t;
}

// Warp-streamed replay over the block's hash tiles.  Each warp owns a 2,048-element
// stretch of every tile and walks it 32 groups (one per lane) at a time: it hashes the
// groups, appends the members of subspace r.k to its shared-memory buffer with one ballot
// per word slot, and whenever the buffer holds BATCH members it processes them, BATCH / 32
// per lane, every lane busy, so the hashing (ALU) interleaves with the members' scattered
// loads and stores.  The warps' leftovers (fewer than BATCH each) are pooled and processed
// by the whole block at the end; `flush` then runs once.  Every warp runs the same
// iterations, so the full-warp ballots and shuffles see all 32 lanes.  MASK: membership
// comes from r.mask (non-null) instead of the hash; a compile-time choice, so the hashing
// variant carries no mask code.
template <int BATCH, bool MASK, typename Fn, typename Flush>
__device__ __forceinline__ void replay_stream(const ReplayArgs &r, uint64_t n_alloc, uint32_t *wbuf,
                                              uint64_t (*s_g0)[kReplayTilesPerBlock], uint32_t *pool,
                                              int *pool_n, Fn process, Flush flush) {
  constexpr int U = BATCH / 32;
  const uint32_t lane = threadIdx.x & 31u;
  const uint32_t warp = threadIdx.x >> 5;
  const uint64_t per_block = (r.n_tiles + gridDim.x - 1) / gridDim.x;  // at most what replay_blocks took
  const uint64_t t_first = blockIdx.x * per_block;
  const uint64_t t_end = min(t_first + per_block, r.n_tiles);
  // buffer entries are (tile within the block) << 16 | (offset within the tile); each warp
  // keeps the tiles' first global indices in its own row of s_g0
  uint64_t *wg0 = s_g0[warp];
  auto global = [&](uint32_t e) { return wg0[e >> 16] + (e & 0xFFFFu); };
  const uint32_t lt = (1u << lane) - 1u;  // lanes below this one
  int pending = 0;  // warp-uniform
  // One iteration: the warp hashes 32 groups (128 elements, one group per lane) and
  // appends their members with one ballot per word slot; FULL drops the tile-end check.
  auto iteration = [&](const ReplayTile &t, uint64_t tile, uint32_t tag, uint32_t q_lo0, uint32_t q_hi,
                       uint32_t e, auto full) {
    bool m[4];  // membership of the group's 4 elements
    if constexpr (MASK) {
      const uint32_t nib = r.mask[tile * kMaskWordsPerTile + (e >> 5)] >> (e & 31u);
#pragma unroll
      for (int i = 0; i < 4; ++i) m[i] = (nib >> i) & 1u;
    } else {
      uint32_t x[4];
      philox4x32_10_rk(q_lo0 + (e >> 2), q_hi, t.tensor_id, COPES_TAG_PARTITION, r.rk, x);
#pragma unroll
      for (int i = 0; i < 4; ++i)
        // floor(x K / 2^32) == k  <=>  x - lo <= span in 32-bit unsigned arithmetic
        m[i] = x[i] - r.lo <= r.span && (decltype(full)::value || e + i < t.len);
    }
#pragma unroll
    for (int i = 0; i < 4; ++i) {
      const uint32_t bal = __ballot_sync(0xffffffffu, m[i]);
      if (m[i]) wbuf[pending + __popc(bal & lt)] = tag | (e + i);
      pending += __popc(bal);
    }
    __syncwarp();
    while (pending >= BATCH) {  // take the newest BATCH entries
      uint64_t g[U];
      bool ok[U];
#pragma unroll
      for (int u = 0; u < U; ++u) {
        g[u] = global(wbuf[pending - BATCH + u * 32 + lane]);
        ok[u] = true;
      }
      __syncwarp();  // read before the next append overwrites these slots
      pending -= BATCH;
      process(g, ok);
    }
  };
  for (uint64_t tile = t_first; tile < t_end; ++tile) {
    const ReplayTile t = replay_tile(r, n_alloc, tile);
    const uint32_t tag = (uint32_t)(tile - t_first) << 16;
    // q0 is a multiple of 4096 and the tile has 4096 groups, so q0 + group never carries
    // out of 32 bits
    const uint32_t q_lo0 = (uint32_t)t.q0, q_hi = (uint32_t)(t.q0 >> 32);
    if (lane == 0) wg0[tile - t_first] = t.g0;
    __syncwarp();
    const uint32_t e0 = warp * (4u * kReplayWarpGroups) + 4u * lane;  // this lane's first group
    if (t.len == (uint32_t)kReplayTile) {
      for (int it = 0; it < kReplayIters; ++it)
        iteration(t, tile, tag, q_lo0, q_hi, e0 + 128u * it, std::true_type{});
    } else if (t.len > 0) {
      for (int it = 0; it < kReplayIters; ++it)
        iteration(t, tile, tag, q_lo0, q_hi, e0 + 128u * it, std::false_type{});
    }
  }
  // pool the leftovers and process them with the whole block
  int at = 0;
  if (lane == 0 && pending) at = atomicAdd(pool_n, pending);
  at = __shfl_sync(0xffffffffu, at, 0);
  for (int p = lane; p < pending; p += 32) pool[at + p] = wbuf[p];
  __syncthreads();
  const int n = *pool_n;
  wg0 = s_g0[0];  // every warp recorded the same tiles
  for (int p0 = threadIdx.x; p0 < n; p0 += kThreads * U) {
    uint64_t g[U];
    bool ok[U];
#pragma unroll
    for (int u = 0; u < U; ++u) {
      const int p = p0 + kThreads * u;
      ok[u] = p < n;
      g[u] = ok[u] ? global(pool[p]) : wg0[0];
    }
    process(g, ok);
  }
  flush();
}

template <int OP>
constexpr uint32_t replay_tag() { return OP == kOpInit ? COPES_TAG_INIT : COPES_TAG_NOISE; }

// A member's noise word, for any counter.
template <int OP>
__device__ __forceinline__ uint32_t replay_word(const ElemArgs &a, uint64_t g) {
  uint32_t x[4];
  philox4x32_10_rk((uint32_t)(g >> 2), (uint32_t)(g >> 34), 0u, replay_tag<OP>(), a.rk, x);
  const uint32_t sel = (uint32_t)g & 3u;
  return sel == 0 ? x[0] : (sel == 1 ? x[1] : (sel == 2 ? x[2] : x[3]));
}
template <int OP>
static __device__ __noinline__ uint32_t replay_word_high(const ElemArgs &a, uint64_t g) {
  return replay_word<OP>(a, g);
}

// Perturb / restore / commit / init over the members of the block's hash tiles: BATCH / 32
// members per lane per batch, their master loads issued together.  The hashing variant is
// bound by its instructions: a batch's noise is formed together, from one word of a Philox
// block each (perturb of 16.8M members of 2^28 elements 370 -> 336 us).  The mask variant is
// bound by scattered sectors and keeps fewer registers instead (pair 373 us, 378 with single
// words).
//
// Batches of 128, but 64 for the hashing pair of sparse subspaces: a warp's stretch then has about
// one batch or none, what is left over is processed by the block one or two at a time, and
// more warps fit an SM (38 registers for 56).  Pair of 200M elements, 128 / 64: bf16 K = 2 615 /
// 636 us, K = 4 420 / 426, K = 16 278 / 275, K = 64 240 / 227; fp32 K = 16 343 / 358, K = 64 242 / 227.
// The pool's places that hold no member form no noise, where the test costs no more than it
// saves: not in the fp32 pair of dense subspaces and in init (45M, K = 2: 172 / 179 and 160 / 173).
template <typename WT>
constexpr int sparse_k() { return sizeof(WT) == 2 ? 16 : 32; }

template <int OP, typename WT, bool MASK, int BATCH>
__global__ void __launch_bounds__(kThreads) replay_elem_kernel(const __grid_constant__ ElemArgs a,
                                                               const __grid_constant__ ReplayArgs r) {
  constexpr int U = BATCH / 32;
  __shared__ uint32_t s_buf[kThreads / 32][BATCH + 128];
  __shared__ uint32_t s_pool[(kThreads / 32) * BATCH];
  __shared__ uint64_t s_g0[kThreads / 32][kReplayTilesPerBlock];
  __shared__ int s_pool_n;
  constexpr bool kNoise = OP != kOpRestore && OP != kOpPartner;
  constexpr bool kSkip = OP == kOpPerturb || (OP == kOpPerturbPair && (BATCH == 64 || sizeof(WT) == 2));
  __shared__ __align__(16) float4 s_tab[kNoise ? SlimTable::kFloat4s : 1];
  if (threadIdx.x == 0) s_pool_n = 0;
  if (kNoise) SlimTable::fill(s_tab);
  __syncthreads();
  const SlimTable tab(s_tab);
  float *__restrict__ master = a.master;
  replay_stream<BATCH, MASK>(r, a.n_alloc, s_buf[threadIdx.x >> 5], s_g0, s_pool, &s_pool_n,
                             [&](const uint64_t (&g)[U], const bool (&ok_in)[U]) {
    bool ok[U];
    float th[U];
    WT partner[U];  // of the partner copy: all loads before the first store
#pragma unroll
    for (int u = 0; u < U; ++u) {
      ok[u] = ok_in[u];
      if ((OP == kOpPerturbPair || OP == kOpPartner) && ok[u] &&
          (g[u] < a.partner_base || g[u] - a.partner_base >= a.partner_len)) {
        replay_flag(kErrPartnerRange);
        ok[u] = false;
      }
      th[u] = (OP != kOpInit && OP != kOpPartner && ok[u]) ? master[g[u]] : 0.0f;
      if (OP == kOpPartner && ok[u]) partner[u] = reinterpret_cast<const WT *>(a.partner)[g[u] - a.partner_base];
    }
    float eps[U];
    if constexpr (kNoise && !MASK) {
      uint32_t wd[U];
#pragma unroll
      for (int u = 0; u < U; ++u) {
        if (kSkip && !ok_in[u]) continue;  // known when compiled but for the pool
        const uint64_t m = (uint64_t)kPhiloxM0 * (uint32_t)(g[u] >> 2);
        const bool h = (uint32_t)g[u] & 2u, odd = (uint32_t)g[u] & 1u;
        wd[u] = a.n_alloc > 1ull << 34
                    ? replay_word_high<OP>(a, g[u])
                    : philox4x32_10_word((uint32_t)m, (uint32_t)(m >> 32), a.fk, h, odd, h ? a.rk[16] : a.rk[17],
                                         h ? a.rk[19] : a.rk[18]);
      }
#pragma unroll
      for (int u = 0; u < U; u += 2) {
        if (kSkip && !ok_in[u]) continue;  // then u + 1 is not either
        unpack_f32x2(normal_pair(wd[u], !kSkip || ok_in[u + 1] ? wd[u + 1] : 0u, tab), eps[u], eps[u + 1]);
      }
    }
#pragma unroll
    for (int u = 0; u < U; ++u) {
      if (!ok[u]) continue;
      if constexpr (OP == kOpPartner) {
        reinterpret_cast<WT *>(a.w)[g[u]] = partner[u];
        continue;
      }
      float v, vp = 0.0f;
      if constexpr (OP == kOpRestore) {
        v = th[u];
      } else {
        if (MASK) eps[u] = normal_from_word(replay_word<OP>(a, g[u]), tab);
        v = __fmaf_rn(a.a, eps[u], OP == kOpInit ? a.b : th[u]);
        if (OP == kOpPerturbPair) vp = __fmaf_rn(-a.a, eps[u], th[u]);
        if (OP == kOpInit) master[g[u]] = v;
      }
      WStore<WT>::one(a.w, g[u], v);
      if (OP == kOpRestore || OP == kOpInit) store_copies_one<WT>(a.copies, g[u], v);
      if (OP == kOpPerturbPair) WStore<WT>::one(a.partner, g[u] - a.partner_base, vp);
    }
  }, [] {});
}

// The fused update over the members of the block's hash tiles: two members per lane per
// batch, each regenerating the P normals of its element.
template <typename WT, bool COMMIT, bool MASK>
__global__ void __launch_bounds__(kThreads) replay_update_kernel(const __grid_constant__ UpdateArgs a,
                                                                 const __grid_constant__ ReplayArgs r) {
  constexpr int BATCH = 64;
  constexpr int U = BATCH / 32;
  extern __shared__ __align__(128) char s_update[];
  __shared__ uint32_t s_buf[kThreads / 32][BATCH + 128];
  __shared__ uint32_t s_pool[(kThreads / 32) * BATCH];
  __shared__ uint64_t s_g0[kThreads / 32][kReplayTilesPerBlock];
  __shared__ int s_pool_n;
  if (threadIdx.x == 0) s_pool_n = 0;
  const GatherSmem s = gather_prologue(a, s_update);  // ends with __syncthreads
  float *__restrict__ master = a.master;
  replay_stream<BATCH, MASK>(r, a.n_alloc, s_buf[threadIdx.x >> 5], s_g0, s_pool, &s_pool_n,
                             [&](const uint64_t (&g)[U], const bool (&ok)[U]) {
    float acc[U];
    gather_noise_sum(a, s, g, acc);
#pragma unroll
    for (int u = 0; u < U; ++u) {
      if (!ok[u]) continue;
      const float v = __fmaf_rn(a.coef, acc[u], master[g[u]]);
      master[g[u]] = v;
      if (COMMIT) {
        WStore<WT>::one(a.w, g[u], v);
        store_copies_one<WT>(a.copies, g[u], v);
      }
    }
  }, [] {});
}

// Tiles per block: 4, whose members share the pool of leftovers, while that leaves 608 blocks;
// fewer below, where SMs would be idle: K = 4, 1M and 11.1M elements, perturb 34.6 -> 9.3 and 48.4 ->
// 28.4 us, update (P = 16) 180 -> 51 and 262 -> 165 (4 / these).
static unsigned replay_blocks(uint64_t n_tiles, uint64_t per) {
  per = std::min<uint64_t>(std::max<uint64_t>(per, 1), kReplayTilesPerBlock);
  return (unsigned)((n_tiles + per - 1) / per);
}
static unsigned replay_elem_blocks(uint64_t n_tiles) { return replay_blocks(n_tiles, n_tiles / 608); }

// The update's blocks also fill a table, and for few noise vectors that is much of their time: a
// second wave of a few blocks costs more than fewer blocks do.  P = 1, K = 4, 16 and 64 in the
// mean, 22M, 30M and 36M elements, tiles as above / one more, 55 / 49, 73 / 68 and 81 / 75 us; P = 4
// and 16, K = 4, 24M 121 / 134 and 318 / 362.
static unsigned replay_update_blocks(uint64_t n_tiles, int n_noise) {
  return replay_blocks(n_tiles, n_tiles / 608 + (n_noise <= 2 && n_tiles >= 2 * 608 ? 1 : 0));
}

// Membership mask of subspace r.k: bit (e mod 32) of word tile * 512 + e / 32 is set when
// element e of hash tile `tile` belongs to it.  One block per hash tile; each lane hashes
// one group per step and 8 lanes' 4-bit nibbles make a word.  Tiles the table maps outside
// the arena are flagged and written as empty.
__global__ void __launch_bounds__(kThreads) replay_mask_kernel(const __grid_constant__ ReplayArgs r,
                                                               uint64_t n_alloc, uint32_t *mask) {
  const uint64_t tile = blockIdx.x;
  const ReplayTile t = replay_tile(r, n_alloc, tile);
  const uint32_t lane = threadIdx.x & 31u, warp = threadIdx.x >> 5;
  const uint32_t q_lo0 = (uint32_t)t.q0, q_hi = (uint32_t)(t.q0 >> 32);
  for (int it = 0; it < kReplayIters; ++it) {
    const uint32_t e = warp * (4u * kReplayWarpGroups) + 128u * it + 4u * lane;
    uint32_t nib = 0;
    if (e < t.len) {
      uint32_t x[4];
      philox4x32_10_rk(q_lo0 + (e >> 2), q_hi, t.tensor_id, COPES_TAG_PARTITION, r.rk, x);
#pragma unroll
      for (int i = 0; i < 4; ++i)
        nib |= (x[i] - r.lo <= r.span && e + i < t.len) ? (1u << i) : 0u;
    }
    uint32_t word = nib << (4u * (lane & 7u));
    word |= __shfl_xor_sync(0xffffffffu, word, 1);
    word |= __shfl_xor_sync(0xffffffffu, word, 2);
    word |= __shfl_xor_sync(0xffffffffu, word, 4);
    if ((lane & 7u) == 0) mask[tile * kMaskWordsPerTile + (e >> 5)] = word;
  }
}

cudaError_t launch_replay_mask(const ReplayArgs &r, uint64_t n_alloc, uint32_t *mask, cudaStream_t s) {
  if (r.n_tiles == 0) return cudaSuccess;
  replay_mask_kernel<<<(unsigned)r.n_tiles, kThreads, 0, s>>>(r, n_alloc, mask);
  return cudaGetLastError();
}

template <int OP, typename WT>
static cudaError_t launch_replay_elem_typed(const ElemArgs &a, const ReplayArgs &r, cudaStream_t s) {
  if (r.n_tiles == 0) return cudaSuccess;
  const unsigned blocks = replay_elem_blocks(r.n_tiles);
  if (r.mask) {
    replay_elem_kernel<OP, WT, true, 128><<<blocks, kThreads, 0, s>>>(a, r);
    return cudaGetLastError();
  }
  if constexpr (OP == kOpPerturbPair)
    if (r.K >= sparse_k<WT>()) {
      replay_elem_kernel<OP, WT, false, 64><<<blocks, kThreads, 0, s>>>(a, r);
      return cudaGetLastError();
    }
  replay_elem_kernel<OP, WT, false, 128><<<blocks, kThreads, 0, s>>>(a, r);
  return cudaGetLastError();
}

template <typename WT>
static cudaError_t launch_replay_elem_dtype(int op, const ElemArgs &a, const ReplayArgs &r,
                                            cudaStream_t s) {
  switch (op) {
    case kOpPerturb: return launch_replay_elem_typed<kOpPerturb, WT>(a, r, s);
    case kOpRestore: return launch_replay_elem_typed<kOpRestore, WT>(a, r, s);
    case kOpPerturbPair: return launch_replay_elem_typed<kOpPerturbPair, WT>(a, r, s);
    case kOpPartner: return launch_replay_elem_typed<kOpPartner, WT>(a, r, s);
    case kOpInit: return launch_replay_elem_typed<kOpInit, WT>(a, r, s);
    default: return cudaErrorInvalidValue;  // the other ops have no replay form
  }
}

cudaError_t launch_replay_elementwise(int op, int dtype, const ElemArgs &a, const ReplayArgs &r,
                                      cudaStream_t s) {
  return dtype == COPES_BF16 ? launch_replay_elem_dtype<__nv_bfloat16>(op, a, r, s)
                             : launch_replay_elem_dtype<float>(op, a, r, s);
}

template <typename WT, bool COMMIT>
static cudaError_t launch_replay_update_typed(const UpdateArgs &a, const ReplayArgs &r, cudaStream_t s) {
  if (r.n_tiles == 0) return cudaSuccess;
  const uint32_t smem = gather_smem_bytes(a.n_noise);
  auto kernel = r.mask ? replay_update_kernel<WT, COMMIT, true> : replay_update_kernel<WT, COMMIT, false>;
  // 8.5 KB static
  const cudaError_t e = allow_smem((const void *)kernel, smem + 16 * 1024, gather_smem_bytes(COPES_MAX_NOISE));
  if (e != cudaSuccess) return e;
  kernel<<<replay_update_blocks(r.n_tiles, a.n_noise), kThreads, smem, s>>>(a, r);
  return cudaGetLastError();
}

cudaError_t launch_replay_update(int dtype, const UpdateArgs &a, const ReplayArgs &r, cudaStream_t s) {
  if (dtype == COPES_BF16)
    return a.fuse_commit ? launch_replay_update_typed<__nv_bfloat16, true>(a, r, s)
                         : launch_replay_update_typed<__nv_bfloat16, false>(a, r, s);
  return a.fuse_commit ? launch_replay_update_typed<float, true>(a, r, s)
                       : launch_replay_update_typed<float, false>(a, r, s);
}

unsigned read_and_clear_replay_errors() {
  unsigned v = 0, zero = 0;
  cudaMemcpyFromSymbol(&v, g_replay_error, sizeof(v));
  if (v) cudaMemcpyToSymbol(g_replay_error, &zero, sizeof(zero));
  return v;
}

}  // namespace copes
