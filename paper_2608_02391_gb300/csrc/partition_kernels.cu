// Partition kernels (Eq. 7; Algorithm 1 "sample a partition"; Supp. A.8 partition
// replay): the hash partition's per-tile histogram, per-bucket exclusive scan and
// order-preserving scatter into sorted int64 lists, and the random-chunk map.
#include "copes_internal.h"

namespace copes {

__device__ unsigned int g_partition_error = 0;

constexpr int kPartThreads = 256;

// The tensor owning hash tile `tile`: the last entry with tile_begin <= tile (the host
// table lists only tensors with at least one element).  By a whole warp: 32 probes a step,
// so that a table of 400 tensors takes 2 dependent loads instead of 9.
__device__ int owner_tensor(const HashTensor *tensors, int n_tensors, uint64_t tile) {
  const int lane = threadIdx.x & 31;
  int lo = 0, n = n_tensors;
  while (n > 1) {
    const int stride = (n + 31) / 32, at = lane * stride;
    const bool below = at < n && tensors[lo + at].tile_begin <= tile;
    const int c = max(__popc(__ballot_sync(0xffffffffu, below)) - 1, 0);
    lo += c * stride;
    n = min(stride, n - c * stride);
  }
  return lo;
}

// A hash tile and the folded keys of its elements' partition counters (e >> 2, tensor id):
// q0 = e0 >> 2 is a multiple of 4,096 and the tile has 4,096 groups, so the counters' high
// word is one value.
struct PartTile {
  HashTensor T;
  uint64_t e0;
  uint32_t len;
  uint32_t u[20];
  __device__ __forceinline__ PartTile(const HashTensor *tensors, int n_tensors, uint64_t tile, uint64_t seed) {
    T = tensors[owner_tensor(tensors, n_tensors, tile)];
    e0 = (tile - T.tile_begin) * kHashTile;
    len = (uint32_t)min(kHashTile, T.numel - e0);
    uint32_t rk[20];
    philox_round_keys((uint32_t)seed, (uint32_t)(seed >> 32), rk);
    philox_folded_keys(rk, COPES_TAG_PARTITION, u, (uint32_t)(e0 >> 34), T.tensor_id);
  }
  // The words of group `group` of the tile.
  __device__ __forceinline__ void words(uint32_t group, uint32_t (&x)[4]) const {
    const uint64_t m = (uint64_t)kPhiloxM0 * ((uint32_t)(e0 >> 2) + group);
    philox4x32_10_folded((uint32_t)m, (uint32_t)(m >> 32), u, x);
  }
};

// floor(x K / 2^32): a shift when K is 2^shift > 1, which a multiply-high would give the same.
struct Bucket {
  uint32_t K, shift;  // shift 0: multiply
  __device__ __forceinline__ explicit Bucket(int k) : K(k) { shift = k > 1 && (k & (k - 1)) == 0 ? 31 - __clz(k) : 0; }
  __device__ __forceinline__ uint32_t operator()(uint32_t x) const {
    return shift ? x >> (32 - shift) : __umulhi(x, K);
  }
};

// One block per hash tile.  Every lane counts into its own column of a K x 32 table, so that
// the shared-memory adds of a warp hit 32 banks.
__global__ void __launch_bounds__(kPartThreads) hash_hist_kernel(
    const HashTensor *tensors, int n_tensors, int K, uint64_t seed, uint32_t *hist,
    unsigned long long *totals) {
  __shared__ uint32_t s_h[COPES_MAX_K * 32];
  const uint64_t tile = blockIdx.x;
  const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
  for (int i = threadIdx.x; i < K * 32; i += kPartThreads) s_h[i] = 0;
  const PartTile t(tensors, n_tensors, tile, seed);
  const Bucket bucket(K);
  __syncthreads();
  uint32_t *column = s_h + lane;
  if (t.len == kHashTile) {
#pragma unroll 4
    for (uint32_t g = threadIdx.x; g < kHashTile / 4; g += kPartThreads) {
      uint32_t x[4];
      t.words(g, x);
#pragma unroll
      for (int i = 0; i < 4; ++i) atomicAdd(column + bucket(x[i]) * 32, 1u);
    }
  } else {
    for (uint32_t e = 4u * threadIdx.x; e < t.len; e += 4u * kPartThreads) {
      uint32_t x[4];
      t.words(e >> 2, x);
#pragma unroll
      for (int i = 0; i < 4; ++i)
        if (e + i < t.len) atomicAdd(column + bucket(x[i]) * 32, 1u);
    }
  }
  __syncthreads();
  for (int k = warp; k < K; k += kPartThreads / 32) {
    const uint32_t n = __reduce_add_sync(0xffffffffu, s_h[k * 32 + lane]);
    if (lane == 0) {
      hist[tile * K + k] = n;
      if (n) atomicAdd(&totals[k], (unsigned long long)n);
    }
  }
}

// Inclusive sum over the warp's lanes.
__device__ __forceinline__ uint32_t warp_scan(uint32_t v) {
  const int lane = threadIdx.x & 31;
#pragma unroll
  for (int d = 1; d < 32; d <<= 1) {
    const uint32_t o = __shfl_up_sync(0xffffffffu, v, d);
    if (lane >= d) v += o;
  }
  return v;
}

// The exclusive prefix sums of hist[tile][k] over the tiles, per bucket k, in chunks of tiles.  A
// chunk's block sums the tiles before it itself while that is little (hash_scan_rereads);
// beyond, two launches before it are linear in the tiles: the sums of the chunks, and their
// scan.  Until the last launch, the start of a chunk lies in offsets at the chunk's first
// tile, which is where it belongs.
constexpr int kScanVec = 4;         // consecutive tiles a thread
constexpr int kScanThreads = 256;   // with starts
constexpr int kRereadThreads = 1024;
constexpr uint64_t kScanChunk = kScanVec * kScanThreads;
constexpr int kSumThreads = 1024;
static_assert((uint64_t)kScanVec * kRereadThreads * kHashTile < 1ull << 32, "a chunk's sum fits 32 bits");
static_assert(COPES_MAX_K <= kSumThreads, "a thread per bucket");

// Re-read / with the launches before, us: 12,208 tiles, K = 16 and 64 9.3 / 12.3 and 21 / 26; 30,518
// tiles 13.8 / 14.9 and 58 / 36; 488,282 tiles 915 / 88 and 6,393 / 353; and two launches more.
static bool hash_scan_rereads(uint64_t n_htiles, int K) {
  const uint64_t chunks = (n_htiles + kScanVec * kRereadThreads - 1) / (kScanVec * kRereadThreads);
  return chunks <= 40 && chunks * chunks * (uint64_t)K <= 1600;
}

__global__ void __launch_bounds__(kSumThreads) hash_chunk_sums_kernel(const uint32_t *hist, uint64_t n_htiles, int K,
                                                                       uint64_t *offsets) {
  __shared__ uint32_t s_sum[COPES_MAX_K];
  const uint64_t t0 = blockIdx.x * kScanChunk, rows = min(kScanChunk, n_htiles - t0);
  if (threadIdx.x < K) s_sum[threadIdx.x] = 0;
  __syncthreads();
  const uint32_t at_once = kSumThreads / K, row = threadIdx.x / K, k = threadIdx.x % K;
  uint32_t sum = 0;
  if (row < at_once) {
#pragma unroll 8
    for (uint64_t r = row; r < rows; r += at_once) sum += hist[(t0 + r) * K + k];
    atomicAdd(&s_sum[k], sum);
  }
  __syncthreads();
  if (threadIdx.x < K) offsets[t0 * K + threadIdx.x] = s_sum[threadIdx.x];
}

// Block k: the chunks' sums to their starts, 1,024 chunks a step.
constexpr int kStartThreads = 1024;

__global__ void __launch_bounds__(kStartThreads) hash_chunk_starts_kernel(uint64_t n_chunks, int K, uint64_t *offsets) {
  __shared__ unsigned long long s_warp[kStartThreads / 32];
  const int k = blockIdx.x, warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
  unsigned long long before = 0;  // the sum of the steps before
  for (uint64_t c0 = 0; c0 < n_chunks; c0 += kStartThreads) {
    const uint64_t c = c0 + threadIdx.x;
    uint64_t *const at = offsets + c * kScanChunk * K + k;
    const unsigned long long mine = c < n_chunks ? *at : 0ull;
    unsigned long long upto = mine;
#pragma unroll
    for (int d = 1; d < 32; d <<= 1) {
      const unsigned long long o = __shfl_up_sync(0xffffffffu, upto, d);
      if (lane >= d) upto += o;
    }
    if (lane == 31) s_warp[warp] = upto;
    __syncthreads();
    unsigned long long all = 0;
    for (int w = 0; w < kStartThreads / 32; ++w) {
      if (w == warp) upto += all;
      all += s_warp[w];
    }
    if (c < n_chunks) *at = before + upto - mine;
    before += all;
    __syncthreads();  // before the next step's sums
  }
}

// Block c K + k: chunk c, of kScanVec THREADS tiles, of bucket k.
template <int THREADS, bool REREAD>
__global__ void __launch_bounds__(THREADS) hash_scan_kernel(const uint32_t *hist, uint64_t n_htiles, int K,
                                                            uint64_t *offsets) {
  __shared__ unsigned long long s_before[THREADS / 32];
  __shared__ uint32_t s_warp[THREADS / 32];
  const uint32_t chunk = blockIdx.x / K, k = blockIdx.x % K;
  const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
  const uint64_t t0 = chunk * (uint64_t)(kScanVec * THREADS), t = t0 + (uint64_t)kScanVec * threadIdx.x;
  uint32_t mine[kScanVec], sum = 0;
#pragma unroll
  for (int i = 0; i < kScanVec; ++i) sum += mine[i] = t + i < n_htiles ? hist[(t + i) * K + k] : 0u;
  unsigned long long before = 0;
  if (REREAD) {
#pragma unroll 8
    for (uint64_t p = threadIdx.x; p < t0; p += THREADS) before += hist[p * K + k];
#pragma unroll
    for (int d = 16; d > 0; d >>= 1) before += __shfl_xor_sync(0xffffffffu, before, d);
  } else if (threadIdx.x == 0) {
    before = offsets[t0 * K + k];
  }
  const uint32_t upto = warp_scan(sum);
  if (lane == 31) s_warp[warp] = upto;
  if (lane == 0) s_before[warp] = before;
  __syncthreads();  // the start has been read as well
  unsigned long long at = __reduce_add_sync(0xffffffffu, lane < warp ? s_warp[lane] : 0u) + upto - sum;
#pragma unroll
  for (int w = 0; w < THREADS / 32; ++w) at += s_before[w];
#pragma unroll
  for (int i = 0; i < kScanVec; ++i) {
    if (t + i < n_htiles) offsets[(t + i) * K + k] = at;
    at += mine[i];
  }
}

struct ListTable {
  int64_t *list[COPES_MAX_K];
};

// One block per hash tile, a stable counting sort of its elements by bucket in shared memory.
// Each thread takes 64 consecutive elements: it counts them into its own column of a K x 256
// table (a warp's lanes hit 32 banks); the scan of each row over the threads, started at the
// bucket's first position, turns the counts into positions; and the thread hands its elements
// their positions in order.  Each bucket's stretch is then written to its list by whole
// warps.  So a group of 4 elements is hashed once and the lists are written in full lines.
// 494M elements, K = 16: 4.04 ms when every element hashed its own group and went to its list
// directly, 2.79 ms with ranks from warp matches instead of private columns.
constexpr uint32_t kScatterGroups = (uint32_t)kHashTile / 4 / kPartThreads;  // consecutive groups a thread
constexpr uint32_t kScatterSmem(int K) { return (uint32_t)kHashTile * 2 + (uint32_t)K * kPartThreads * 4; }

__global__ void __launch_bounds__(kPartThreads) hash_scatter_kernel(
    const HashTensor *tensors, int n_tensors, int K, uint64_t seed, const uint64_t *offsets,
    const __grid_constant__ ListTable lists) {
  extern __shared__ __align__(16) uint16_t s_sorted[];
  uint32_t *s_cnt = reinterpret_cast<uint32_t *>(s_sorted + kHashTile);
  __shared__ uint32_t s_start[COPES_MAX_K + 1];
  const uint64_t tile = blockIdx.x;
  const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
  constexpr int kWarps = kPartThreads / 32;
  uint32_t *column = s_cnt + threadIdx.x;
  for (int k = 0; k < K; ++k) column[k * kPartThreads] = 0;
  const PartTile t(tensors, n_tensors, tile, seed);
  const Bucket bucket(K);
  const uint32_t g0 = threadIdx.x * kScatterGroups;  // the thread's first group
  uint32_t packed[kScatterGroups];                   // its groups' buckets
  const uint32_t mine = min(t.len - min(t.len, g0 * 4), kScatterGroups * 4u);  // its elements
#pragma unroll
  for (uint32_t i = 0; i < kScatterGroups; ++i) {
    uint32_t x[4];
    t.words(g0 + i, x);
    packed[i] = 0;
#pragma unroll
    for (uint32_t j = 0; j < 4; ++j) {
      const uint32_t b = bucket(x[j]);
      packed[i] |= b << (8 * j);
      if (i * 4 + j < mine) atomicAdd(column + b * kPartThreads, 1u);
    }
  }
  __syncthreads();
  for (int k = warp; k < K; k += kWarps) {  // the buckets' counts
    uint32_t n = 0;
#pragma unroll
    for (int w = 0; w < kWarps; ++w) n += s_cnt[k * kPartThreads + w * 32 + lane];
    n = __reduce_add_sync(0xffffffffu, n);
    if (lane == 0) s_start[k + 1] = n;
  }
  __syncthreads();
  if (warp == 0) {
    uint32_t lo = warp_scan(lane < K ? s_start[lane + 1] : 0u);
    uint32_t hi = warp_scan(lane + 32 < K ? s_start[lane + 33] : 0u) + __shfl_sync(0xffffffffu, lo, 31);
    s_start[lane + 1] = lo;
    s_start[lane + 33] = hi;
    if (lane == 0) s_start[0] = 0;
  }
  __syncthreads();
  for (int k = warp; k < K; k += kWarps) {
    uint32_t at = s_start[k];
#pragma unroll
    for (int w = 0; w < kWarps; ++w) {
      uint32_t *c = s_cnt + k * kPartThreads + w * 32 + lane;
      const uint32_t n = *c, upto = warp_scan(n);
      *c = at + upto - n;
      at += __shfl_sync(0xffffffffu, upto, 31);
    }
  }
  __syncthreads();
#pragma unroll
  for (uint32_t i = 0; i < kScatterGroups; ++i)
#pragma unroll
    for (int j = 0; j < 4; ++j) {
      if (i * 4 + j < mine)
        s_sorted[atomicAdd(column + (packed[i] >> (8 * j) & 0xFFu) * kPartThreads, 1u)] = (uint16_t)((g0 + i) * 4 + j);
    }
  __syncthreads();
  // the buckets' stretches: whole ones dealt to the warps, or all of them to all warps when
  // they are fewer
  const int64_t first = (int64_t)(t.T.offset + t.e0);
  const bool whole = K >= kWarps;
  const uint32_t lane0 = whole ? 0u : warp * 32u, stride = whole ? 32u : kPartThreads;
  for (int k = whole ? warp : 0; k < K; k += whole ? kWarps : 1) {
    const uint32_t b = s_start[k], n = s_start[k + 1] - b;
    long long *list = reinterpret_cast<long long *>(lists.list[k] + offsets[tile * K + k]);
#pragma unroll 4
    for (uint32_t i = lane0 + lane; i < n; i += stride) __stcs(list + i, (long long)(first + s_sorted[b + i]));
  }
}

// Random chunk map: chunk c has key = word 0 of Philox(seed; c, 0, CHUNK tag) and goes to
// subspace floor(rank K / n), rank = its position in (key, c) order.  The composite keys
// (key << 20) | c (c < 2^20) are distinct, so the ranks are the positions after sorting
// them: a bitonic sort over the caller's workspace (N = a power of two >= n, padded with
// the largest key), with every 4,096-key tile sorted and merged in shared memory and
// only the strides of 4,096 and more done by global-memory passes.
constexpr uint64_t kSortTile = 4096;
constexpr int kSortThreads = 512;

__global__ void __launch_bounds__(kSortThreads) chunk_keys_kernel(uint64_t n, uint64_t N, uint64_t seed,
                                                                   uint64_t *A) {
  const uint64_t i = (uint64_t)blockIdx.x * kSortThreads + threadIdx.x;
  if (i >= N) return;
  if (i < n) {
    uint32_t x[4];
    philox4x32_10((uint32_t)i, (uint32_t)(i >> 32), 0u, COPES_TAG_CHUNK, (uint32_t)seed,
                  (uint32_t)(seed >> 32), x);
    A[i] = ((uint64_t)x[0] << 20) | i;
  } else {
    A[i] = ~0ull;
  }
}

// One compare-exchange step (stage k, stride j) over a tile held in shared memory; the
// direction of each pair comes from its global index.
__device__ __forceinline__ void bitonic_smem_step(uint64_t *s, uint64_t base, uint64_t k, uint64_t j) {
  for (uint32_t t = threadIdx.x; t < kSortTile; t += kSortThreads) {
    const uint32_t l = t ^ (uint32_t)j;
    if (l > t) {
      const bool up = ((base + t) & k) == 0;
      const uint64_t a = s[t], b = s[l];
      if ((a > b) == up) {
        s[t] = b;
        s[l] = a;
      }
    }
  }
  __syncthreads();
}

// k_stage == 0: sort every tile (stages 2 .. kSortTile).  Otherwise: the strides below
// kSortTile of stage k_stage.
__global__ void __launch_bounds__(kSortThreads) bitonic_tile_kernel(uint64_t *A, uint64_t k_stage) {
  __shared__ uint64_t s[kSortTile];
  const uint64_t base = (uint64_t)blockIdx.x * kSortTile;
  for (uint32_t t = threadIdx.x; t < kSortTile; t += kSortThreads) s[t] = A[base + t];
  __syncthreads();
  if (k_stage == 0) {
    for (uint64_t k = 2; k <= kSortTile; k <<= 1)
      for (uint64_t j = k >> 1; j > 0; j >>= 1) bitonic_smem_step(s, base, k, j);
  } else {
    for (uint64_t j = kSortTile >> 1; j > 0; j >>= 1) bitonic_smem_step(s, base, k_stage, j);
  }
  for (uint32_t t = threadIdx.x; t < kSortTile; t += kSortThreads) A[base + t] = s[t];
}

__global__ void __launch_bounds__(kSortThreads) bitonic_global_kernel(uint64_t *A, uint64_t N, uint64_t j,
                                                                      uint64_t k) {
  const uint64_t i = (uint64_t)blockIdx.x * kSortThreads + threadIdx.x;
  if (i >= N) return;
  const uint64_t l = i ^ j;
  if (l > i) {
    const bool up = (i & k) == 0;
    const uint64_t a = A[i], b = A[l];
    if ((a > b) == up) {
      A[i] = b;
      A[l] = a;
    }
  }
}

__global__ void __launch_bounds__(kSortThreads) chunk_map_kernel(const uint64_t *A, uint64_t n, int K,
                                                                 uint32_t *map) {
  const uint64_t i = (uint64_t)blockIdx.x * kSortThreads + threadIdx.x;
  if (i >= n) return;
  map[A[i] & 0xFFFFFull] = (uint32_t)((i * (uint64_t)K) / n);
}

uint64_t chunk_sort_size(uint64_t n_chunks) {
  uint64_t N = kSortTile;
  while (N < n_chunks) N <<= 1;
  return N;
}

cudaError_t launch_hash_hist(const HashTensor *tensors, int n_tensors, uint64_t n_htiles, int K,
                             uint64_t seed, uint32_t *hist, unsigned long long *totals,
                             cudaStream_t s) {
  if (n_htiles == 0) return cudaSuccess;
  hash_hist_kernel<<<(unsigned)n_htiles, kPartThreads, 0, s>>>(tensors, n_tensors, K, seed, hist,
                                                                totals);
  return cudaGetLastError();
}

cudaError_t launch_hash_scan(const uint32_t *hist, uint64_t n_htiles, int K, uint64_t *offsets,
                             cudaStream_t s) {
  if (n_htiles == 0) return cudaSuccess;
  if (hash_scan_rereads(n_htiles, K)) {
    constexpr uint64_t kChunk = kScanVec * kRereadThreads;
    const unsigned blocks = (unsigned)((n_htiles + kChunk - 1) / kChunk * K);
    hash_scan_kernel<kRereadThreads, true><<<blocks, kRereadThreads, 0, s>>>(hist, n_htiles, K, offsets);
  } else {
    const uint64_t chunks = (n_htiles + kScanChunk - 1) / kScanChunk;  // chunks K <= 2^27: n_htiles < 2^31
    hash_chunk_sums_kernel<<<(unsigned)chunks, kSumThreads, 0, s>>>(hist, n_htiles, K, offsets);
    hash_chunk_starts_kernel<<<K, kStartThreads, 0, s>>>(chunks, K, offsets);
    hash_scan_kernel<kScanThreads, false><<<(unsigned)(chunks * K), kScanThreads, 0, s>>>(hist, n_htiles, K, offsets);
  }
  return cudaGetLastError();
}

cudaError_t launch_hash_scatter(const HashTensor *tensors, int n_tensors, uint64_t n_htiles,
                                int K, uint64_t seed, const uint64_t *offsets,
                                int64_t *const *lists, cudaStream_t s) {
  if (n_htiles == 0) return cudaSuccess;
  ListTable t;
  for (int k = 0; k < COPES_MAX_K; ++k) t.list[k] = k < K ? lists[k] : nullptr;
  const uint32_t smem = kScatterSmem(K);
  const cudaError_t e = allow_smem((const void *)hash_scatter_kernel, smem + 1024, kScatterSmem(COPES_MAX_K));
  if (e != cudaSuccess) return e;
  hash_scatter_kernel<<<(unsigned)n_htiles, kPartThreads, smem, s>>>(tensors, n_tensors, K, seed, offsets, t);
  return cudaGetLastError();
}

cudaError_t launch_random_chunk_map(uint64_t n_chunks, int K, uint64_t seed, uint32_t *map,
                                    uint64_t *keys, cudaStream_t s) {
  const uint64_t N = chunk_sort_size(n_chunks);
  const unsigned gblocks = (unsigned)((N + kSortThreads - 1) / kSortThreads);
  const unsigned tiles = (unsigned)(N / kSortTile);
  chunk_keys_kernel<<<gblocks, kSortThreads, 0, s>>>(n_chunks, N, seed, keys);
  bitonic_tile_kernel<<<tiles, kSortThreads, 0, s>>>(keys, 0);
  for (uint64_t k = 2 * kSortTile; k <= N; k <<= 1) {
    for (uint64_t j = k >> 1; j >= kSortTile; j >>= 1)
      bitonic_global_kernel<<<gblocks, kSortThreads, 0, s>>>(keys, N, j, k);
    bitonic_tile_kernel<<<tiles, kSortThreads, 0, s>>>(keys, k);
  }
  const unsigned mblocks = (unsigned)((n_chunks + kSortThreads - 1) / kSortThreads);
  chunk_map_kernel<<<mblocks, kSortThreads, 0, s>>>(keys, n_chunks, K, map);
  return cudaGetLastError();
}

// Tile table of a list of disjoint ranges, written on the device: tile t lies in the range
// r with first[r] <= t < first[r + 1] and covers [begin[r] + (t - first[r]) tile_size,
// min(that + tile_size, end[r])).  The ranges travel in the launch's parameters, so no
// host staging of the table is needed.
__global__ void __launch_bounds__(256) tile_expand_kernel(const __grid_constant__ TileRanges a, uint64_t *tiles) {
  for (uint64_t t = (uint64_t)blockIdx.x * blockDim.x + threadIdx.x; t < a.first[a.n_ranges];
       t += (uint64_t)gridDim.x * blockDim.x) {
    int lo = 0, hi = a.n_ranges - 1;  // the last range whose first tile is <= t
    while (lo < hi) {
      const int mid = (lo + hi + 1) >> 1;
      if (a.first[mid] <= t) lo = mid;
      else hi = mid - 1;
    }
    const uint64_t b = a.begin[lo] + (t - a.first[lo]) * a.tile_size;
    const uint64_t e = min(b + a.tile_size, a.end[lo]);
    reinterpret_cast<ulonglong2 *>(tiles)[t] = make_ulonglong2(b, e);
  }
}

cudaError_t launch_tile_expand(const TileRanges &r, uint64_t *tiles, cudaStream_t s) {
  const uint64_t n = r.first[r.n_ranges];
  if (n == 0) return cudaSuccess;
  const uint64_t want = (n + 255) / 256;
  const unsigned blocks = (unsigned)(want < 4096 ? want : 4096);
  tile_expand_kernel<<<blocks, 256, 0, s>>>(r, tiles);
  return cudaGetLastError();
}

unsigned read_and_clear_partition_errors() {
  unsigned v = 0, zero = 0;
  cudaMemcpyFromSymbol(&v, g_partition_error, sizeof(v));
  if (v) cudaMemcpyToSymbol(g_partition_error, &zero, sizeof(zero));
  return v;
}

}  // namespace copes
