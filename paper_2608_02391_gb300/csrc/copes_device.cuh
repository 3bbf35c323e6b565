// Device helpers: the word -> normal transform, bf16 packing and streaming accesses.
#pragma once

#include <cuda_bf16.h>
#include <stdint.h>

#include "copes_internal.h"
#include "normal_coeffs.h"

namespace copes {

__device__ __forceinline__ uint32_t smem_addr(const void *p) {
  return (uint32_t)__cvta_generic_to_shared(p);
}

__device__ __forceinline__ float lg2_approx(float x) {
  float y;
  asm("lg2.approx.ftz.f32 %0, %1;" : "=f"(y) : "f"(x));
  return y;
}

// Packed fp32 pairs: one instruction performs the two lanes' fp32 operations, each rounded
// exactly as the scalar one, at half the instruction count.
__device__ __forceinline__ unsigned long long pack_f32x2(float lo, float hi) {
  unsigned long long r;
  asm("mov.b64 %0, {%1, %2};" : "=l"(r) : "f"(lo), "f"(hi));
  return r;
}
__device__ __forceinline__ void unpack_f32x2(unsigned long long v, float &lo, float &hi) {
  asm("mov.b64 {%0, %1}, %2;" : "=f"(lo), "=f"(hi) : "l"(v));
}
__device__ __forceinline__ unsigned long long fma_f32x2(unsigned long long a, unsigned long long b,
                                                        unsigned long long c) {
  unsigned long long d;
  asm("fma.rn.f32x2 %0, %1, %2, %3;" : "=l"(d) : "l"(a), "l"(b), "l"(c));
  return d;
}
__device__ __forceinline__ unsigned long long add_f32x2(unsigned long long a, unsigned long long b) {
  unsigned long long d;
  asm("add.rn.f32x2 %0, %1, %2;" : "=l"(d) : "l"(a), "l"(b));
  return d;
}
__device__ __forceinline__ unsigned long long mul_f32x2(unsigned long long a, unsigned long long b) {
  unsigned long long d;
  asm("mul.rn.f32x2 %0, %1, %2;" : "=l"(d) : "l"(a), "l"(b));
  return d;
}
__device__ __forceinline__ unsigned long long splat_f32x2(float c) {
  const unsigned long long b = __float_as_uint(c);
  return (b << 32) | b;
}

// ---------------------------------------------------------------- word -> normal
// Standard normal from one Philox word w: eps = Phi^-1(u), u = ((w & 0x7FFFFE) | 1) 2^-23.
// OR-ing those bits (made odd) under the exponent of 2 gives the float 2 + m 2^-22 with m
// odd, so x = 2u - 1 = that - 3 is exact in one add.  Then
//   eps = sqrt(2) erfinv(x) = x * R(L),  L = log2(1 - x^2),
// with R a parabola in L whose coefficients are entry round(-8 L) of a table
// (normal_coeffs.h).  R is fitted relative to its own value, so eps has a small relative
// error for every x, including x near 0 (L -> 0) and near +-1: at most 1.9e-7, 5.1e-8 in
// the mean, and one form serves the centre and the tail.
//
// A multiply of Philox (IMAD.WIDE) keeps the issue port busy for about 4 slots, so the
// kernels that regenerate noise are bound by issue slots, and the transform's instructions
// count one for one: the parabola takes 8.5 a normal (packed pairs counted as one) where a
// polynomial of degree 9 with a voted branch for the tail took about 11.  Measured on the
// update's loop (P = 16, 2^28 elements): 37.9 -> 33.0 cycles per warp-normal, and the
// bound moves towards the 17 multiplies of a Philox block (16.5 cycles a normal).
//
// The table sits in shared memory as C copies, entry i of copy c at float4 C i + c, and a
// lane reads copy lane % C.  With 8 copies (21,632 bytes) the 8 lanes of a quarter-warp,
// which one 128-byte wavefront serves, always hit distinct banks whatever their entries:
// for the kernels that look up several normals per element they load.  The kernels bound
// by scattered loads or the host link take 1 copy (2,704 bytes), which leaves their
// occupancy as it was.
static __device__ const float4 g_normal_table[COPES_NORMAL_ENTRIES] = COPES_NORMAL_TABLE;

template <int C>
struct NormalTable {
  static_assert(C == 1 || C == 8, "copies");
  static constexpr int kFloat4s = COPES_NORMAL_ENTRIES * C;
  static constexpr int kShift = C == 8 ? 7 : 4;  // log2 of an entry's stride in bytes
  uint32_t base;

  // Fills a block's table (every load in flight before the first store); a __syncthreads
  // must follow before the constructor.  `between` runs after the loads have been asked for.
  template <typename Between>
  static __device__ __forceinline__ void fill(float4 *s_tab, Between between) {
    constexpr int kSteps = (kFloat4s + kThreads - 1) / kThreads;
    float4 v[kSteps];
#pragma unroll
    for (int k = 0; k < kSteps; ++k) {
      const int i = threadIdx.x + k * kThreads;
      if (i < kFloat4s) v[k] = g_normal_table[i / C];
    }
    between();
#pragma unroll
    for (int k = 0; k < kSteps; ++k) {
      const int i = threadIdx.x + k * kThreads;
      if (i < kFloat4s) s_tab[i] = v[k];
    }
  }
  static __device__ __forceinline__ void fill(float4 *s_tab) {
    fill(s_tab, [] {});
  }

  // This lane's view of the table, after the fill's barrier: entry i is at base + (f << kShift)
  // modulo 2^32 with f the bits of the float 2^23 + i.  Volatile, and every lookup depends on
  // it, so that no lookup moves above the barrier.
  __device__ __forceinline__ explicit NormalTable(const float4 *s_tab) {
    base = smem_addr(s_tab) + (threadIdx.x & (C - 1)) * 16u - (0x4B000000u << kShift);
    asm volatile("mov.b32 %0, %0;" : "+r"(base)::"memory");
  }

  __device__ __forceinline__ float4 entry(float f) const {
    float4 v;
    asm("ld.shared.v4.f32 {%0, %1, %2, %3}, [%4];"
        : "=f"(v.x), "=f"(v.y), "=f"(v.z), "=f"(v.w)
        : "r"(base + (__float_as_uint(f) << kShift)));
    return v;
  }
};

using WideTable = NormalTable<8>;
using SlimTable = NormalTable<1>;

// The normals of G Philox blocks as packed pairs: e2[i][p] = (eps_2p, eps_2p+1) of block i.
template <int G, typename Table>
__device__ __forceinline__ void normals_packed(const uint32_t (&w)[G][4], const Table &tab,
                                               unsigned long long (&e2)[G][2]) {
  constexpr float kMagic = 8388608.0f;  // 2^23: adding it rounds to a whole number in the low bits
#pragma unroll
  for (int i = 0; i < G; ++i)
#pragma unroll
    for (int p = 0; p < 2; ++p) {
      const unsigned long long F = pack_f32x2(__uint_as_float((w[i][2 * p] & 0x007FFFFEu) | 0x40000001u),
                                              __uint_as_float((w[i][2 * p + 1] & 0x007FFFFEu) | 0x40000001u));
      const unsigned long long x2 = add_f32x2(F, splat_f32x2(-3.0f));
      float t0, t1;  // x^2 - 1 = -(1 - x^2)
      unpack_f32x2(fma_f32x2(x2, x2, splat_f32x2(-1.0f)), t0, t1);
      const float L0 = lg2_approx(-t0), L1 = lg2_approx(-t1);
      float f0, f1;
      unpack_f32x2(fma_f32x2(pack_f32x2(L0, L1), splat_f32x2(-(float)COPES_NORMAL_SEGMENTS), splat_f32x2(kMagic)), f0,
                   f1);
      const float4 k0 = tab.entry(f0), k1 = tab.entry(f1);
      const float r0 = __fmaf_rn(__fmaf_rn(k0.z, L0, k0.y), L0, k0.x);
      const float r1 = __fmaf_rn(__fmaf_rn(k1.z, L1, k1.y), L1, k1.x);
      e2[i][p] = mul_f32x2(x2, pack_f32x2(r0, r1));
    }
}

// One word, and two words as a packed pair: normals_packed's values bit for bit.
template <typename Table>
__device__ __forceinline__ unsigned long long normal_pair(uint32_t wa, uint32_t wb, const Table &tab) {
  const uint32_t w[1][4] = {{wa, wb, wa, wb}};
  unsigned long long e2[1][2];
  normals_packed<1>(w, tab, e2);
  return e2[0][0];
}

template <typename Table>
__device__ __forceinline__ float normal_from_word(uint32_t w, const Table &tab) {
  const float x = __fadd_rn(__uint_as_float((w & 0x007FFFFEu) | 0x40000001u), -3.0f);
  const float L = lg2_approx(-__fmaf_rn(x, x, -1.0f));
  const float4 k = tab.entry(__fmaf_rn(L, -(float)COPES_NORMAL_SEGMENTS, 8388608.0f));
  return __fmul_rn(x, __fmaf_rn(__fmaf_rn(k.z, L, k.y), L, k.x));
}

__device__ __forceinline__ uint32_t pack_bf16x2(float lo, float hi) {
  __nv_bfloat162 v = __floats2bfloat162_rn(lo, hi);
  return *reinterpret_cast<uint32_t *>(&v);
}

__device__ __forceinline__ uint16_t to_bf16_bits(float x) {
  __nv_bfloat16 v = __float2bfloat16_rn(x);
  return *reinterpret_cast<uint16_t *>(&v);
}

// Streaming (evict-first) 16-byte load of read-once data and matching stores.
__device__ __forceinline__ float4 ld_stream_f4(const float *p) {
  return __ldcs(reinterpret_cast<const float4 *>(p));
}
// 32 bytes (aligned to as many) in one load, past the L1.
__device__ __forceinline__ void ld_stream_f8(const float *p, float (&x)[4], float (&y)[4]) {
  asm volatile("ld.global.L1::no_allocate.v8.f32 {%0, %1, %2, %3, %4, %5, %6, %7}, [%8];"
               : "=f"(x[0]), "=f"(x[1]), "=f"(x[2]), "=f"(x[3]), "=f"(y[0]), "=f"(y[1]), "=f"(y[2]), "=f"(y[3])
               : "l"(p));
}
__device__ __forceinline__ void prefetch_l2(const void *p) { asm volatile("prefetch.global.L2 [%0];" ::"l"(p)); }
__device__ __forceinline__ void st_stream_f4(float *p, float4 v) {
  __stcs(reinterpret_cast<float4 *>(p), v);
}
__device__ __forceinline__ void st_stream_u2(void *p, uint2 v) {
  __stcs(reinterpret_cast<uint2 *>(p), v);
}

// ------------------------------------------------------------------------------------
// Gather-list staging: a block's segment of the int64 index list is brought into shared
// memory by TMA 1D bulk copies (cp.async.bulk) in chunks, double-buffered on mbarriers,
// so the next chunk's indices are in flight while the current chunk is processed.
// Every wait is bounded: after kStageWaitLimit polls the block records kErrStageTimeout,
// waits (bounded again) for its own copies, and stops.
constexpr int kStageChunk = 1024;         // indices per chunk (8 KB)
constexpr int kStageWaitLimit = 1 << 22;  // mbarrier polls before giving up

__device__ __forceinline__ void mbar_init(uint64_t *bar, uint32_t count) {
  asm volatile("mbarrier.init.shared::cta.b64 [%0], %1;" ::"r"(smem_addr(bar)), "r"(count));
}

__device__ __forceinline__ void mbar_fence_init() {
  asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
}

// One producer arrival announcing `bytes` of transaction, then the bulk copy itself.
__device__ __forceinline__ void stage_copy(uint64_t *bar, void *dst, const void *src, uint32_t bytes) {
  asm volatile("mbarrier.arrive.expect_tx.shared::cta.b64 _, [%0], %1;" ::"r"(smem_addr(bar)), "r"(bytes)
               : "memory");
  if (bytes)
    asm volatile(
        "cp.async.bulk.shared::cluster.global.mbarrier::complete_tx::bytes [%0], [%1], %2, [%3];" ::"r"(
            smem_addr(dst)),
        "l"(src), "r"(bytes), "r"(smem_addr(bar))
        : "memory");
}

// Polls the barrier's phase `parity` at most kStageWaitLimit times; true once complete.
__device__ __forceinline__ bool mbar_wait_bounded(uint64_t *bar, uint32_t parity) {
  for (int it = 0; it < kStageWaitLimit; ++it) {
    uint32_t done;
    asm volatile(
        "{\n .reg .pred p;\n mbarrier.try_wait.parity.shared::cta.b64 p, [%1], %2;\n selp.u32 %0, 1, 0, p;\n}"
        : "=r"(done)
        : "r"(smem_addr(bar)), "r"(parity)
        : "memory");
    if (done) return true;
  }
  return false;
}

// Walks the block's segment [s0, s1) of `index` in chunks staged through shared memory;
// body(const int64_t *chunk_in_smem, int count, uint64_t first_position) runs on every
// chunk with all threads of the block.  A chunk of odd length copies its even prefix by
// TMA (sizes must be multiples of 16 bytes) and its last index from global memory into
// shared memory.  Returns false (after flagging) if a wait timed out.
template <typename Body, typename Flag>
__device__ __forceinline__ bool staged_index_segment(const int64_t *index, uint64_t s0, uint64_t s1,
                                                     int64_t (*buf)[kStageChunk], uint64_t *bar,
                                                     Flag flag, Body body) {
  const int n_chunks = (int)((s1 - s0 + kStageChunk - 1) / kStageChunk);
  auto chunk_count = [&](int c) { return (int)min((uint64_t)kStageChunk, s1 - s0 - (uint64_t)c * kStageChunk); };
  auto issue = [&](int c) {
    const int cnt = chunk_count(c);
    stage_copy(&bar[c & 1], buf[c & 1], index + s0 + (uint64_t)c * kStageChunk, (uint32_t)(cnt & ~1) * 8u);
  };
  if (threadIdx.x == 0) {
    mbar_init(&bar[0], 1);
    mbar_init(&bar[1], 1);
    mbar_fence_init();
  }
  __syncthreads();
  if (threadIdx.x == 0) {
    issue(0);
    if (n_chunks > 1) issue(1);
  }
  for (int c = 0; c < n_chunks; ++c) {
    const int slot = c & 1;
    const int cnt = chunk_count(c);
    if (!mbar_wait_bounded(&bar[slot], (uint32_t)((c >> 1) & 1))) {
      if (threadIdx.x == 0) flag();
      // the copy into this block's shared memory may still be in flight: wait once more
      mbar_wait_bounded(&bar[slot], (uint32_t)((c >> 1) & 1));
      return false;
    }
    if ((cnt & 1) && threadIdx.x == 0) buf[slot][cnt - 1] = index[s0 + (uint64_t)c * kStageChunk + cnt - 1];
    __syncthreads();
    body((const int64_t *)buf[slot], cnt, s0 + (uint64_t)c * kStageChunk);
    __syncthreads();  // every thread is done reading this slot before it is refilled
    if (threadIdx.x == 0 && c + 2 < n_chunks) {
      asm volatile("fence.proxy.async.shared::cta;" ::: "memory");
      issue(c + 2);
    }
  }
  return true;
}

}  // namespace copes
