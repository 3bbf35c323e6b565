// The elementwise noise ops' values, stores and vector step, shared by their kernels over default
// tiles (es_kernels.cu) and over any others (elem_ragged.cu).
#pragma once

#include "es_common.cuh"

namespace copes {

// A "group" is the 4 consecutive global indices 4q .. 4q+3, which share Philox counter q.

// Ops whose values are the context (restore / commit, init) go to the other working copies
// too; perturbations go to the buffers their call names.
template <int OP>
constexpr bool writes_context() { return OP == kOpRestore || OP == kOpInit; }

// Noise vectors and values an op forms per element: the perturb theta + a eps, the pair also
// theta - a eps, the two pairs theta +- a eps_A and theta +- a eps_B, init b + a eps.
template <int OP>
constexpr int op_noises() { return OP == kOpPerturbTwoPairs ? 2 : 1; }
template <int OP>
constexpr int op_values() { return OP == kOpPerturbTwoPairs ? 4 : (OP == kOpPerturbPair ? 2 : 1); }

// The values of one group from its noise (e2[s]: noise vector s as packed pairs) and theta:
// v[0] = fma(a, eps, theta), and with the antithetic sign v[1] = fma(-a, eps, theta) (pair;
// the two pairs' v[2], v[3] from the second vector): each bit for bit what kOpPerturb
// computes with that noise vector and sign.
template <int OP>
__device__ __forceinline__ void group_values(const ElemArgs &a, const unsigned long long (*e2)[2],
                                             const float (&th)[4], float (&v)[op_values<OP>()][4]) {
#pragma unroll
  for (int p = 0; p < 2; ++p) {
    const unsigned long long t2 = OP == kOpInit ? splat_f32x2(a.b) : pack_f32x2(th[2 * p], th[2 * p + 1]);
#pragma unroll
    for (int m = 0; m < op_values<OP>(); ++m)
      unpack_f32x2(fma_f32x2(splat_f32x2((m & 1) ? -a.a : a.a), e2[m >> 1][p], t2), v[m][2 * p], v[m][2 * p + 1]);
  }
}

// Value m of an op goes to w (m = 0), the partner buffer (the pair's m = 1) or the further
// working copies (the two pairs' m = 1 .. 3); the context's only value to all copies.
template <int OP, typename WT>
__device__ __forceinline__ void store_values_full(const ElemArgs &a, uint64_t g, const float (&v)[op_values<OP>()][4]) {
  if (OP == kOpInit) st_stream_f4(a.master + g, make_float4(v[0][0], v[0][1], v[0][2], v[0][3]));
  WStore<WT>::full(a.w, g, v[0]);
  if constexpr (writes_context<OP>()) store_copies_full<WT>(a.copies, g, v[0]);
  if constexpr (OP == kOpPerturbPair) WStore<WT>::full(a.partner, g - a.partner_base, v[1]);
  if constexpr (OP == kOpPerturbTwoPairs) {
#pragma unroll
    for (int m = 1; m < 4; ++m) WStore<WT>::full(a.copies.p[m - 1], g, v[m]);
  }
}

template <int OP, typename WT>
__device__ __forceinline__ void store_values_one(const ElemArgs &a, uint64_t g, const float (&v)[op_values<OP>()][4],
                                                 int k) {
  if (OP == kOpInit) a.master[g] = v[0][k];
  WStore<WT>::one(a.w, g, v[0][k]);
  if constexpr (writes_context<OP>()) store_copies_one<WT>(a.copies, g, v[0][k]);
  if constexpr (OP == kOpPerturbPair) WStore<WT>::one(a.partner, g - a.partner_base, v[1][k]);
  if constexpr (OP == kOpPerturbTwoPairs) {
#pragma unroll
    for (int m = 1; m < 4; ++m) WStore<WT>::one(a.copies.p[m - 1], g, v[m][k]);
  }
}

// The noise words of the group whose counter has the low word q, by folded keys for its high word:
// the launch's, for 0 (LowKeys), or those of another one (HighWord).  Both noise vectors of the
// two pairs share the counter's product M0 q.
struct LowKeys {};
struct HighWord {
  HighKeys k, k_b;
  __device__ __forceinline__ HighWord(const ElemArgs &a, uint32_t q_hi) : k(a.fk, a.rk, q_hi), k_b(a.fk_b, a.rk_b, q_hi) {}
};

template <int OP>
__device__ __forceinline__ void group_words(const ElemArgs &a, LowKeys, uint32_t q, uint32_t (*w)[4]) {
  constexpr int kLast = op_noises<OP>() - 1;
  const uint64_t m = (uint64_t)kPhiloxM0 * q;
  philox4x32_10_folded((uint32_t)m, (uint32_t)(m >> 32), a.fk, w[0]);
  if (kLast) philox4x32_10_folded((uint32_t)m, (uint32_t)(m >> 32), a.fk_b, w[kLast]);
}
template <int OP>
__device__ __forceinline__ void group_words(const ElemArgs &, const HighWord &h, uint32_t q, uint32_t (*w)[4]) {
  constexpr int kLast = op_noises<OP>() - 1;
  const uint64_t m = (uint64_t)kPhiloxM0 * q;
  philox4x32_10_folded((uint32_t)m, (uint32_t)(m >> 32), h.k, w[0]);
  if (kLast) philox4x32_10_folded((uint32_t)m, (uint32_t)(m >> 32), h.k_b, w[kLast]);
}

// One step: the thread's G groups at b + off + 4 kThreads i: their loads, then their Philox
// calls, then their transforms and values.  EDGE: groups outside [b + skip, b + n) are
// generated but neither loaded nor stored.
template <int OP, typename WT, int G, bool EDGE = false, typename Keys>
__device__ __forceinline__ void elem_step(const ElemArgs &a, const Keys &keys, const WideTable &tab, uint64_t b,
                                          uint32_t off, uint32_t skip = 0, uint32_t n = 0) {
  constexpr int NP = op_noises<OP>();
  const float *__restrict__ mt = a.master + b;
  float th[G][4];
#pragma unroll
  for (int i = 0; i < G; ++i) {
    if (OP != kOpInit && (!EDGE || off + 4u * kThreads * i - skip < n - skip)) {
      const float4 v = ld_stream_f4(mt + off + 4u * kThreads * i);
      th[i][0] = v.x, th[i][1] = v.y, th[i][2] = v.z, th[i][3] = v.w;
    } else {
#pragma unroll
      for (int k = 0; k < 4; ++k) th[i][k] = 0.0f;
    }
  }
  uint32_t w[G * NP][4];
  const uint32_t q0 = (uint32_t)(b >> 2);
#pragma unroll
  for (int i = 0; i < G; ++i) group_words<OP>(a, keys, q0 + ((off >> 2) + kThreads * i), &w[i * NP]);
  unsigned long long e2[G * NP][2];
  normals_packed<G * NP>(w, tab, e2);
#pragma unroll
  for (int i = 0; i < G; ++i) {
    if (EDGE && off + 4u * kThreads * i - skip >= n - skip) continue;
    float v[op_values<OP>()][4];
    group_values<OP>(a, &e2[i * NP], th[i], v);
    store_values_full<OP, WT>(a, b + off + 4u * kThreads * i, v);
  }
}

// The elements [b, e) of one group cut by a stretch's end.  Out of line, so that it takes no
// registers from the forms above (with its tests inlined, the pair perturb of 12M elements
// took 21.8 us instead of 18.4).
template <int OP, typename WT, typename Keys>
__device__ __noinline__ void elem_partial_group(const ElemArgs &a, const Keys &keys, const WideTable &tab, uint64_t b,
                                                uint64_t e) {
  const uint64_t g4 = b & ~3ull;
  float th[4];
#pragma unroll
  for (int k = 0; k < 4; ++k) th[k] = (OP != kOpInit && g4 + k >= b && g4 + k < e) ? a.master[g4 + k] : 0.0f;
  constexpr int NP = op_noises<OP>();
  uint32_t w[NP][4];
  group_words<OP>(a, keys, (uint32_t)(g4 >> 2), w);
  unsigned long long e2[NP][2];
  normals_packed<NP>(w, tab, e2);
  float v[op_values<OP>()][4];
  group_values<OP>(a, e2, th, v);
#pragma unroll
  for (int k = 0; k < 4; ++k)
    if (g4 + k >= b && g4 + k < e) store_values_one<OP, WT>(a, g4 + k, v, k);
}

}  // namespace copes
