// agg.cuh -- neighbour-community aggregation shared by the local-move and
// screening kernels: exact group sums inside a warp, open-addressing tables
// (community label -> summed edge weight) in shared or global memory, the
// exact integer gain S and a total-order argmax.
#pragma once

#include <climits>

#include "common.cuh"

namespace dcd {

// Gain of moving v from C to D (Sec. III-A; expanded form in the appendix
// proof of Lemma 3.2):  S = m2 (e_{v->D} - e_{v->C\v}) - k_v (a_D - (a_C - k_v)),
// i.e. (2m)^2 times the paper's Delta Q_{v->D}.  ST = int64 is exact when
// m2 < 2^31 (both products stay below 2^62); otherwise ST = int128.
template <typename ST>
__device__ __forceinline__ ST gain(int64_t m2, int64_t kv, int64_t eD, int64_t eC, int64_t aD, int64_t aC) {
  return (ST)m2 * (ST)(eD - eC) - (ST)kv * (ST)(aD - aC + kv);
}

// No community can gain S > 0 for v: of S, e_{v->D} is at most k_v - e_{v->C\v}
// and a_D at least 0, so S <= m2 (k_v - 2 e_{v->C\v}) + k_v (a_C - k_v).  Exact (64
// bits hold both products and, each below 2^62, their sum), and known before the
// row is summed by community: true for most vertices once the labels settle.
template <typename ST>
__device__ __forceinline__ bool stays(int64_t m2, int64_t kv, int64_t eC, int64_t aC) {
  return (ST)m2 * (ST)(kv - 2 * eC) + (ST)kv * (ST)(aC - kv) <= 0;
}

template <typename ST>
__device__ __forceinline__ ST gain_lowest();
template <>
__device__ __forceinline__ long long gain_lowest<long long>() {
  return LLONG_MIN;
}
template <>
__device__ __forceinline__ i128 gain_lowest<i128>() {
  return -((i128)1 << 126) * 2;
}

__device__ __forceinline__ long long shfl_xor_st(long long x, int o) { return __shfl_xor_sync(0xffffffffu, x, o); }
__device__ __forceinline__ i128 shfl_xor_st(i128 x, int o) {
  unsigned long long lo = (unsigned long long)x, hi = (unsigned long long)(x >> 64);
  lo = __shfl_xor_sync(0xffffffffu, lo, o);
  hi = __shfl_xor_sync(0xffffffffu, hi, o);
  return (i128)(((unsigned __int128)hi << 64) | lo);
}
__device__ __forceinline__ long long shfl_st(long long x, int src) { return __shfl_sync(0xffffffffu, x, src); }
__device__ __forceinline__ i128 shfl_st(i128 x, int src) {
  unsigned long long lo = (unsigned long long)x, hi = (unsigned long long)(x >> 64);
  lo = __shfl_sync(0xffffffffu, lo, src);
  hi = __shfl_sync(0xffffffffu, hi, src);
  return (i128)(((unsigned __int128)hi << 64) | lo);
}

// The move a vertex in community C proposes from its best (S, D) over the
// neighbouring communities D != C (Algorithm 1's rule, synchronous reading):
// move iff S > 0 (staying wins ties); a singleton does not move into a
// singleton of larger label (the minimum-label guard against two singletons
// swapping).  size: community sizes under the pass's snapshot.
template <typename ST>
__device__ __forceinline__ int32_t move_proposal(ST S, int32_t D, int32_t C, const int32_t* size) {
  const bool mv = D != INT_MAX && S > 0;
  const int32_t Dm = mv ? D : C;
  const int32_t sC = size[C], sD = size[Dm];
  return (mv && sC == 1 && sD == 1 && Dm > C) ? C : Dm;
}

// (S, D) order of the greedy choice: larger gain first, then smaller label.
template <typename ST>
__device__ __forceinline__ bool better(ST s1, int32_t d1, ST s2, int32_t d2) {
  return s1 > s2 || (s1 == s2 && d1 < d2);
}

// Whole-warp argmax of (S, D); every lane ends with the result (128-bit gains).
__device__ __forceinline__ void warp_argmax(i128& S, int32_t& D) {
  using ST = i128;
#pragma unroll
  for (int o = 16; o > 0; o >>= 1) {
    ST s2 = shfl_xor_st(S, o);
    int32_t d2 = __shfl_xor_sync(0xffffffffu, D, o);
    if (better(s2, d2, S, D)) {
      S = s2;
      D = d2;
    }
  }
}

// Whole-warp argmax of (S, D) for 64-bit gains with redux.sync over the full
// warp: the maximum of the high words, then of the low words among the lanes
// holding that high word, then the smallest label among the lanes holding
// the maximum (labels are >= 0, the sentinel INT_MAX).  Lanes outside each
// step contribute the neutral value, so no lane diverges.
__device__ __forceinline__ void warp_argmax(long long& S, int32_t& D) {
  const unsigned long long u = (unsigned long long)S ^ 0x8000000000000000ull;
  const unsigned hi = (unsigned)(u >> 32), lo = (unsigned)u;
  const unsigned mhi = __reduce_max_sync(0xffffffffu, hi);
  const unsigned mlo = __reduce_max_sync(0xffffffffu, hi == mhi ? lo : 0u);
  const bool top = hi == mhi && lo == mlo;
  const unsigned dmin = __reduce_min_sync(0xffffffffu, top ? (unsigned)D : 0xffffffffu);
  S = (long long)((((unsigned long long)mhi << 32) | mlo) ^ 0x8000000000000000ull);
  D = (int32_t)dmin;
}

// Argmax of (S, D) over the SEG-lane segment of the calling lane, all lanes of
// the warp calling.  Below a whole warp it runs on shuffles: a redux over a
// part of the warp executes once per segment, one after another, where the
// shuffles take all segments in the same instruction.
template <int SEG, typename ST>
__device__ __forceinline__ void seg_argmax(ST& S, int32_t& D) {
  if constexpr (SEG == 32) {
    warp_argmax(S, D);
  } else {
#pragma unroll
    for (int o = SEG / 2; o > 0; o >>= 1) {
      const ST s2 = shfl_xor_st(S, o);
      const int32_t d2 = __shfl_xor_sync(0xffffffffu, D, o);
      if (better(s2, d2, S, D)) {
        S = s2;
        D = d2;
      }
    }
  }
}

// Exact sum of non-negative weights over the lanes of `peers` (a match_any
// group), from 16-bit slices reduced with redux.sync: no slice sum can carry
// out of 32 bits, so the result is exact for any int64 weight.
__device__ __forceinline__ int64_t group_sum_exact(unsigned peers, int64_t w) {
  unsigned long long x = (unsigned long long)w;
  int64_t s = 0;
#pragma unroll
  for (int q = 0; q < 4; q++) {
    unsigned part = (unsigned)(x >> (16 * q)) & 0xffffu;
    s += (int64_t)__reduce_add_sync(peers, part) << (16 * q);
  }
  return s;
}

// ---- open-addressing table: key -1 = empty; capacity a power of two that is
// at least twice the number of distinct keys, so probing always ends. ----
template <typename VT>
__device__ __forceinline__ int64_t tbl_get(const int32_t* keys, const VT* vals, uint32_t mask, int32_t lab) {
  uint32_t s = hash_label(lab, mask);
  for (;;) {
    int32_t k = keys[s];
    if (k == lab) return (int64_t)vals[s];
    if (k == -1) return 0;
    s = (s + 1) & mask;
  }
}

// Width of the shared-table sums: with 64-bit gains 2m < 2^31 bounds every
// sum of a vertex's weights, so 32 bits hold them exactly (smaller tables,
// more warps per SM); with 128-bit gains the sums are 64-bit.
template <typename ST>
struct TblVal {
  using type = unsigned long long;
};
template <>
struct TblVal<long long> {
  using type = unsigned;
};

// The slot of `lab` in the table (claimed when absent); `claimed` is set when
// this call took an empty slot for it.
__device__ __forceinline__ uint32_t probe_claim(int32_t* keys, uint32_t mask, int32_t lab, bool& claimed) {
  uint32_t s = hash_label(lab, mask);
  for (;;) {
    const int32_t k = keys[s];
    if (k == lab) return s;
    if (k == -1) {
      const int32_t old = atomicCAS(&keys[s], -1, lab);
      if (old == -1) {
        claimed = true;
        return s;
      }
      if (old == lab) return s;
    }
    s = (s + 1) & mask;
  }
}

// Sum over the S lanes of the calling lane's segment, all lanes of the warp
// calling: 32-bit sums are exact with 64-bit gains (every sum of a vertex's
// weights is below 2m < 2^31), 64-bit sums with 128-bit gains.
template <int S>
__device__ __forceinline__ int64_t seg_total(unsigned x) {
  if constexpr (S == 32) {
    return (int64_t)__reduce_add_sync(0xffffffffu, x);
  } else {
#pragma unroll
    for (int o = S / 2; o > 0; o >>= 1) x += __shfl_xor_sync(0xffffffffu, x, o);
    return (int64_t)x;
  }
}
template <int S>
__device__ __forceinline__ int64_t seg_total(unsigned long long x) {
#pragma unroll
  for (int o = S / 2; o > 0; o >>= 1) x += __shfl_xor_sync(0xffffffffu, x, o);
  return (int64_t)x;
}

__host__ __device__ __forceinline__ uint32_t table_cap(int64_t deg) {
  uint32_t c = 64;
  while ((int64_t)c < 2 * deg) c <<= 1;
  return c;
}

// ---- 128-bit sums and the stop rule ----
__device__ __forceinline__ void add128(unsigned long long* lo, unsigned long long* hi, unsigned __int128 v) {
  const unsigned long long vlo = (unsigned long long)v, vhi = (unsigned long long)(v >> 64);
  if (!(vlo | vhi)) return;
  const unsigned long long old = atomicAdd(lo, vlo);
  const unsigned long long carry = (old + vlo < old) ? 1ull : 0ull;
  if (vhi + carry) atomicAdd(hi, vhi + carry);
}

__device__ __forceinline__ bool below_tau(i128 gain, i128 base, int64_t tau_inv) {
  // gain <= floor(|base| / tau_inv), without the 128-bit division where the
  // product fits (tau_inv < 2^31)
  const i128 y = base < 0 ? -base : base;
  if (gain <= 0) return true;
  if (gain < ((i128)1 << 95)) return gain * (i128)tau_inv <= y;
  return gain <= y / (i128)tau_inv;
}

__device__ __forceinline__ i128 ld128(const int64_t* lo) {
  return (i128)(((unsigned __int128)(unsigned long long)lo[1] << 64) | (unsigned long long)lo[0]);
}
__device__ __forceinline__ void st128(int64_t* lo, i128 x) {
  lo[0] = (int64_t)(unsigned long long)x;
  lo[1] = (int64_t)(unsigned long long)((unsigned __int128)x >> 64);
}

}  // namespace dcd
