// rows.cuh -- shared-memory layouts for summing one row by community, used by
// the local move and by the screening (louvain.cu describes both schemes).
#pragma once

#include "agg.cuh"

namespace dcd {

// ---- table: at least twice the row, so every probe sequence ends ----

__host__ __device__ constexpr int seg_cap(int row) {
  int c = 32;
  while (c < 2 * row) c <<= 1;
  return c;
}

// Shared memory of one row table: keys (int32), sums (VT), the claimed-slot
// list (one uint16 per row entry); a multiple of 16 bytes.
template <int ROW, typename VT>
__host__ __device__ constexpr size_t row_tbl_bytes() {
  return ((size_t)seg_cap(ROW) * (4 + sizeof(VT)) + (size_t)ROW * 2 + 15) / 16 * 16;
}

// ---- lists ----

template <typename VT>
struct ListEnt;  // a list entry: one shared-memory word of 8 or 16 bytes
template <>
struct __align__(8) ListEnt<unsigned> {
  int32_t lab;
  unsigned w;
};
template <>
struct __align__(16) ListEnt<unsigned long long> {
  unsigned long long w;
  int32_t lab, pad;
};

constexpr int kCap32 = 16;  // foreign entries a lane's list holds, rows of 17 to 32 entries

// Shared memory of a warp: the lanes' lists, then (rows can be longer than
// CAP) a whole-row list per segment with two entries of padding.
template <int S, int Q, int CAP, typename VT>
__host__ __device__ constexpr size_t vert_bytes() {
  return (size_t)CAP * 32 * sizeof(ListEnt<VT>) +
         (S * Q > CAP ? (size_t)(32 / S) * (S * Q + 2) * sizeof(ListEnt<VT>) : 0);
}

// One segment's whole list: each lane takes K entries and sums the list's
// weights of the same community (entries of one community get the same sum and
// gain, so none has to be singled out).  All lanes of the warp call it; every
// list is padded to nmax, made even.
template <typename V, typename ST, int S, int K, typename VT>
__device__ __forceinline__ void list_best(const V& g, const ListEnt<VT>* list, int n, int nmax, int64_t kv,
                                          int64_t eC, int64_t aC, int64_t m2v, int sl, ST& Sb, int32_t& D,
                                          int64_t& eD) {
  int32_t l[K];
  VT e[K];
#pragma unroll
  for (int k = 0; k < K; k++) {
    l[k] = k * S + sl < n ? list[k * S + sl].lab : -1;
    e[k] = 0;
  }
  for (int j = 0; j < nmax; j += 2) {
    const ListEnt<VT> x = list[j], y = list[j + 1];
#pragma unroll
    for (int k = 0; k < K; k++) {
      if (x.lab == l[k]) e[k] += x.w;
      if (y.lab == l[k]) e[k] += y.w;
    }
  }
#pragma unroll
  for (int k = 0; k < K; k++)
    if (l[k] >= 0) {
      const ST x = gain<ST>(m2v, kv, (int64_t)e[k], eC, g.a[l[k]], aC);
      if (better(x, l[k], Sb, D)) {
        Sb = x;
        D = l[k];
      }
    }
  seg_argmax<S>(Sb, D);
  eD = 0;
#pragma unroll
  for (int k = 0; k < K; k++)
    if (l[k] == D) eD = (int64_t)e[k];
#pragma unroll
  for (int o = S / 2; o > 0; o >>= 1) {  // known where an entry is in D; equal there
    const int64_t x = __shfl_xor_sync(0xffffffffu, eD, o);
    eD = x > eD ? x : eD;
  }
}

}  // namespace dcd
