// rows.cuh -- shared-memory layouts for summing one row by community, used by
// the local move and by the screening (louvain.cu describes both schemes), and
// the walk over entries in CSR order whatever rows they belong to.
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

// ---- entry-linear walks ----

// Row of entry e for entry-linear walks: a warp walks a range of
// consecutive entries, finds the row of its first entry by binary search,
// then advances 32 entries at a time with the row ends of the next 32 rows
// in its lanes.
struct RowWalk {
  int64_t r;     // row of the chunk's first entry
  int64_t rb;    // lane i holds the end of row rb + i (valid while chunks stay below `last`)
  int64_t bk, last;
  __device__ __forceinline__ void load(const int64_t* __restrict__ rp, int64_t n, int64_t r0) {
    rb = r0;
    bk = (r0 + 1 + lane_id() <= n) ? rp[r0 + 1 + lane_id()] : INT64_MAX;
    last = __shfl_sync(0xffffffffu, bk, 31);
  }
  __device__ __forceinline__ void start(const int64_t* __restrict__ rp, int64_t n, int64_t E0) {
    int64_t x = 0;
    if (lane_id() == 0) {  // last row whose start is <= E0
      int64_t lo = 0, hi = n - 1;
      while (lo < hi) {
        const int64_t mid = (lo + hi + 1) >> 1;
        if (rp[mid] <= E0) lo = mid; else hi = mid - 1;
      }
      x = lo;
    }
    r = __shfl_sync(0xffffffffu, x, 0);
    load(rp, n, r);
  }
  // row of entry c0 + lane (entries past the segment get the last row); the
  // ends of 32 rows stay in the lanes across chunks and are reloaded only when
  // a chunk runs past them
  __device__ __forceinline__ int64_t row(const int64_t* __restrict__ rp, int64_t n, int64_t c0, bool valid) {
    const int lane = lane_id();
    const int64_t e = c0 + lane;
    if (last <= c0 + 31) load(rp, n, r);
    int64_t rw;
    if (last <= c0 + 31) {
      // more than 31 rows end inside this chunk (empty rows): search per lane
      int64_t lo = r, hi = n - 1, x = valid ? e : c0;
      while (lo < hi) {
        const int64_t mid = (lo + hi + 1) >> 1;
        if (rp[mid] <= x) lo = mid; else hi = mid - 1;
      }
      rw = lo;
    } else {
      int cntv = 0;
      const int64_t x = valid ? e : c0;
#pragma unroll
      for (int step = 16; step > 0; step >>= 1) {
        const int64_t v = __shfl_sync(0xffffffffu, bk, cntv + step - 1);
        if (v <= x) cntv += step;
      }
      rw = rb + cntv;
    }
    r = __shfl_sync(0xffffffffu, rw, 31);
    return rw;
  }
};

}  // namespace dcd
