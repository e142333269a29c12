// pull.cuh -- marking by pull: vertices look for a marked neighbour and stop at
// the first.  Used by the screening (R_t) and the learned screen's pool.
//
// A warp reads the first kPullFirst entries of a row, which decide most rows; who is
// undecided and has more is deferred: its remaining entries become work items of
// kPullChunk, a CTA each, so that a long row without a marked neighbour is spread
// over the chip (a warp on a row of 200,000 entries: 3.7 ms).  Items of a vertex
// that is decided meanwhile return at once.
#pragma once

#include "prims.cuh"
#include "state.cuh"

namespace dcd {

constexpr int kPullFirst = 64;
constexpr int kPullThreads = 256;
constexpr int kPullChunk = 2048;

struct PullRest {
  int32_t* list;   // deferred vertices
  int32_t* found;  // 1: decided
  int64_t* items;  // place in the list << 32 | chunk
  int32_t* cnt;    // [0] vertices, [1] items; zeroed
};

// Device buffers behind it: room for every row above kPullFirst of nnz entries.
struct PullBufs {
  Buf<int32_t> list, found;
  Buf<int64_t> items;
  int alloc(DevMem* m, int64_t n, int64_t nnz, int32_t* cnt, PullRest* out) {
    const int64_t rows = nnz / kPullFirst < n ? nnz / kPullFirst : n;
    DCD_TRY(list.alloc(m, rows + 1));
    DCD_TRY(found.alloc(m, rows + 1));
    DCD_TRY(items.alloc(m, rows + nnz / kPullChunk + 1));
    *out = PullRest{list.get(), found.get(), items.get(), cnt};
    return DCD_OK;
  }
};

// All lanes of a warp call it; more: vertex v of d entries is undecided.
__device__ __forceinline__ void pull_defer(const PullRest& p, bool more, int64_t v, int64_t d) {
  const unsigned bal = __ballot_sync(0xffffffffu, more);
  if (!bal) return;
  const int nch = more ? (int)((d - kPullFirst + kPullChunk - 1) / kPullChunk) : 0;
  const int incl = warp_incl_scan(nch), total = __shfl_sync(0xffffffffu, incl, 31);
  int at = 0, base = 0;
  if (lane_id() == 0) {
    at = atomicAdd(&p.cnt[0], __popc(bal));
    base = atomicAdd(&p.cnt[1], total);
  }
  at = __shfl_sync(0xffffffffu, at, 0) + __popc(bal & lanemask_lt());
  base = __shfl_sync(0xffffffffu, base, 0) + incl - nch;
  if (more) {
    p.list[at] = (int32_t)v;
    p.found[at] = 0;
    for (int x = 0; x < nch; x++) p.items[base + x] = (int64_t)at << 32 | (uint32_t)x;
  }
}

// The deferred entries: out[v] = 1 (and *count one more, when given) where a
// neighbour is marked.
template <typename Marked>
__global__ void __launch_bounds__(kPullThreads) pull_rest(const int64_t* __restrict__ rp,
                                                          const int32_t* __restrict__ col, PullRest p, Marked marked,
                                                          uint8_t* __restrict__ out,
                                                          unsigned long long* __restrict__ count) {
  constexpr int U = kPullChunk / kPullThreads;
  __shared__ int s_found;
  const int n = p.cnt[1];
  for (int i = blockIdx.x; i < n; i += gridDim.x) {
    const int64_t it = p.items[i];
    const int at = (int)(it >> 32);
    if (threadIdx.x == 0) s_found = *(volatile const int32_t*)&p.found[at];
    __syncthreads();
    if (s_found) {
      __syncthreads();
      continue;
    }
    const int32_t v = p.list[at];
    const int64_t b = rp[v] + kPullFirst + (int64_t)(uint32_t)it * kPullChunk, e1 = rp[v + 1];
    int32_t x[U];
#pragma unroll
    for (int q = 0; q < U; q++) {
      const int64_t e = b + q * kPullThreads + threadIdx.x;
      x[q] = e < e1 ? col[e] : -1;
    }
    bool hit = false;
#pragma unroll
    for (int q = 0; q < U; q++) hit |= x[q] >= 0 && marked(x[q]);
    if (__syncthreads_or(hit) && threadIdx.x == 0 && atomicExch(&p.found[at], 1) == 0) {
      out[v] = 1;
      if (count) atomicAdd(count, 1ull);
    }
  }
}

}  // namespace dcd
