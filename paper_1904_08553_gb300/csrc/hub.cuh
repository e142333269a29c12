// hub.cuh -- aggregation of very long rows (hubs) over many CTAs, shared by
// the local-move kernels and the screening kernels.
//
// A hub's row is split into chunks of kHubChunk entries, a CTA each, so that
// many CTAs work on one hub at once.  Each hub owns a region of a global
// open-addressing table (capacity: 2 x degree rounded up to a power of two, so
// probing always ends) and of a list of the slots it claimed:
//   hub_agg   chunk c of hub h: the chunk is summed by community in a table in
//             shared memory (the hub's own community in registers), whose
//             distinct sums are then added into h's table, listing new keys.
// The caller then reads the tables (gains, lookups) and, to reuse them,
// empties the claimed slots.  The view V has rp, col, w, L and nlab (labels in
// entry order, or NULL).
#pragma once

#include "agg.cuh"
#include "state.cuh"

namespace dcd {

// A chunk is one load round of a CTA: every thread has its kHubItems entries in
// flight at once.  With 4096 entries a chunk (16 dependent rounds, each ending
// in global atomics) a few dozen hubs took 53-85 us a pass whatever their size;
// now 25-39 us.
constexpr int64_t kHubChunk = 1024;
constexpr int kHubThreads = 256;
constexpr int kHubItems = (int)kHubChunk / kHubThreads;
constexpr int kHubCap = 2 * (int)kHubChunk;

struct HubTables {
  const int32_t* list = nullptr;  // hub vertices (the bin's list segment)
  int64_t H = 0;                  // hubs
  const int64_t* toff = nullptr;  // table offset of hub h (H + 1)
  const int64_t* soff = nullptr;  // claimed-slot list offset of hub h (H + 1)
  const int64_t* coff = nullptr;  // first chunk of hub h (H + 1)
  int32_t* keys = nullptr;        // all tables (-1: empty)
  unsigned long long* vals = nullptr;
  int32_t* slots = nullptr;       // claimed-slot lists (table-relative slot)
  int32_t* nslot = nullptr;       // claimed slots of hub h (this pass)
  int32_t* nprev = nullptr;       // the same, kept for hub_clear
  long long* part = nullptr;      // per chunk: gain (2 words), label
};

__device__ __forceinline__ int64_t hub_of_chunk(const HubTables& t, int64_t c) {
  int64_t lo = 0, hi = t.H - 1;
  while (lo < hi) {
    const int64_t mid = (lo + hi + 1) >> 1;
    if (t.coff[mid] <= c) lo = mid; else hi = mid - 1;
  }
  return lo;
}

template <typename W, typename ST, typename V>
__global__ void __launch_bounds__(kHubThreads) hub_agg(V g, HubTables t) {
  using VT = typename TblVal<ST>::type;
  __shared__ int32_t sk[kHubCap];
  __shared__ VT sv[kHubCap];
  __shared__ uint16_t ss[kHubChunk];
  __shared__ int32_t s_n;
  const int tid = threadIdx.x;
  for (int x = tid; x < kHubCap; x += kHubThreads) {
    sk[x] = -1;
    sv[x] = 0;
  }
  if (tid == 0) s_n = 0;
  __syncthreads();
  const int64_t nch = t.coff[t.H];
  for (int64_t c = blockIdx.x; c < nch; c += gridDim.x) {
    const int64_t h = hub_of_chunk(t, c);
    const int32_t v = t.list[h];
    const int64_t b = g.rp[v], d = g.rp[v + 1] - b;
    const int64_t e0 = (c - t.coff[h]) * kHubChunk;
    const int32_t C = g.L[v];
    const uint32_t mask = (uint32_t)(t.toff[h + 1] - t.toff[h]) - 1;
    int32_t* keys = t.keys + t.toff[h];
    unsigned long long* vals = t.vals + t.toff[h];
    int32_t* slots = t.slots + t.soff[h];
    int32_t lab[kHubItems];
    W wt[kHubItems];
#pragma unroll
    for (int q = 0; q < kHubItems; q++) {
      const int64_t e = e0 + q * kHubThreads + tid;
      lab[q] = -1;
      wt[q] = W(0);
      if (e < d) {
        lab[q] = ld_stream((g.nlab ? g.nlab : g.col) + b + e);
        wt[q] = ld_stream(g.w + b + e);
      }
    }
    if (!g.nlab) {
#pragma unroll
      for (int q = 0; q < kHubItems; q++) {
        const int32_t u = lab[q];
        lab[q] = (u >= 0 && u != v) ? g.L[u] : -1;
      }
    }
    VT own = 0;
#pragma unroll
    for (int q = 0; q < kHubItems; q++) {
      bool claimed = false;
      uint32_t s = 0;
      if (lab[q] == C) {
        own += (VT)wt[q];
      } else if (lab[q] >= 0) {
        s = probe_claim(sk, kHubCap - 1, lab[q], claimed);
        atomicAdd(&sv[s], (VT)wt[q]);
      }
      const unsigned bal = __ballot_sync(0xffffffffu, claimed);
      int at = 0;
      if (lane_id() == 0 && bal) at = atomicAdd(&s_n, __popc(bal));
      at = __shfl_sync(0xffffffffu, at, 0);
      if (claimed) ss[at + __popc(bal & lanemask_lt())] = (uint16_t)s;
    }
    __syncthreads();
    const int nd = s_n;
    const VT ow = (VT)seg_total<32>(own);
    // the warps' own-community sums go into the table directly, behind the
    // chunk's distinct sums
    for (int x0 = tid & ~31; x0 < nd || (x0 == (tid & ~31)); x0 += kHubThreads) {
      const int x = x0 + (int)lane_id();
      int32_t key = -1;
      unsigned long long val = 0;
      if (x < nd) {
        const uint32_t s = ss[x];
        key = sk[s];
        val = sv[s];
        sk[s] = -1;
        sv[s] = 0;
      }
      for (int round = 0; round < 2; round++) {
        if (round == 1) {  // once per warp: its own-community sum
          if (x0 != (tid & ~31)) break;
          key = (lane_id() == 0 && ow) ? C : -1;
          val = ow;
        }
        bool fresh = false;
        uint32_t sl = 0;
        if (key >= 0) {
          sl = hash_label(key, mask);
          for (;;) {
            const int32_t k = keys[sl];
            if (k == key) break;
            if (k == -1) {
              const int32_t old = atomicCAS(&keys[sl], -1, key);
              if (old == -1) fresh = true;
              if (old == -1 || old == key) break;
            }
            sl = (sl + 1) & mask;
          }
          atomicAdd(&vals[sl], val);
        }
        const unsigned bal = __ballot_sync(0xffffffffu, fresh);
        int at = 0;
        if (lane_id() == 0 && bal) at = atomicAdd(&t.nslot[h], __popc(bal));
        at = __shfl_sync(0xffffffffu, at, 0);
        if (fresh) slots[at + __popc(bal & lanemask_lt())] = (int32_t)sl;
      }
    }
    __syncthreads();
    if (tid == 0) s_n = 0;
    __syncthreads();
  }
}

// sizes of the hub tables (hub h: table 2 x degree rounded up to a power of
// two, slot list = degree, chunks = degree / kHubChunk rounded up)
template <int UNUSED>
__global__ void hub_sizes(const int32_t* __restrict__ list, int64_t H, const int64_t* __restrict__ rp,
                          int64_t* __restrict__ cap, int64_t* __restrict__ deg, int64_t* __restrict__ nch) {
  for (int64_t h = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; h < H; h += (int64_t)gridDim.x * blockDim.x) {
    const int32_t v = list[h];
    const int64_t d = rp[v + 1] - rp[v];
    cap[h] = table_cap(d);
    deg[h] = d;
    nch[h] = cdiv(d, kHubChunk);
  }
}

// Device buffers behind a HubTables view (step arena).
struct HubBufs {
  Buf<int64_t> toff, soff, coff;
  Buf<int32_t> keys, slots, nslot, nprev;
  Buf<unsigned long long> vals;
  Buf<long long> part;
  int64_t chunks = 0;
  HubTables t;
};

// louvain.cu: sizes, offsets and empty tables for the H hubs of list.
int hub_setup(dcd_ctx* c, const int32_t* list, int64_t H, const int64_t* rp, HubBufs* b);
// CTAs for a launch over the hubs' chunks.
unsigned hub_grid(dcd_ctx* c, const HubBufs& b);

}  // namespace dcd
