// bins.cuh -- degree bins: how many of the wanted vertices fall in each bin of
// a plan, and the vertices listed bin by bin.  Shared by the local move (the
// active vertices of a level) and the screening (the sources of a batch).
#pragma once

#include "agg.cuh"
#include "prims.cuh"
#include "state.cuh"

namespace dcd {

// The vertices wanted: active ones of graphs that still run ...
struct WantActive {
  static constexpr bool kEmptyRows = false;  // a vertex without entries has nothing to choose
  const uint8_t* active;  // NULL: all
  const int32_t* gid;
  const GraphState* gs;
  __device__ __forceinline__ bool operator()(int64_t v) const {
    return (!active || active[v]) && (!gid || gs[gid[v]].running);
  }
  __device__ __forceinline__ int64_t size(int64_t, int64_t deg) const { return deg; }
};
// ... or the sources of the batch's pairs, whose kernels walk over the pairs as
// well as the row: a vertex that lost its edges, or whose edges the batch repeats,
// has many pairs and a short row, and takes the kernel its pairs want (to the
// largest one with a table in shared memory; the hub kernels are for long rows).
struct WantSource {
  static constexpr bool kEmptyRows = true;  // a source may have lost its last edge: its deletes still mark
  const int32_t* pair_ptr;
  __device__ __forceinline__ bool operator()(int64_t v) const { return pair_ptr[v + 1] > pair_ptr[v]; }
  __device__ __forceinline__ int64_t size(int64_t v, int64_t deg) const {
    const int64_t p = pair_ptr[v + 1] - pair_ptr[v], most = lm_variant_max(kLmCta4k);
    const int64_t q = p < most ? p : most;
    return deg > q ? deg : q;
  }
};

// Wanted vertices per bin (of the size Want gives them), their degree sums and largest degree
// (DevScalars bcnt, bdeg, bmax; all of them, rows without entries included:
// ncomm and act_deg).  Lane b of a warp keeps bin b's figures in registers: a
// ballot and two reductions per bin and 32 vertices, no shared-memory traffic
// until the end.
template <typename Want>
__global__ void __launch_bounds__(256) bin_count(const int64_t* __restrict__ rp, int64_t n, Want want, DevScalars* d,
                                                 BinPlan plan, const int32_t* __restrict__ pre) {
  __shared__ unsigned long long s_cnt[kMaxBins], s_deg[kMaxBins];
  __shared__ unsigned s_max[kMaxBins];
  const int lane = lane_id();
  if (threadIdx.x < kMaxBins) {
    s_cnt[threadIdx.x] = 0;
    s_deg[threadIdx.x] = 0;
    s_max[threadIdx.x] = 0;
  }
  __syncthreads();
  unsigned long long cnt = 0, dsum = 0, deg_sum = 0, act = 0, pre_deg = 0, pre_cnt = 0;
  unsigned dmax = 0;
  const int64_t stride = (int64_t)gridDim.x * blockDim.x;
  for (int64_t base = (blockIdx.x * (int64_t)blockDim.x) + (threadIdx.x & ~31); base < n; base += stride) {
    const int64_t v = base + lane;
    const bool ok = v < n && want(v);
    if (!__any_sync(0xffffffffu, ok)) continue;
    const unsigned deg = ok ? (unsigned)(rp[v + 1] - rp[v]) : 0u;  // columns are int32: a row has fewer than 2^31
    deg_sum += deg;
    act += ok ? 1 : 0;
    const int bin = ok && (deg > 0 || Want::kEmptyRows) ? bin_of(plan, want.size(v, deg)) : -1;
    // a first-pass proposal from the screening, which the table kernels take
    // (the hub kernels evaluate their rows all the same)
    if (pre && deg > 0 && pre[v] >= 0 && plan.var[bin] != kLmHub) {
      pre_deg += deg;
      pre_cnt += 1;
    }
    const bool wide = __any_sync(0xffffffffu, deg >= (1u << 26));  // 32 of them may pass 2^32
    for (int b = 0; b < plan.nb; b++) {
      const unsigned bal = __ballot_sync(0xffffffffu, bin == b);
      if (!bal) continue;
      const unsigned x = bin == b ? deg : 0u;
      unsigned long long sum = wide ? (unsigned long long)__reduce_add_sync(0xffffffffu, x & 0xffffu) +
                                          ((unsigned long long)__reduce_add_sync(0xffffffffu, x >> 16) << 16)
                                    : (unsigned long long)__reduce_add_sync(0xffffffffu, x);
      const unsigned mx = __reduce_max_sync(0xffffffffu, x);
      if (lane == b) {
        cnt += __popc(bal);
        dsum += sum;
        dmax = mx > dmax ? mx : dmax;
      }
    }
  }
  if (lane < plan.nb && cnt) {
    atomicAdd(&s_cnt[lane], cnt);
    atomicAdd(&s_deg[lane], dsum);
    atomicMax(&s_max[lane], dmax);
  }
  deg_sum = warp_sum(deg_sum);
  act = warp_sum(act);
  if (pre) {
    pre_deg = warp_sum(pre_deg);
    pre_cnt = warp_sum(pre_cnt);
    if (lane == 0 && pre_cnt) {
      atomicAdd((unsigned long long*)&d->pre_deg, pre_deg);
      atomicAdd((unsigned long long*)&d->pre_verts, pre_cnt);
    }
  }
  if (lane == 0 && act) {
    atomicAdd((unsigned long long*)&d->act_deg, deg_sum);
    atomicAdd((unsigned long long*)&d->ncomm, act);
  }
  __syncthreads();
  if (threadIdx.x < plan.nb && s_cnt[threadIdx.x]) {
    const int b = threadIdx.x;
    atomicAdd((unsigned long long*)&d->bcnt[b], s_cnt[b]);
    atomicAdd((unsigned long long*)&d->bdeg[b], s_deg[b]);
    atomicMax((long long*)&d->bmax[b], (long long)s_max[b]);
  }
}

// The wanted vertices, bin after bin (bin b starts where the
// counts of the bins before it end).  A CTA places a block of consecutive
// vertices: ranks within the block in shared memory, then one reservation per
// bin and block in global memory, so that the cursors are not the bottleneck
// (a reservation per warp and bin took 195 us for 2 M vertices, this 20) and a
// bin's list stays close to vertex order.
constexpr int kBinThreads = 256;
// Vertices a thread: few small blocks leave a small graph to a handful of SMs
// (10 K vertices: 12 us with 8 a thread, 4 with 1).
constexpr int kBinItems = 8;
constexpr int64_t kBinSmall = (int64_t)1 << 18;
template <typename Want, int ITEMS>
__global__ void __launch_bounds__(kBinThreads) bin_scatter(const int64_t* __restrict__ rp, int64_t n, Want want,
                                                           const DevScalars* __restrict__ d,
                                                           int32_t* __restrict__ cursor, int32_t* __restrict__ list,
                                                           BinPlan plan) {
  __shared__ int32_t s_cnt[kMaxBins], s_base[kMaxBins];
  const int tid = threadIdx.x;
  const int64_t block = (int64_t)kBinThreads * ITEMS;
  for (int64_t v0 = blockIdx.x * block; v0 < n; v0 += gridDim.x * block) {
    if (tid < kMaxBins) s_cnt[tid] = 0;
    __syncthreads();
    int bin[ITEMS], rank[ITEMS];
#pragma unroll
    for (int i = 0; i < ITEMS; i++) {
      const int64_t v = v0 + i * kBinThreads + tid;
      bin[i] = -1;
      if (v < n && want(v)) {
        const int64_t deg = rp[v + 1] - rp[v];
        if (deg > 0 || Want::kEmptyRows) bin[i] = bin_of(plan, want.size(v, deg));
      }
    }
#pragma unroll
    for (int i = 0; i < ITEMS; i++) {
      const unsigned peers = __match_any_sync(0xffffffffu, bin[i]);
      int at = 0;
      const int lead = __ffs(peers) - 1;
      if (bin[i] >= 0 && lead == (int)lane_id()) at = atomicAdd(&s_cnt[bin[i]], __popc(peers));
      rank[i] = __shfl_sync(0xffffffffu, at, lead) + __popc(peers & lanemask_lt());
    }
    __syncthreads();
    if (tid < plan.nb) {
      int64_t o = 0;
#pragma unroll
      for (int b = 0; b < kMaxBins - 1; b++) o += b < tid ? d->bcnt[b] : 0;
      s_base[tid] = (int32_t)o + (s_cnt[tid] ? atomicAdd(&cursor[tid], s_cnt[tid]) : 0);
    }
    __syncthreads();
#pragma unroll
    for (int i = 0; i < ITEMS; i++)
      if (bin[i] >= 0) list[s_base[bin[i]] + rank[i]] = (int32_t)(v0 + i * kBinThreads + tid);
    __syncthreads();
  }
}

template <typename Want>
void launch_bin_scatter(cudaStream_t s, const int64_t* rp, int64_t n, const Want& want, const DevScalars* d,
                        int32_t* cursor, int32_t* list, const BinPlan& plan) {
  if (n < kBinSmall)
    count_launch(), bin_scatter<Want, 1><<<grid_for(n, kBinThreads), kBinThreads, 0, s>>>(rp, n, want, d, cursor, list,
                                                                                          plan);
  else
    count_launch(), bin_scatter<Want, kBinItems><<<grid_for(cdiv(n, kBinItems), kBinThreads), kBinThreads, 0, s>>>(
        rp, n, want, d, cursor, list, plan);
}

}  // namespace dcd
