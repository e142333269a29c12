// noalloc.cu -- dcd_modularity_noalloc: modularity of a partition on a
// caller-owned device CSR, computed without allocating any device memory.
//
// Why it exists: some callers cannot allocate device memory at the moment
// they need an answer -- code whose device memory is already fully reserved
// by another allocator (a framework's caching allocator holding the free
// memory), code running where cudaMalloc/cudaFree must not be called (a host
// callback on a stream) or must not add their implicit synchronisation.  This
// entry point takes its scratch (community degree sums and reduction
// partials) from one fixed array in device memory that the library reserves
// at load time, on every GPU that loads it, until the process exits.
//
// Limits and sharing: at most kNoAllocMaxN labels (the array holds 8 MiB).
// Every call on a device uses the same array and leaves its contents behind;
// each call clears what it needs first, so consecutive calls are independent,
// but two calls whose device work overlaps (different streams, or different
// host threads) race on the array and give wrong results.
#include <cstring>

#include "prims.cuh"
#include "state.cuh"

namespace dcd {
namespace {

constexpr int64_t kNoAllocWords = (int64_t)1 << 20;  // 8 MiB of 64-bit words
constexpr int kNoAllocCtas = 256;                     // partials of the sum of squares
constexpr int64_t kNoAllocTail = 8;                   // m2, in, N lo/hi, error word
constexpr int64_t kNoAllocMaxN = kNoAllocWords - 2 * kNoAllocCtas - kNoAllocTail;

static __device__ __align__(256) unsigned long long g_noalloc_scratch[kNoAllocWords];

// tail words: [0] m2, [1] in, [2] N lo, [3] N hi, [4] error flag
__global__ void na_clear(unsigned long long* s, int64_t n) {
  for (int64_t i = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; i < n; i += (int64_t)gridDim.x * blockDim.x)
    s[i] = 0;
  if (blockIdx.x == 0 && threadIdx.x < kNoAllocTail) s[kNoAllocWords - kNoAllocTail + threadIdx.x] = 0;
}

// Per row u: d_w(u), the intra-community weight of the row, and a_C += d_w(u).
//
// Bound by the gather of a label per entry, a 32-byte sector each (a bare gather
// of as many runs at 250 G sectors/s).  A CTA takes 256 consecutive rows: bounds
// and labels coalesced, then 8 lanes a row (4 rows a warp step) with 8 entries a
// lane in flight, and rows above kNaLong entries by the whole CTA: 255 us for
// 1 M rows and 42 M entries (16 or 32 lanes a row: 275-330).  A warp a row, one
// entry a lane in flight, took 635 us.
constexpr int kNaThreads = 256, kNaGroup = 8, kNaUnroll = 8, kNaLong = 512;

// Entries [e0, e1) of a row with label Lu by `step` threads, kNaUnroll at once.
__device__ __forceinline__ void na_entries(int64_t e0, int64_t e1, int step, int64_t n, const int32_t* __restrict__ col,
                                           const int32_t* __restrict__ w, const int32_t* __restrict__ L, int32_t Lu,
                                           unsigned long long& ks, unsigned long long& is, bool& bad) {
  for (int64_t e = e0; e < e1; e += (int64_t)step * kNaUnroll) {
    int32_t y[kNaUnroll], x[kNaUnroll];
#pragma unroll
    for (int i = 0; i < kNaUnroll; i++) {
      const int64_t f = e + (int64_t)i * step;
      y[i] = 0;
      x[i] = 0;
      if (f < e1) {
        y[i] = ld_stream(col + f);
        x[i] = ld_stream(w + f);
      }
    }
#pragma unroll
    for (int i = 0; i < kNaUnroll; i++) {
      const bool ok = y[i] >= 0 && y[i] < n;
      bad |= !ok;
      const unsigned long long wv = (unsigned long long)(int64_t)x[i];
      ks += wv;
      if (ok && L[y[i]] == Lu) is += wv;  // (a lane past the row adds a weight of 0)
    }
  }
}

__global__ void __launch_bounds__(kNaThreads) na_rows(int64_t n, const int64_t* __restrict__ rp,
                                                      const int32_t* __restrict__ col, const int32_t* __restrict__ w,
                                                      const int32_t* __restrict__ L, unsigned long long* s) {
  __shared__ int32_t s_long[kNaThreads];
  __shared__ int s_nlong;
  __shared__ unsigned long long red[2][kNaThreads / 32];
  unsigned long long* tail = s + kNoAllocWords - kNoAllocTail;
  const int tid = threadIdx.x, lane = lane_id(), grp = lane / kNaGroup, gl = lane % kNaGroup;
  unsigned long long m2 = 0, in = 0;
  bool bad = false;
  for (int64_t u0 = (int64_t)blockIdx.x * kNaThreads; u0 < n; u0 += (int64_t)gridDim.x * kNaThreads) {
    if (tid == 0) s_nlong = 0;
    __syncthreads();
    const int64_t u = u0 + tid;
    int64_t b = 0, e = 0;
    int32_t Lu = 0;
    if (u < n) {
      b = rp[u];
      e = rp[u + 1];
      Lu = L[u];
      if (Lu < 0 || Lu >= n) bad = true;
      if (e - b > kNaLong) {
        s_long[atomicAdd(&s_nlong, 1)] = tid;
        e = b;
      }
    }
    unsigned long long ks_l = 0;
    for (int t = 0; t < kNaGroup; t++) {  // the warp's rows, four at a time
      const int src = t * (32 / kNaGroup) + grp;
      const int64_t rb = __shfl_sync(0xffffffffu, b, src), re = __shfl_sync(0xffffffffu, e, src);
      const int32_t rl = __shfl_sync(0xffffffffu, Lu, src);
      unsigned long long ks = 0, is = 0;
      na_entries(rb + gl, re, kNaGroup, n, col, w, L, rl, ks, is, bad);
      in += is;
#pragma unroll
      for (int o = kNaGroup / 2; o > 0; o >>= 1) ks += __shfl_xor_sync(0xffffffffu, ks, o);
      const unsigned long long mine = __shfl_sync(0xffffffffu, ks, (lane & (32 / kNaGroup - 1)) * kNaGroup);
      if (lane / (32 / kNaGroup) == t) ks_l = mine;
    }
    if (ks_l && Lu >= 0 && Lu < n) atomicAdd(&s[Lu], ks_l);
    m2 += ks_l;
    __syncthreads();
    for (int i = 0; i < s_nlong; i++) {
      const int64_t v = u0 + s_long[i];
      const int32_t vl = L[v];
      unsigned long long ks = 0;
      na_entries(rp[v] + tid, rp[v + 1], kNaThreads, n, col, w, L, vl, ks, in, bad);
      m2 += ks;
      ks = warp_sum(ks);
      if (lane == 0 && ks && vl >= 0 && vl < n) atomicAdd(&s[vl], ks);
    }
    __syncthreads();
  }
  if (bad) tail[4] = 1;
  m2 = warp_sum(m2);
  in = warp_sum(in);
  if (lane == 0) {
    red[0][tid >> 5] = m2;
    red[1][tid >> 5] = in;
  }
  __syncthreads();
  if (tid < 2) {
    unsigned long long t = 0;
    for (int x = 0; x < kNaThreads / 32; x++) t += red[tid][x];
    if (t) atomicAdd(&tail[tid], t);
  }
}

__global__ void na_sumsq(int64_t n, unsigned long long* s) {
  __shared__ unsigned long long lo_s[8], hi_s[8];
  unsigned __int128 acc = 0;
  for (int64_t c = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; c < n; c += (int64_t)gridDim.x * blockDim.x)
    acc += (unsigned __int128)s[c] * s[c];
  unsigned long long lo = (unsigned long long)acc, hi = (unsigned long long)(acc >> 64);
#pragma unroll
  for (int o = 16; o > 0; o >>= 1) {
    const unsigned long long lo2 = __shfl_xor_sync(0xffffffffu, lo, o), hi2 = __shfl_xor_sync(0xffffffffu, hi, o);
    const unsigned long long nl = lo + lo2;
    hi = hi + hi2 + (nl < lo ? 1ull : 0ull);
    lo = nl;
  }
  if (lane_id() == 0) {
    lo_s[threadIdx.x >> 5] = lo;
    hi_s[threadIdx.x >> 5] = hi;
  }
  __syncthreads();
  if (threadIdx.x == 0) {
    unsigned __int128 t = 0;
    for (int x = 0; x < 8; x++) t += ((unsigned __int128)hi_s[x] << 64) | lo_s[x];
    s[n + 2 * blockIdx.x] = (unsigned long long)t;
    s[n + 2 * blockIdx.x + 1] = (unsigned long long)(t >> 64);
  }
}

// One CTA of kNoAllocCtas threads: the partials of the sum of squares in a
// tree (integers: any order gives the same total), then N.
__global__ void __launch_bounds__(kNoAllocCtas) na_final(int64_t n, unsigned long long* s) {
  __shared__ unsigned long long lo_s[kNoAllocCtas], hi_s[kNoAllocCtas];
  const int b = threadIdx.x;
  lo_s[b] = s[n + 2 * b];
  hi_s[b] = s[n + 2 * b + 1];
  __syncthreads();
  for (int o = kNoAllocCtas / 2; o > 0; o >>= 1) {
    if (b < o) {
      const unsigned long long x = lo_s[b], y = x + lo_s[b + o];
      lo_s[b] = y;
      hi_s[b] += hi_s[b + o] + (y < x ? 1ull : 0ull);
    }
    __syncthreads();
  }
  if (b == 0) {
    unsigned long long* tail = s + kNoAllocWords - kNoAllocTail;
    const unsigned __int128 sq = ((unsigned __int128)hi_s[0] << 64) | lo_s[0];
    const __int128 N = (__int128)(long long)tail[0] * (__int128)(long long)tail[1] - (__int128)sq;
    tail[2] = (unsigned long long)N;
    tail[3] = (unsigned long long)((unsigned __int128)N >> 64);
  }
}

// Device address of the scratch array on the current device.  Looked up on
// every call (the lookup allocates nothing and is cheap): a cached address
// would be shared by host threads without synchronisation and would outlive
// a device reset.  The first lookup on a device loads the module there.
int scratch_for_current_device(unsigned long long** out) {
  void* p = nullptr;
  DCD_TRY_CUDA(cudaGetSymbolAddress(&p, g_noalloc_scratch));
  *out = static_cast<unsigned long long*>(p);
  return DCD_OK;
}

}  // namespace
}  // namespace dcd

static_assert(dcd::kNoAllocMaxN == DCD_NOALLOC_MAX_N, "header limit and scratch layout disagree");

extern "C" int dcd_modularity_noalloc(int64_t n, const int64_t* d_row_ptr, const int32_t* d_col,
                                      const int32_t* d_w, const int32_t* d_labels, void* cuda_stream,
                                      double* q_out, int64_t* m2_out) {
  using namespace dcd;
  if (n <= 0 || n > kNoAllocMaxN || !d_row_ptr || !d_col || !d_w || !d_labels || !q_out) return DCD_EINVAL;
  cudaStream_t s = static_cast<cudaStream_t>(cuda_stream);
  unsigned long long* sc = nullptr;
  DCD_TRY(scratch_for_current_device(&sc));
  const int T = 256;
  count_launch(), na_clear<<<grid_for(n, T), T, 0, s>>>(sc, n);
  count_launch(), na_rows<<<grid_for(n, kNaThreads), kNaThreads, 0, s>>>(n, d_row_ptr, d_col, d_w, d_labels, sc);
  count_launch(), na_sumsq<<<kNoAllocCtas, T, 0, s>>>(n, sc);
  count_launch(), na_final<<<1, kNoAllocCtas, 0, s>>>(n, sc);
  DCD_LAUNCH_CHECK();
  unsigned long long tail[kNoAllocTail];
  DCD_TRY_CUDA(cudaMemcpyAsync(tail, sc + kNoAllocWords - kNoAllocTail, sizeof(tail), cudaMemcpyDeviceToHost, s));
  DCD_TRY_CUDA(cudaStreamSynchronize(s));
  if (tail[4]) return DCD_EINVAL;
  const int64_t m2 = (int64_t)tail[0];
  const __int128 N = (__int128)(((unsigned __int128)tail[3] << 64) | tail[2]);
  *q_out = m2 == 0 ? 0.0 : (double)N / ((double)m2 * (double)m2);
  if (m2_out) *m2_out = m2;
  return DCD_OK;
}
