// features.cu -- the learned screen around Delta-screening (not in the paper).
//
// Pool P = R_t of Delta-screening, plus every vertex touched by the batch and
// its neighbours in G_t.  For each pool vertex of positive degree, under
// C_{t-1} on G_t, twelve features:
//   0 log1p(degree)            1 log1p(d_w)             2 log1p(inserted pairs)
//   3 log1p(deleted pairs)     4 inserted weight / d_w  5 e_{v->C\v} / d_w
//   6 e_{v->D*} / d_w          7 S(v->D*) / (d_w 2m)    8 a_C / 2m
//   9 a_{D*} / 2m             10 log1p(|C|)            11 [v in R_t]
// where D* is the best other neighbouring community by the exact gain S.  The
// network scores each row; R'_t = (R_t with p >= theta_keep) + (P \ R_t with
// p >= theta_add).  Labels for training: 1 when the vertex's community after
// the level-0 local moving of a full re-evaluation (R_t = V) differs from
// C_{t-1}.
#include "agg.cuh"
#include "prims.cuh"
#include "pull.cuh"
#include "state.cuh"

namespace dcd {
namespace {

constexpr uint8_t kPairIns = 1, kPairDel = 2, kPairPresent = 4;

// pool[v] = R_t[v] | (v has a pair) | (v is a neighbour of a vertex with a pair).
// Push: a warp a vertex with pairs writes a byte per entry of its row.
__global__ void pool_mark(int64_t n, const int64_t* __restrict__ rp, const int32_t* __restrict__ col,
                          const int32_t* __restrict__ pair_ptr, const uint8_t* __restrict__ rds,
                          uint8_t* __restrict__ pool) {
  const int64_t nw = ((int64_t)gridDim.x * blockDim.x) >> 5;
  for (int64_t u = (blockIdx.x * (int64_t)blockDim.x + threadIdx.x) >> 5; u < n; u += nw) {
    if (lane_id() == 0 && rds[u]) pool[u] = 1;
    if (pair_ptr[u + 1] == pair_ptr[u]) continue;
    if (lane_id() == 0) pool[u] = 1;
    for (int64_t e = rp[u] + lane_id(); e < rp[u + 1]; e += 32) pool[col[e]] = 1;
  }
}

// Pull: the vertices that the first two terms leave out look for a neighbour
// with a pair, a warp a row (the rest of a long row: pull_rest), and stop at the
// first.  Reads at most the rows of the vertices without pairs, where push reads (and writes a byte for) those with
// pairs: taken when these hold half of the entries (kPoolPull).  1 M vertices, 21 M
// entries, nearly all of them in rows with pairs: 414 us by push, below 5 so.
constexpr int kPoolPull = 2;
struct HasPair {
  const int32_t* pair_ptr;
  __device__ __forceinline__ bool operator()(int32_t x) const { return pair_ptr[x + 1] != pair_ptr[x]; }
};
__global__ void pool_pull(int64_t n, const int64_t* __restrict__ rp, const int32_t* __restrict__ col,
                          const int32_t* __restrict__ pair_ptr, const uint8_t* __restrict__ rds,
                          uint8_t* __restrict__ pool, PullRest rest) {
  const HasPair marked{pair_ptr};
  const int64_t stride = (int64_t)gridDim.x * blockDim.x;
  const int lane = lane_id();
  for (int64_t base = blockIdx.x * (int64_t)blockDim.x + (threadIdx.x & ~31); base < n; base += stride) {
    const int64_t v = base + lane;
    bool in = v < n && (rds[v] || pair_ptr[v + 1] != pair_ptr[v]);
    unsigned left = __ballot_sync(0xffffffffu, v < n && !in);
    int64_t deg = 0;  // of an undecided vertex
    while (left) {
      const int src = __ffs(left) - 1;
      left &= left - 1;
      const int64_t u = base + src, b = rp[u], d = rp[u + 1] - b;
      const int64_t end = b + (d < kPullFirst ? d : kPullFirst);
      bool hit = false;
      for (int64_t e0 = b; e0 < end && !hit; e0 += 32) {
        const int64_t e = e0 + lane;
        hit = __any_sync(0xffffffffu, e < end && marked(col[e]));
      }
      if (lane == src) {
        in = hit;
        deg = d;
      }
    }
    if (v < n) pool[v] = in ? 1 : 0;
    pull_defer(rest, v < n && !in && deg > kPullFirst, v, deg);
  }
}

// Inserted and deleted pairs (high and low word) and inserted weight of every
// source.  32 consecutive pairs a warp, whatever sources they belong to: the pairs
// are sorted by source, so each run of equal sources counts by ballots, sums its
// weights by shuffles and adds once.
__global__ void __launch_bounds__(256) source_sums(int64_t P, const uint64_t* __restrict__ pkey,
                                                   const uint8_t* __restrict__ pflag, const int32_t* __restrict__ pw,
                                                   unsigned long long* __restrict__ cnt,
                                                   unsigned long long* __restrict__ wsum) {
  const int64_t stride = (int64_t)gridDim.x * blockDim.x;
  const int lane = lane_id();
  for (int64_t base = blockIdx.x * (int64_t)blockDim.x + (threadIdx.x & ~31); base < P; base += stride) {
    const int64_t p = base + lane;
    const int32_t u = p < P ? (int32_t)(pkey[p] >> 32) : -1;
    const uint8_t f = p < P ? pflag[p] : 0;
    const bool ins = f & kPairIns, del = (f & kPairDel) && (f & kPairPresent);
    unsigned long long w = ins ? (unsigned long long)pw[p] : 0ull;
    const int32_t before = __shfl_up_sync(0xffffffffu, u, 1);
    const unsigned heads = __ballot_sync(0xffffffffu, lane == 0 || u != before);
    const unsigned above = lane == 31 ? 0u : heads & (0xfffffffeu << lane);
    const int end = above ? __ffs(above) - 1 : 32;  // first lane behind this one's run
#pragma unroll
    for (int o = 1; o < 32; o <<= 1) {  // sums of the run from this lane on
      const unsigned long long y = __shfl_down_sync(0xffffffffu, w, o);
      if (lane + o < end) w += y;
    }
    const unsigned bi = __ballot_sync(0xffffffffu, ins), bd = __ballot_sync(0xffffffffu, del);
    if ((heads >> lane & 1) && u >= 0) {
      const unsigned run = (end == 32 ? 0xffffffffu : (1u << end) - 1u) & (0xffffffffu << lane);
      const unsigned long long x = (unsigned long long)__popc(bi & run) << 32 | (unsigned)__popc(bd & run);
      if (x) atomicAdd(&cnt[u], x);
      if (w) atomicAdd(&wsum[u], w);
    }
  }
}

// A thread a row; the 32 x 12 features of a warp are written as one run of 384
// floats.  1 M rows and 6.2 M pairs: 616 us with a thread walking its row's pairs
// and storing 12 floats at a stride of 48 bytes, 56 here and 35 in source_sums so;
// what is left are the gathers by vertex and community.
constexpr int kAsmThreads = 256;
__global__ void __launch_bounds__(kAsmThreads) assemble(
    int64_t m, const int32_t* __restrict__ list, const int64_t* __restrict__ rp, const int64_t* __restrict__ k,
    const int32_t* __restrict__ L, const int64_t* __restrict__ a, const int32_t* __restrict__ size,
    const unsigned long long* __restrict__ pcnt, const unsigned long long* __restrict__ pwsum,
    const int64_t* __restrict__ eC, const int64_t* __restrict__ eB, const int32_t* __restrict__ dB,
    const double* __restrict__ sB, const uint8_t* __restrict__ rds, int64_t m2, float* __restrict__ X) {
  __shared__ float s_x[kAsmThreads / 32][32 * 13];  // a row has 13 words here: no bank conflicts
  const int lane = lane_id(), wid = threadIdx.x >> 5;
  const int64_t stride = (int64_t)gridDim.x * blockDim.x;
  for (int64_t base = blockIdx.x * (int64_t)blockDim.x + (threadIdx.x & ~31); base < m; base += stride) {
    const bool has = base + lane < m;
    const int64_t j = has ? base + lane : base;
    const int32_t v = list[j];
    const unsigned long long pc = pcnt[v];
    const int64_t nins = (int64_t)(pc >> 32), ndel = (int64_t)(pc & 0xffffffffu), wins = (int64_t)pwsum[v];
    const int64_t deg = rp[v + 1] - rp[v];
    const int64_t kv = k[v];
    const int32_t C = L[v];
    const float fk = (float)kv, fm = (float)m2;
    const int32_t D = dB[j];
    float* x = &s_x[wid][lane * 13];
    x[0] = log1pf((float)deg);
    x[1] = log1pf(fk);
    x[2] = log1pf((float)nins);
    x[3] = log1pf((float)ndel);
    x[4] = kv > 0 ? fminf((float)wins / fk, 1.f) : 0.f;
    x[5] = kv > 0 ? (float)eC[j] / fk : 0.f;
    x[6] = kv > 0 ? (float)eB[j] / fk : 0.f;
    x[7] = (kv > 0 && m2 > 0) ? (float)(sB[j] / ((double)kv * (double)m2)) : 0.f;
    x[8] = m2 > 0 ? (float)a[C] / fm : 0.f;
    x[9] = (m2 > 0 && D >= 0) ? (float)a[D] / fm : 0.f;
    x[10] = log1pf((float)size[C]);
    x[11] = rds[v] ? 1.f : 0.f;
    __syncwarp();
    const int rows = m - base < 32 ? (int)(m - base) : 32;
    for (int q = lane; q < rows * 12; q += 32) X[base * 12 + q] = s_x[wid][(q / 12) * 13 + q % 12];
    __syncwarp();
  }
}

__global__ void learned_rset(int64_t m, const int32_t* __restrict__ list, const float* __restrict__ p,
                             const uint8_t* __restrict__ rds, float theta_keep, float theta_add,
                             uint8_t* __restrict__ r, unsigned long long* __restrict__ count) {
  unsigned long long c = 0;
  for (int64_t i = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; i < m; i += (int64_t)gridDim.x * blockDim.x) {
    const int32_t v = list[i];
    const uint8_t x = rds[v] ? (p[i] >= theta_keep) : (p[i] >= theta_add);
    r[v] = x;
    c += x;
  }
  c = warp_sum(c);
  if (lane_id() == 0 && c) atomicAdd(count, c);
}

__global__ void move_labels(int64_t m, const int32_t* __restrict__ list, const int32_t* __restrict__ before,
                            const int32_t* __restrict__ after, float* __restrict__ y) {
  for (int64_t i = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; i < m; i += (int64_t)gridDim.x * blockDim.x) {
    const int32_t v = list[i];
    y[i] = before[v] != after[v] ? 1.f : 0.f;
  }
}

}  // namespace

int screen_features(dcd_ctx* c, const Csr<int32_t>& g, const int32_t* L0, const int64_t* k, const int64_t* a,
                    const int32_t* size, const MergeOut& mo, int64_t source_deg, const uint8_t* rds, EntryLabels* nlab,
                    LearnedPool* out) {
  cudaStream_t s = c->stream;
  const int64_t n = g.n;
  const int T = 256;
  Buf<uint8_t> pool;
  DCD_TRY(pool.alloc(&c->mem, n));
  if (kPoolPull * source_deg >= g.nnz) {
    PullBufs bufs;
    PullRest rest{};
    int32_t* cnt = c->dsc.get()->rest_cnt;  // the screening is done with it
    DCD_TRY(bufs.alloc(&c->mem, n, g.nnz, cnt, &rest));
    DCD_TRY_CUDA(cudaMemsetAsync(cnt, 0, 2 * sizeof(int32_t), s));
    count_launch(), pool_pull<<<grid_for(n, T), T, 0, s>>>(n, g.rp, g.col, mo.pair_ptr.get(), rds, pool.get(), rest);
    count_launch(), pull_rest<<<4 * c->sms, kPullThreads, 0, s>>>(g.rp, g.col, rest, HasPair{mo.pair_ptr.get()},
                                                                  pool.get(), nullptr);
  } else {
    DCD_TRY_CUDA(cudaMemsetAsync(pool.get(), 0, n, s));
    count_launch(), pool_mark<<<grid_for(n * 32, T, 16), T, 0, s>>>(n, g.rp, g.col, mo.pair_ptr.get(), rds,
                                                                    pool.get());
  }
  DCD_LAUNCH_CHECK();
  DCD_TRY(pool_stats(c, g, L0, k, a, size, pool.get(), nlab, &out->st));
  const int64_t m = out->st.count;
  DCD_TRY(c->feat_X.ensure(&c->mem, 12 * (m > 0 ? m : 1)));
  DCD_TRY(c->feat_v.ensure(&c->mem, m > 0 ? m : 1));
  if (m > 0) {
    Buf<unsigned long long> pcnt;
    DCD_TRY(pcnt.alloc(&c->mem, 2 * n));
    DCD_TRY_CUDA(cudaMemsetAsync(pcnt.get(), 0, 2 * n * sizeof(unsigned long long), s));
    if (mo.npairs > 0) {
      count_launch(), source_sums<<<grid_for(mo.npairs, T), T, 0, s>>>(mo.npairs, mo.pkey.get(), mo.pflag.get(),
                                                                       mo.pw.get(), pcnt.get(), pcnt.get() + n);
      DCD_LAUNCH_CHECK();
    }
    count_launch(), assemble<<<grid_for(m, kAsmThreads), kAsmThreads, 0, s>>>(
        m, out->st.list.get(), g.rp, k, L0, a, size, pcnt.get(), pcnt.get() + n,
        out->st.eC.get(), out->st.eB.get(), out->st.dB.get(), out->st.sB.get(), rds, c->hgs[0].m2, c->feat_X.get());
    DCD_LAUNCH_CHECK();
    DCD_TRY_CUDA(cudaMemcpyAsync(c->feat_v.get(), out->st.list.get(), m * sizeof(int32_t), cudaMemcpyDeviceToDevice, s));
  }
  c->feat_n = m;
  return DCD_OK;
}

int learned_rset_build(dcd_ctx* c, const LearnedPool& lp, const uint8_t* rds, const float* p, uint8_t* r,
                       int64_t* r_size) {
  cudaStream_t s = c->stream;
  DevScalars* d = c->dsc.get();
  const int64_t n = c->n;
  const int64_t m = lp.st.count;
  DCD_TRY_CUDA(cudaMemsetAsync(r, 0, n, s));
  DCD_TRY_CUDA(cudaMemsetAsync(&d->r_size, 0, sizeof(int64_t), s));
  if (m > 0) {
    count_launch(), learned_rset<<<grid_for(m, 256), 256, 0, s>>>(m, lp.st.list.get(), p, rds, c->theta_keep,
                                                                   c->theta_add, r, (unsigned long long*)&d->r_size);
    DCD_LAUNCH_CHECK();
  }
  DCD_TRY_CUDA(cudaMemcpyAsync(c->hscratch + 11, &d->r_size, sizeof(int64_t), cudaMemcpyDeviceToHost, s));
  DCD_TRY_CUDA(cudaStreamSynchronize(s));
  *r_size = c->hscratch[11];
  return DCD_OK;
}

int screen_labels(dcd_ctx* c, const int32_t* before, const int32_t* after) {
  const int64_t m = c->feat_n;
  DCD_TRY(c->feat_y.ensure(&c->mem, m > 0 ? m : 1));
  if (m > 0) {
    count_launch(), move_labels<<<grid_for(m, 256), 256, 0, c->stream>>>(m, c->feat_v.get(), before, after,
                                                                          c->feat_y.get());
    DCD_LAUNCH_CHECK();
  }
  c->feat_has_y = true;
  return DCD_OK;
}

}  // namespace dcd
