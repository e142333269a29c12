// levels.cu -- the coarse levels of Algorithm 1 as one kernel.
//
// After level 0 the graph is usually small, tens to hundreds of communities,
// held as a dense matrix of summed weights.  Run as launches, each further
// level costs a binning, a graph instantiation, a dozen launches a pass, a
// compaction and five host round trips, about 0.2 ms a level whatever its size
// (47 communities: 0.22 ms, of which 0.02 are evaluation and apply).  Here all
// of them run in one launch, 10 us at that size: passes, stop rules, compaction
// to the next matrix, level stop rule.  Updates of 2 K vertices went from 0.86
// to 0.64 ms, of 64 graphs (500 to 200 K vertices, 39 M entries in all) from 8.7
// to 7.2.  A graph of the context gets a cluster of 1 to 8 CTAs, which meet at
// the cluster barrier (a hardware barrier of CTAs that are resident together),
// twice a pass.
//
// What bounds it is latency, so the work of a pass is laid out without
// gathers: E(D, i) = the summed weight from vertex i into community D, the
// self-loop left out, starts as the matrix itself (singletons) and follows the
// movers.  A CTA owns a slice of the columns i and keeps E for it, D-major, in
// shared memory when it fits; a lane evaluates one vertex and walks D, warps
// split the range of D.  Labels, a_C, |C| and k are replicated in every CTA,
// which all apply the same moves.  The sums are integers, so their order does
// not matter and every result equals the one of the general path.
#include <algorithm>
#include <type_traits>

#include "agg.cuh"
#include "prims.cuh"
#include "state.cuh"

namespace dcd {

namespace {

constexpr int kLvThreads = 512;
constexpr int kLvWarps = kLvThreads / 32;
constexpr int kLvMaxCluster = 8;  // portable cluster size
// columns a CTA of a cluster takes at least: below this the barrier costs more
// than the walk over D that another CTA would share
constexpr int kLvColumns = 64;

__device__ __forceinline__ unsigned cluster_rank() {
  unsigned r;
  asm volatile("mov.u32 %0, %%cluster_ctarank;" : "=r"(r));
  return r;
}
__device__ __forceinline__ unsigned cluster_size() {
  unsigned r;
  asm volatile("mov.u32 %0, %%cluster_nctarank;" : "=r"(r));
  return r;
}
// Every thread of the cluster arrives; global and shared writes before it are
// visible after it to the whole cluster.
__device__ __forceinline__ void cluster_sync() {
  asm volatile("barrier.cluster.arrive.release.aligned;\n\tbarrier.cluster.wait.acquire.aligned;" ::: "memory");
}
__device__ __forceinline__ unsigned long long now_ns() {
  unsigned long long t;
  asm volatile("mov.u64 %0, %%globaltimer;" : "=l"(t));
  return t;
}

// One coarse level over all graphs: what the step statistics count.
struct LevelRec {
  unsigned long long verts, iso, cnt[4], deg[4];
  unsigned passes, pad;
};

struct LevelsArgs {
  const int64_t* co;  // first cell of graph g's matrix (NULL: one graph)
  const int64_t* cb;  // its communities are cb[g] .. cb[g + 1] - 1
  int64_t nz;         // one graph: its communities
  const void* H;      // the matrices
  void* W;            // room for the later levels' matrices (cells)
  void* E;            // room for E (cells) when it is not in shared memory
  const int64_t* kc;  // weighted degrees
  int32_t* label;     // out: label of every community (a community id of its graph)
  int32_t* prop;      // scratch, one per community
  long long* part;    // scratch, kLvMaxCluster per graph
  GraphState* gs;
  LevelRec* rec;      // zeroed, rec_cap of them
  LevelTotals* tot;   // zeroed
  uint32_t* ticket;   // zeroed
  BinPlan plan;
  int32_t rec_cap, cap;  // cap: communities of the largest graph
  int32_t level, max_levels, max_iters;
  int64_t tau_inv;
};

// Shared arrays of a CTA for graphs of up to cap communities.
inline __host__ __device__ size_t level_smem(int cap, int slice, size_t st) {
  return (size_t)cap * (2 * 8 + 6 * 4) + (size_t)slice * 8 + (size_t)kLvThreads * (st + 8);
}

// VT: cells of 32 bits (2m < 2^31 bounds every sum, gains fit 64 bits) or 64.
// ES: E in shared memory.
template <typename VT, bool ES>
__global__ void __launch_bounds__(kLvThreads, 1) level_loop(LevelsArgs p) {
  using ST = typename std::conditional<sizeof(VT) == 4, long long, i128>::type;
  extern __shared__ __align__(16) unsigned char smem[];
  __shared__ unsigned long long red[kLvWarps][3];
  __shared__ unsigned long long s_deg[4], s_cnt[4];
  __shared__ int s_flag, s_moves;
  const int tid = threadIdx.x, lane = lane_id(), wid = tid >> 5;
  const int CL = (int)cluster_size(), rk = (int)cluster_rank(), g = blockIdx.x / CL;
  const int cap = p.cap, slice_cap = (cap + CL - 1) / CL;
  // 16-byte elements first
  ST* bS = reinterpret_cast<ST*>(smem);
  int64_t* k = reinterpret_cast<int64_t*>(bS + kLvThreads);
  int64_t* a = k + cap;
  int64_t* dg = a + cap;  // self-loops of the slice
  int32_t* L = reinterpret_cast<int32_t*>(dg + slice_cap);
  int32_t* size = L + cap;
  int32_t* np = size + cap;   // proposals of all vertices
  int32_t* cid = np + cap;
  int32_t* comp = cid + cap;  // current vertex of every vertex of the first level
  int32_t* mv = comp + cap;   // movers
  int32_t* bD = mv + cap;
  int32_t* bC = bD + kLvThreads;
  VT* Esm = reinterpret_cast<VT*>(bC + kLvThreads);  // 16-byte alignment is not needed: 4- or 8-byte cells
  GraphState& X = p.gs[g];
  const int64_t cb = p.cb ? p.cb[g] : 0, co = p.co ? p.co[g] : 0;
  const int nz1 = (int)(p.cb ? p.cb[g + 1] - cb : p.nz);
  if (!X.done) {
    const int64_t m2 = X.m2;
    const VT* M = static_cast<const VT*>(p.H) + co;
    VT* W = static_cast<VT*>(p.W) + co;
    int32_t* prop = p.prop + cb;
    long long* part = p.part + (int64_t)g * kLvMaxCluster;
    i128 N = ld128(&X.n_cur_lo);  // every thread keeps it: the decisions are uniform
    int64_t in = X.in_cur;
    int nz = nz1, level = p.level, pass_sum = 0;
    long long moves_sum = 0;
    unsigned long long t_eval = 0, t_apply = 0, t_comp = 0, t0 = now_ns();
    for (int x = tid; x < nz; x += kLvThreads) {
      const int64_t kv = p.kc[cb + x];
      k[x] = a[x] = kv;
      L[x] = comp[x] = x;
      size[x] = 1;
    }
    for (;;) {
      const int sl = (nz + CL - 1) / CL, i0 = min(rk * sl, nz), w = min(sl, nz - i0);
      VT* E = ES ? Esm : static_cast<VT*>(p.E) + co + (int64_t)i0 * nz;
      for (int D = wid; D < nz; D += kLvWarps)
        for (int il = lane; il < w; il += 32) {
          const VT v = __ldcg(M + (uint32_t)(D * nz + i0 + il));
          const bool self = D == i0 + il;
          E[(uint32_t)(D * w + il)] = self ? VT(0) : v;
          if (self) dg[il] = (int64_t)v;
        }
      if (tid < 4) s_deg[tid] = s_cnt[tid] = 0;
      __syncthreads();
      const i128 N_start = N;
      int passes = 0;
      const int nblk = (w + 31) / 32, nbr = max(1, min(nblk, kLvWarps)), parts = kLvWarps / nbr;
      const int dl = (nz + parts - 1) / parts;
      unsigned long long t1 = now_ns();
      t_comp += t1 - t0;
      for (;;) {
        // evaluate the slice under the snapshot
        for (int b0 = 0; b0 < nblk; b0 += nbr) {
          const int pt = wid / nbr, il = (b0 + wid % nbr) * 32 + lane;
          const bool has = pt < parts && il < w;
          ST Sb = gain_lowest<ST>();
          int32_t Db = INT_MAX;
          int cnt = 0;
          if (has) {
            const int i = i0 + il, C = L[i];
            const int64_t kv = k[i], aC = a[C], eC = (int64_t)E[(uint32_t)(C * w + il)];
            const int d1 = min(nz, (pt + 1) * dl);
            int D = pt * dl;
            constexpr int U = 8;
            for (; D < d1; D += U) {
              VT e[U];
#pragma unroll
              for (int u = 0; u < U; u++) e[u] = D + u < d1 ? E[(uint32_t)((D + u) * w + il)] : VT(0);
#pragma unroll
              for (int u = 0; u < U; u++) {
                if (!e[u]) continue;
                cnt++;
                if (D + u == C) continue;
                const ST x = gain<ST>(m2, kv, (int64_t)e[u], eC, a[D + u], aC);
                if (x > Sb) {  // D ascends: ties stay with the smaller label
                  Sb = x;
                  Db = D + u;
                }
              }
            }
          }
          bS[tid] = Sb;
          bD[tid] = Db;
          bC[tid] = cnt;
          __syncthreads();
          if (wid < nbr && il < w) {
            for (int q = 1; q < parts; q++) {
              const int o = tid + q * nbr * 32;
              cnt += bC[o];
              if (better(bS[o], bD[o], Sb, Db)) {
                Sb = bS[o];
                Db = bD[o];
              }
            }
            __stcg(prop + i0 + il, move_proposal(Sb, Db, L[i0 + il], size));
            if (passes == 0) {
              const int d = cnt + (dg[il] != 0 ? 1 : 0);
              const int c = lm_variant_class(p.plan.var[bin_of(p.plan, d)]);
              if (d > 0) {
                atomicAdd(&s_cnt[c], 1ull);
                atomicAdd(&s_deg[c], (unsigned long long)d);
              }
            }
          }
          __syncthreads();
        }
        if (tid == 0) s_moves = 0;
        cluster_sync();
        const unsigned long long t2 = now_ns();
        t_eval += t2 - t1;
        for (int x0 = 0; x0 < nz; x0 += kLvThreads) {
          const int x = x0 + tid;
          bool m = false;
          if (x < nz) {
            np[x] = __ldcg(prop + x);
            m = np[x] != L[x];
          }
          const unsigned bal = __ballot_sync(0xffffffffu, m);
          int base = 0;
          if (lane == 0 && bal) base = atomicAdd(&s_moves, __popc(bal));
          base = __shfl_sync(0xffffffffu, base, 0);
          if (m) mv[base + __popc(bal & lanemask_lt())] = x;
        }
        __syncthreads();
        const int moves = s_moves;
        passes++;
        moves_sum += moves;
        if (moves == 0) {
          t1 = now_ns();
          t_apply += t1 - t2;
          break;
        }
        for (int q = tid; q < moves; q += kLvThreads) {
          const int j = mv[q], A = L[j], B = np[j];
          atomicAdd((unsigned long long*)&a[A], (unsigned long long)(-k[j]));
          atomicAdd((unsigned long long*)&a[B], (unsigned long long)k[j]);
          atomicAdd(&size[A], -1);
          atomicAdd(&size[B], 1);
        }
        for (int q = wid; q < moves; q += kLvWarps) {
          const int j = mv[q], A = L[j], B = np[j];
          for (int il = lane; il < w; il += 32) {
            const VT v = __ldcg(M + (uint32_t)(j * nz + i0 + il));
            if (v && i0 + il != j) {
              atomicAdd(&E[(uint32_t)(A * w + il)], (VT)(VT(0) - v));
              atomicAdd(&E[(uint32_t)(B * w + il)], v);
            }
          }
        }
        __syncthreads();
        for (int q = tid; q < moves; q += kLvThreads) L[mv[q]] = np[mv[q]];
        __syncthreads();
        // sum_i e_{i->C(i)} of the slice, sum_C a_C^2 of all
        unsigned long long s_in = 0;
        unsigned __int128 sq = 0;
        for (int il = tid; il < w; il += kLvThreads)
          s_in += (unsigned long long)E[(uint32_t)(L[i0 + il] * w + il)] + (unsigned long long)dg[il];
        for (int x = tid; x < nz; x += kLvThreads) sq += (unsigned __int128)(unsigned long long)a[x] * (unsigned long long)a[x];
        unsigned long long lo = (unsigned long long)sq, hi = (unsigned long long)(sq >> 64);
#pragma unroll
        for (int o = 16; o > 0; o >>= 1) {
          s_in += __shfl_xor_sync(0xffffffffu, s_in, o);
          const unsigned long long lo2 = __shfl_xor_sync(0xffffffffu, lo, o);
          const unsigned long long hi2 = __shfl_xor_sync(0xffffffffu, hi, o);
          const unsigned long long nlo = lo + lo2;
          hi = hi + hi2 + (nlo < lo ? 1ull : 0ull);
          lo = nlo;
        }
        if (lane == 0) {
          red[wid][0] = s_in;
          red[wid][1] = lo;
          red[wid][2] = hi;
        }
        __syncthreads();
        if (tid == 0) {
          unsigned long long t = 0;
          for (int q = 0; q < kLvWarps; q++) t += red[q][0];
          __stcg(part + rk, (long long)t);
        }
        cluster_sync();
        int64_t in_new = 0;
        for (int q = 0; q < CL; q++) in_new += __ldcg(part + q);
        sq = 0;
        for (int q = 0; q < kLvWarps; q++) sq += ((unsigned __int128)red[q][2] << 64) | red[q][1];
        const i128 N_new = (i128)m2 * (i128)in_new - (i128)sq;
        const bool stop = below_tau(N_new - N, N, p.tau_inv) || passes >= p.max_iters;
        in = in_new;
        N = N_new;
        t1 = now_ns();
        t_apply += t1 - t2;
        if (stop) break;
      }
      t0 = now_ns();
      __syncthreads();
      // communities in use, numbered in label order
      int nc = 0;
      for (int x0 = 0; x0 < nz; x0 += kLvThreads) {
        const int x = x0 + tid;
        const int used = x < nz && size[x] > 0 ? 1 : 0;
        int tot;
        const int pre = block_excl_scan<int, kLvThreads>(used, &tot);
        if (used) cid[x] = nc + pre;
        nc += tot;
      }
      __syncthreads();
      LevelRec& rec = p.rec[min(level - p.level, p.rec_cap - 1)];
      if (tid < 4 && s_cnt[tid]) {
        atomicAdd(&rec.cnt[tid], s_cnt[tid]);
        atomicAdd(&rec.deg[tid], s_deg[tid]);
      }
      if (rk == 0 && tid == 0) {
        atomicMax(&rec.passes, (unsigned)passes);
        atomicAdd(&rec.verts, (unsigned long long)nz);
        atomicAdd(&rec.iso, (unsigned long long)X.iso);
      }
      level++;
      pass_sum += passes;
      const bool done = nc == nz || below_tau(N - N_start, N_start, p.tau_inv) || level >= p.max_levels;
      for (int x = tid; x < nz1; x += kLvThreads) comp[x] = done ? L[comp[x]] : cid[L[comp[x]]];
      if (done) break;
      // the next level's matrix
      for (int64_t x = (int64_t)rk * kLvThreads + tid; x < (int64_t)nc * nc; x += (int64_t)CL * kLvThreads)
        __stcg(W + x, VT(0));
      cluster_sync();
      for (int D = wid; D < nz; D += kLvWarps) {
        if (size[D] == 0) continue;
        const int y = cid[D];
        for (int il = lane; il < w; il += 32) {
          const int C = L[i0 + il];
          const VT v = E[(uint32_t)(D * w + il)] + (C == D ? (VT)dg[il] : VT(0));
          if (v) atomicAdd(W + (uint32_t)(cid[C] * nc + y), v);
        }
      }
      for (int x = tid; x < nz; x += kLvThreads)
        if (size[x] > 0) k[cid[x]] = a[x];  // k of this level is no longer read
      cluster_sync();
      for (int x = tid; x < nc; x += kLvThreads) {
        a[x] = k[x];
        L[x] = x;
        size[x] = 1;
      }
      M = W;
      nz = nc;
      __syncthreads();
    }
    __syncthreads();
    for (int x = rk * kLvThreads + tid; x < nz1; x += CL * kLvThreads) p.label[cb + x] = (int32_t)cb + comp[x];
    if (rk == 0 && tid == 0) {
      X.in_cur = in;
      st128(&X.n_cur_lo, N);
      X.running = 0;
      X.done = 1;
      X.lv_passes = pass_sum;
      X.lv_moves = moves_sum;
      X.lv_levels = level;
      t_comp += now_ns() - t0;
      atomicMax(&p.tot->t_eval_ns, t_eval);
      atomicMax(&p.tot->t_apply_ns, t_apply);
      atomicMax(&p.tot->t_compact_ns, t_comp);
    }
  }
  // the last CTA adds the levels up
  __threadfence();
  __syncthreads();
  if (tid == 0) s_flag = atomicAdd(p.ticket, 1u) == gridDim.x - 1;
  __syncthreads();
  if (s_flag && tid == 0) {
    __threadfence();
    LevelTotals& t = *p.tot;
    for (int l = 0; l < p.rec_cap; l++) {
      const LevelRec& r = p.rec[l];
      const unsigned long long ps = __ldcg(&r.passes);
      if (!ps) break;
      t.levels++;
      t.passes += ps;
      t.verts += (__ldcg(&r.verts) + __ldcg(&r.iso)) * ps;
      for (int c = 0; c < 4; c++) {
        t.verts_bin[c] += __ldcg(&r.cnt[c]) * ps;
        t.edges_bin[c] += __ldcg(&r.deg[c]) * ps;
        t.edges += __ldcg(&r.deg[c]) * ps;
      }
    }
  }
}

template <typename VT>
int launch_levels(dcd_ctx* c, LevelsArgs p, int G, int64_t cells, Buf<VT>& E) {
  using ST = typename std::conditional<sizeof(VT) == 4, long long, i128>::type;
  int CL = 1;
  while (CL < kLvMaxCluster && CL * kLvColumns < p.cap) CL *= 2;
  const int slice = (p.cap + CL - 1) / CL;
  size_t sm = level_smem(p.cap, slice, sizeof(ST));
  const size_t smE = sm + (size_t)slice * p.cap * sizeof(VT);
  const bool es = smE <= kLevelSmem;
  auto* kern = es ? level_loop<VT, true> : level_loop<VT, false>;
  if (es) {
    sm = smE;
  } else {
    DCD_TRY(E.alloc(&c->mem, cells));
    p.E = E.get();
  }
  // the attribute belongs to the process: always the same value, so that another
  // thread's context cannot lower it between this and the launch
  DCD_TRY_CUDA(cudaFuncSetAttribute(kern, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)kLevelSmem));
  cudaLaunchConfig_t cfg{};
  cfg.gridDim = dim3((unsigned)(G * CL));
  cfg.blockDim = dim3(kLvThreads);
  cfg.dynamicSmemBytes = sm;
  cfg.stream = c->stream;
  cudaLaunchAttribute at[1];
  at[0].id = cudaLaunchAttributeClusterDimension;
  at[0].val.clusterDim.x = (unsigned)CL;
  at[0].val.clusterDim.y = at[0].val.clusterDim.z = 1;
  cfg.attrs = at;
  cfg.numAttrs = 1;
  count_launch();
  DCD_TRY_CUDA(cudaLaunchKernelEx(&cfg, kern, p));
  tracef("coarse levels: one launch, %d CTAs a graph, sums in %s memory", CL, es ? "shared" : "global");
  return DCD_OK;
}

}  // namespace

int coarse_levels(dcd_ctx* c, const LevelsIn& in, LevelsBufs* b) {
  cudaStream_t s = c->stream;
  const int G = c->G;
  LevelsArgs p{};
  p.co = in.co;
  p.cb = in.cb;
  p.nz = in.nz;
  p.H = in.H;
  p.kc = in.kc;
  p.label = in.label;
  p.gs = c->gs.get();
  p.plan = c->bin_plan;
  p.cap = (int32_t)in.max_nz;
  // a level has fewer communities than the one before
  p.rec_cap = (int32_t)std::min<int64_t>(in.max_nz + 1, std::max<int64_t>(1, (int64_t)c->cfg.max_levels - in.level));
  p.level = in.level;
  p.max_levels = c->cfg.max_levels;
  p.max_iters = c->cfg.max_iters;
  p.tau_inv = c->cfg.tau_inv;
  // one block of scratch: totals, ticket, level records (zeroed), then parts and proposals
  const size_t head = 256, recs = sizeof(LevelRec) * (size_t)p.rec_cap;
  static_assert(sizeof(LevelTotals) <= 240, "totals and ticket share the head");
  DCD_TRY(b->scratch.alloc(&c->mem, head + recs + (size_t)G * kLvMaxCluster * 8 + (size_t)in.nz * 4));
  unsigned char* q = b->scratch.get();
  DCD_TRY_CUDA(cudaMemsetAsync(q, 0, head + recs, s));
  p.tot = b->tot = reinterpret_cast<LevelTotals*>(q);
  p.ticket = reinterpret_cast<uint32_t*>(q + 240);
  p.rec = reinterpret_cast<LevelRec*>(q + head);
  p.part = reinterpret_cast<long long*>(q + head + recs);
  p.prop = reinterpret_cast<int32_t*>(q + head + recs + (size_t)G * kLvMaxCluster * 8);
  if (in.wide) {
    DCD_TRY(b->w64.alloc(&c->mem, in.cells));
    p.W = b->w64.get();
    return launch_levels<unsigned long long>(c, p, G, in.cells, b->e64);
  }
  DCD_TRY(b->w32.alloc(&c->mem, in.cells));
  p.W = b->w32.get();
  return launch_levels<unsigned>(c, p, G, in.cells, b->e32);
}

}  // namespace dcd
