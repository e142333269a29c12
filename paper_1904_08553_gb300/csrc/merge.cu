// merge.cu -- Delta_t into G_t: batch records sorted by (source, sink), their
// effect on G_{t-1}, and a tiled merge of the CSR with the pairs.  The
// weighted degrees d_w (Sec. III-A), 2m and sum_i e_{i->C(i)} of G_t follow
// from their values on G_{t-1} and the batch's weight changes.
//
// The changes are stored as ordered pairs (i,j) and (j,i) (Sec. III-E).  The
// paper only adds edges; the reading for deletions is: every delete of the
// step acts first and removes the whole edge, then every insert adds its
// weight (a new edge or a larger multiplicity).
//
// Records.  A record is one 64-bit word, sink << 32 | weight (0: a delete),
// in its source's segment.  Records of one (source, sink) stay next to each
// other as null pairs (no flag, no weight change) behind which the last one
// stands for all; so the pairs of source u are [off[u], off[u+1]) with no
// compaction, and nothing has to be counted on the host before the merge.
#include "prims.cuh"
#include "rows.cuh"
#include "state.cuh"

namespace dcd {

namespace {

constexpr uint8_t kPairIns = 1, kPairDel = 2, kPairPresent = 4, kPairAdded = 8, kPairRemoved = 16;

__device__ __forceinline__ bool record_ok(const dcd_edge& e, int64_t n, bool is_ins) {
  return e.u >= 0 && e.v >= 0 && e.u < n && e.v < n && e.u != e.v && (!is_ins || e.w > 0);
}

__global__ void validate_records(const dcd_edge* __restrict__ ins, int64_t n_ins,
                                 const dcd_edge* __restrict__ del, int64_t n_del, int64_t n,
                                 uint32_t* __restrict__ err) {
  int64_t tot = n_ins + n_del;
  bool bad = false;
  for (int64_t i = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; i < tot;
       i += (int64_t)gridDim.x * blockDim.x) {
    const dcd_edge e = i < n_ins ? ins[i] : del[i - n_ins];
    bad |= !record_ok(e, n, i < n_ins);
  }
  if (__any_sync(0xffffffffu, bad) && lane_id() == 0) atomicOr(err, kErrBadRecord);
}

// Records per source, and each record's place in its source's segment (the
// atomic's return value, so the scatter needs no atomic of its own).  Batches
// staged from device memory are first checked here: a bad record is reported
// and takes no place.
__global__ void rec_count(const dcd_edge* __restrict__ ins, int64_t n_ins, const dcd_edge* __restrict__ del,
                          int64_t n_del, int64_t n, int32_t* __restrict__ cnt, int2* __restrict__ rank,
                          uint32_t* __restrict__ err) {
  const int64_t tot = n_ins + n_del;
  bool bad = false;
  for (int64_t i = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; i < tot; i += (int64_t)gridDim.x * blockDim.x) {
    const dcd_edge e = i < n_ins ? ins[i] : del[i - n_ins];
    if (!record_ok(e, n, i < n_ins)) {
      bad = true;
      continue;
    }
    int2 r;
    r.x = atomicAdd(&cnt[e.u], 1);
    r.y = atomicAdd(&cnt[e.v], 1);
    rank[i] = r;
  }
  if (bad) atomicOr(err, kErrBadRecord);
}

__global__ void rec_scatter(const dcd_edge* __restrict__ ins, int64_t n_ins, const dcd_edge* __restrict__ del,
                            int64_t n_del, int64_t n, const int32_t* __restrict__ off, const int2* __restrict__ rank,
                            uint64_t* __restrict__ rec) {
  const int64_t tot = n_ins + n_del;
  for (int64_t i = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; i < tot; i += (int64_t)gridDim.x * blockDim.x) {
    const dcd_edge e = i < n_ins ? ins[i] : del[i - n_ins];
    if (!record_ok(e, n, i < n_ins)) continue;
    const int2 r = rank[i];
    const uint64_t w = i < n_ins ? (uint32_t)e.w : 0u;
    rec[off[e.u] + r.x] = (uint64_t)(uint32_t)e.v << 32 | w;
    rec[off[e.v] + r.y] = (uint64_t)(uint32_t)e.u << 32 | w;
  }
}

// ---- pairs and their effect on G_{t-1} ----

struct PairView {
  const int32_t* off;  // n + 1: records (pairs) of source u are [off[u], off[u+1])
  const int64_t* rp;   // G_{t-1}
  const int32_t* col;
  const int32_t* w;
  const int32_t* lab0;  // C_{t-1} when sum e_{i->C(i)} is tracked, else NULL
  const int32_t* gid;
  uint64_t* pkey;   // source << 32 | sink
  int32_t* pw;      // summed insert weight
  uint8_t* pflag;
  int32_t* pdelta;  // weight in G_t minus weight in G_{t-1}
  int64_t* epos;    // first entry of G_{t-1} not before the pair (CSR order)
  int32_t* net;     // +1 adds an entry, -1 removes one
  GraphState* gs;   // m2 and in_cur receive the changes
  int64_t* npairs;  // distinct pairs
  uint32_t* err;
};

// What one record contributes to the sums of its CTA.
struct PairSum {
  long long m2 = 0, in = 0;
  int heads = 0;
};

// Pair (u, v) at place p: W the summed insert weight, e its place in row u
// (first entry with sink >= v), head: the record that stands for its pair.
__device__ __forceinline__ int32_t put_pair(const PairView& o, int64_t p, int32_t u, int32_t v, int64_t W, bool isins,
                                            bool isdel, bool head, int64_t e, bool present, PairSum& acc) {
  uint8_t f = 0;
  int64_t dlt = 0;
  int32_t net = 0;
  if (head) {
    // deletes remove the whole edge first, then inserts add their weight
    const int64_t w_old = present ? (int64_t)o.w[e] : 0;
    const int64_t w_new = (present && !isdel ? w_old : 0) + W;
    if (isins && w_new > INT32_MAX) atomicOr(o.err, kErrOverflow);
    const bool add = isins && !present, rem = !isins && isdel && present;
    dlt = w_new - w_old;
    net = add ? 1 : rem ? -1 : 0;
    f = (isins ? kPairIns : 0) | (isdel ? kPairDel : 0) | (present ? kPairPresent : 0) | (add ? kPairAdded : 0) |
        (rem ? kPairRemoved : 0);
    acc.m2 += dlt;
    if (o.lab0 && dlt != 0 && o.lab0[u] == o.lab0[v]) acc.in += dlt;
    acc.heads++;
  }
  o.pkey[p] = (uint64_t)(uint32_t)u << 32 | (uint32_t)v;
  o.pw[p] = (int32_t)W;
  o.pflag[p] = f;
  o.pdelta[p] = (int32_t)dlt;
  o.epos[p] = e;
  o.net[p] = net;
  return (int32_t)dlt;
}

// First entry of [lo, hi) with a[x] >= v.
template <typename I>
__device__ __forceinline__ I lower_bound_col(const int32_t* a, I lo, I hi, int32_t v) {
  while (lo < hi) {
    const I mid = (lo + hi) >> 1;
    if (a[mid] < v) lo = mid + 1; else hi = mid;
  }
  return lo;
}

// The CTA's sums into the graph's (every thread of the CTA calls it).  uni:
// all records of the CTA belong to graph g.
template <int NT>
__device__ __forceinline__ void pair_sums_out(const PairView& o, int g, const PairSum& acc) {
  __shared__ unsigned long long red[3][NT / 32];
  const unsigned long long m2 = warp_sum((unsigned long long)acc.m2), in = warp_sum((unsigned long long)acc.in);
  const unsigned heads = __reduce_add_sync(0xffffffffu, (unsigned)acc.heads);
  const int wid = threadIdx.x >> 5;
  if (lane_id() == 0) {
    red[0][wid] = m2;
    red[1][wid] = in;
    red[2][wid] = heads;
  }
  __syncthreads();
  if (threadIdx.x == 0) {
    unsigned long long a = 0, b = 0, h = 0;
    for (int x = 0; x < NT / 32; x++) {
      a += red[0][x];
      b += red[1][x];
      h += red[2][x];
    }
    if (a) atomicAdd((unsigned long long*)&o.gs[g].m2, a);
    if (b) atomicAdd((unsigned long long*)&o.gs[g].in_cur, b);
    if (h) atomicAdd((unsigned long long*)o.npairs, h);
  }
  __syncthreads();
}

// A record's sums straight into its graph's (CTAs whose sources belong to
// several graphs).
__device__ __forceinline__ void pair_sums_add(const PairView& o, int g, PairSum& acc) {
  if (acc.m2) atomicAdd((unsigned long long*)&o.gs[g].m2, (unsigned long long)acc.m2);
  if (acc.in) atomicAdd((unsigned long long*)&o.gs[g].in_cur, (unsigned long long)acc.in);
  acc.m2 = acc.in = 0;
}

// Segments of at most kSegSmall records are ranked by pair_tile; of at most
// kSegMid and kSegLarge by a CTA each with a bitonic network in shared memory; of
// at most kSegHuge by a CTA's radix sort in global memory.  Longer ones (a batch
// centred on one vertex, or one that repeats an edge) are only counted on the way
// (DevScalars::n_long): what is merged then is of no use, and when the host has
// read the count, merge_long sorts them over the whole device and merges again.
// The usual batch has none and pays nothing for them.
constexpr int kSegSmall = 64, kSegMid = 512, kSegLarge = 4096, kSegHuge = 32768;

// A CTA takes NS consecutive sources: their records (a counting sort put them
// next to each other) and the columns of their rows are staged in shared memory
// with coalesced loads; a thread then ranks one record in its segment, and in a
// second round takes the record that comes x-th: it sums the weights of equal
// sinks, which are neighbours now, looks the sink up in the row, and writes the
// pair next to its neighbours'.  Sources without records only get their k.
//
// Bound by latency and instructions, not by traffic: a chain of staging, search
// and label gather per CTA, so the tile is small enough for 12 to 16 of them on an
// SM (with 26 KB and 64 registers, 8, and barriers and loads were half of the
// stalls), and the row search, 5-8 probes, which in global memory costs a sector a
// probe and lane, runs on the staged copy.  Segments of other classes and rows
// that do not fit are left out of the staging one by one.
constexpr int kPairThreads = 128;
constexpr int kPairRecs = 640;
constexpr int kPairCols = 2048;
constexpr int kPairRow = 512;  // longest row staged on its own

// NS by the records a source, R / n, so that a CTA has about 64 or more: 2 M
// sources and 12.4 M records take 458 us with 32 sources (555 with the 64 and
// 26 KB of before), 4.2 M sources and 2.0 M records 309 with 128 (485), 2 M and
// 84 K 96 (142).  A graph of fewer sources than four CTAs of 128 an SM has too few
// CTAs of 128 or 64: 32.
inline int64_t pair_wide() { return (int64_t)128 * 4 * num_sms(); }

template <int NS>
__global__ void __launch_bounds__(kPairThreads, 12) pair_tile(PairView o, int64_t n, const uint64_t* __restrict__ rec,
                                                              const int64_t* __restrict__ k_old,
                                                              int64_t* __restrict__ k_new, int32_t* __restrict__ big,
                                                              int32_t* __restrict__ big_cnt,
                                                              int32_t* __restrict__ n_long) {
  static_assert(NS <= kPairThreads, "a thread a source");
  __shared__ uint32_t s_v[kPairRecs], s_w[kPairRecs];  // sinks and weights of the staged records
  __shared__ uint16_t s_perm[kPairRecs];               // record that comes x-th
  __shared__ uint8_t s_src[kPairRecs];                 // its source
  __shared__ int32_t s_col[kPairCols];
  __shared__ int32_t s_off[NS + 1], s_a[NS + 1];  // first record of a source: in the batch, staged
  __shared__ int32_t s_c[NS];                     // first staged column of its row (-1: not staged)
  __shared__ int64_t s_rp[NS + 1];
  __shared__ unsigned long long s_dk[NS];
  const int tid = threadIdx.x;
  const int64_t v0 = (int64_t)blockIdx.x * NS;
  const int ns = (int)(n - v0 < NS ? n - v0 : NS);
  for (int x = tid; x <= ns; x += kPairThreads) {
    s_off[x] = o.off[v0 + x];
    s_rp[x] = o.rp[v0 + x];
  }
  const int64_t kv = tid < ns ? k_old[v0 + tid] : 0;
  if (tid < NS) s_dk[tid] = 0;
  __syncthreads();
  if (s_off[ns] > s_off[0]) {
    // records of the segments ranked here; longer ones: a CTA each, later
    const int len = tid < ns ? s_off[tid + 1] - s_off[tid] : 0;
    const int small = len <= kSegSmall ? len : 0;
    if (len > kSegSmall) {
      const int c = len <= kSegMid ? 0 : len <= kSegLarge ? 1 : 2;
      // (merge_long's sources at the end of the third list)
      const int64_t at = len <= kSegHuge ? (int64_t)c * n + atomicAdd(&big_cnt[c], 1) : 3 * n - 1 - atomicAdd(n_long, 1);
      big[at] = (int32_t)(v0 + tid);
    }
    int nrec;
    const int a0 = block_excl_scan<int, kPairThreads>(small, &nrec);
    if (tid < ns) s_a[tid] = a0;
    if (tid == 0) s_a[ns] = nrec;
    const int64_t c0 = s_rp[0], ncol = s_rp[ns] - c0;
    // a search costs a record about log2(row) probes of a sector each;
    // staging costs an eighth of a sector an entry
    const bool flat = ncol <= kPairCols && ncol <= 32 * (int64_t)nrec;
    if (flat) {
      if (tid < ns) s_c[tid] = (int)(s_rp[tid] - c0);
      for (int x = tid; x < (int)ncol; x += kPairThreads) s_col[x] = ld_stream(o.col + c0 + x);
    } else {
      const int64_t row = tid < ns ? s_rp[tid + 1] - s_rp[tid] : 0;
      const int take = row <= kPairRow && row <= 32 * (int64_t)small ? (int)row : 0;
      int all;
      const int at = block_excl_scan<int, kPairThreads>(take, &all);
      if (tid < ns) s_c[tid] = take > 0 && at + take <= kPairCols ? at : -1;
    }
    __syncthreads();
    if (!flat)
      for (int x = tid >> 5; x < ns; x += kPairThreads / 32) {
        const int at = s_c[x];
        if (at < 0) continue;
        const int64_t b = s_rp[x];
        const int row = (int)(s_rp[x + 1] - b);
        for (int y = lane_id(); y < row; y += 32) s_col[at + y] = ld_stream(o.col + b + y);
      }
    auto source_of = [&](int x) {  // last source whose staged records start at or before x
      int lo = 0, hi = ns - 1;
      while (lo < hi) {
        const int mid = (lo + hi + 1) >> 1;
        if (s_a[mid] <= x) lo = mid; else hi = mid - 1;
      }
      return lo;
    };
    const int g0 = graph_of(o.gid, v0);
    const bool uni = !o.gid || g0 == o.gid[v0 + ns - 1];
    PairSum acc;
    auto put = [&](int lo, int64_t p, uint32_t v, int64_t W, bool isdel, bool head) {
      int64_t e;
      bool present;
      const int cs = s_c[lo];
      const int64_t e0 = s_rp[lo], e1 = s_rp[lo + 1];
      if (cs >= 0) {
        const int q1 = cs + (int)(e1 - e0);
        const int q = lower_bound_col<int>(s_col, cs, q1, (int32_t)v);
        present = q < q1 && s_col[q] == (int32_t)v;
        e = e0 + (q - cs);
      } else {
        e = lower_bound_col<int64_t>(o.col, e0, e1, (int32_t)v);
        present = e < e1 && o.col[e] == (int32_t)v;
      }
      const int32_t u = (int32_t)(v0 + lo);
      const int32_t d = put_pair(o, p, u, (int32_t)v, W, W > 0, isdel, head, e, present, acc);
      if (d) atomicAdd(&s_dk[lo], (unsigned long long)(long long)d);
      if (!uni) pair_sums_add(o, graph_of(o.gid, u), acc);
    };
    if (nrec <= kPairRecs) {
      for (int x = tid; x < nrec; x += kPairThreads) {
        const int lo = source_of(x);
        const uint64_t me = rec[s_off[lo] + (x - s_a[lo])];
        s_src[x] = (uint8_t)lo;
        s_v[x] = (uint32_t)(me >> 32);
        s_w[x] = (uint32_t)me;
      }
      __syncthreads();
      for (int x = tid; x < nrec; x += kPairThreads) {
        const int lo = s_src[x], a = s_a[lo], b = s_a[lo + 1];
        const uint32_t v = s_v[x];
        int rank = a;  // equal sinks keep their order
        for (int j = a; j < x; j++) rank += s_v[j] <= v ? 1 : 0;
        for (int j = x + 1; j < b; j++) rank += s_v[j] < v ? 1 : 0;
        s_perm[rank] = (uint16_t)x;
      }
      __syncthreads();
      for (int x = tid; x < nrec; x += kPairThreads) {
        const int lo = s_src[x], a = s_a[lo], b = s_a[lo + 1];
        const uint32_t v = s_v[s_perm[x]];
        const bool head = x + 1 == b || s_v[s_perm[x + 1]] != v;
        int64_t W = 0;
        bool isdel = false;
        if (head)
          for (int j = x; j >= a; j--) {
            const int y = s_perm[j];
            if (s_v[y] != v) break;
            W += (int64_t)s_w[y];
            isdel |= s_w[y] == 0;
          }
        put(lo, (int64_t)s_off[lo] + (x - a), v, W, isdel, head);
      }
    } else {
      __syncthreads();  // the staged columns
      for (int x = tid; x < nrec; x += kPairThreads) {
        const int lo = source_of(x), m = s_a[lo + 1] - s_a[lo], y = x - s_a[lo];
        const uint64_t* seg = rec + s_off[lo];
        const uint64_t me = seg[y];
        const uint32_t v = (uint32_t)(me >> 32);
        int rank = 0;
        int64_t W = 0;
        bool isdel = false, head = true;
        for (int j = 0; j < m; j++) {
          const uint64_t kj = seg[j];
          const bool before = (uint32_t)(kj >> 32) < v || ((uint32_t)(kj >> 32) == v && j < y);
          rank += before ? 1 : 0;
          if ((uint32_t)(kj >> 32) == v) {
            W += (int64_t)(uint32_t)kj;
            isdel |= (uint32_t)kj == 0;
            head &= before || j == y;
          }
        }
        put(lo, (int64_t)s_off[lo] + rank, v, head ? W : 0, isdel, head);
      }
    }
    __syncthreads();
    pair_sums_out<kPairThreads>(o, g0, acc);
  }
  if (tid < ns) k_new[v0 + tid] = kv + (int64_t)s_dk[tid];
}

// One pair of a long segment whose sorted neighbourhood the caller knows; the
// row is searched in global memory.
__device__ __forceinline__ int32_t put_searched(const PairView& o, int64_t p, int32_t u, uint32_t v, int64_t W,
                                                bool isdel, bool head, PairSum& acc) {
  const int64_t e1 = o.rp[u + 1];
  const int64_t e = lower_bound_col<int64_t>(o.col, o.rp[u], e1, (int32_t)v);
  const bool present = e < e1 && o.col[e] == (int32_t)v;
  return put_pair(o, p, u, (int32_t)v, W, W > 0, isdel, head, e, present, acc);
}

// k and the graph's sums of one long segment.
template <int NT>
__device__ __forceinline__ void segment_out(const PairView& o, int32_t u, const PairSum& acc, int64_t* k_new) {
  const unsigned long long dk = warp_sum((unsigned long long)acc.m2);
  if (lane_id() == 0 && dk) atomicAdd((unsigned long long*)&k_new[u], dk);
  pair_sums_out<NT>(o, graph_of(o.gid, u), acc);
}

// The pairs of a sorted segment s[0 .. len) of source u at place a; s_col: the
// row of u in shared memory (may be NULL).  A record a thread, whole warps: the
// last of a run of equal sinks walks back over it, and what is left of a run of
// more than kRunWalk is summed by the warp (an edge repeated 20,000 times in a
// batch: 1.6 ms by walking alone, 0.23 so).
constexpr int kRunWalk = 32;
template <typename P>
__device__ __forceinline__ void put_sorted(const PairView& o, int32_t u, int64_t a, int len, const P* s, int tid,
                                           int NT, PairSum& acc, const int32_t* s_col = nullptr) {
  const int lane = lane_id();
  for (int x0 = tid & ~31; x0 < len; x0 += NT) {
    const int x = x0 + lane;
    const uint32_t v = x < len ? (uint32_t)(s[x] >> 32) : 0u;
    const bool head = x < len && (x + 1 == len || (uint32_t)(s[x + 1] >> 32) != v);
    int64_t W = 0;
    bool isdel = false;
    int left = 0;  // records of the run before those walked over end here
    if (head) {
      int j = x;
      for (; j >= 0 && x - j < kRunWalk && (uint32_t)(s[j] >> 32) == v; j--) {
        W += (int64_t)(uint32_t)s[j];
        isdel |= (uint32_t)s[j] == 0;
      }
      if (x - j == kRunWalk && j >= 0 && (uint32_t)(s[j] >> 32) == v) left = j + 1;
    }
    for (unsigned more = __ballot_sync(0xffffffffu, left > 0); more; more &= more - 1) {
      const int who = __ffs(more) - 1, end = __shfl_sync(0xffffffffu, left, who);
      const uint32_t vw = __shfl_sync(0xffffffffu, v, who);
      int lo = 0, hi = end;  // first record of the run
      while (lo < hi) {
        const int m = (lo + hi) >> 1;
        if ((uint32_t)(s[m] >> 32) < vw) lo = m + 1; else hi = m;
      }
      unsigned long long sum = 0;
      bool del = false;
      for (int j = lo + lane; j < end; j += 32) {
        sum += (unsigned long long)(uint32_t)s[j];
        del |= (uint32_t)s[j] == 0;
      }
      sum = warp_sum(sum);
      del = __any_sync(0xffffffffu, del);
      if (lane == who) {
        W += (int64_t)sum;
        isdel |= del;
      }
    }
    if (x >= len) continue;
    if (s_col) {
      const int n = (int)(o.rp[u + 1] - o.rp[u]);
      const int q = lower_bound_col<int>(s_col, 0, n, (int32_t)v);
      put_pair(o, a + x, u, (int32_t)v, W, W > 0, isdel, head, o.rp[u] + q, q < n && s_col[q] == (int32_t)v, acc);
    } else {
      put_searched(o, a + x, u, v, W, isdel, head, acc);
    }
  }
}

// In place, P a power of two, by every thread of the CTA.
template <int NT>
__device__ __forceinline__ void bitonic_sort(uint64_t* s, int P) {
  for (int k = 2; k <= P; k <<= 1)
    for (int j = k >> 1; j > 0; j >>= 1) {
      for (int q = threadIdx.x; q < P / 2; q += NT) {
        const int x = ((q & ~(j - 1)) << 1) | (q & (j - 1)), y = x | j;  // the q-th pair at distance j
        const uint64_t kx = s[x], ky = s[y];
        if ((kx > ky) == ((x & k) == 0)) {
          s[x] = ky;
          s[y] = kx;
        }
      }
      __syncthreads();
    }
}

// Segments of kSegSmall + 1 .. kSegMid records: a CTA each, sorted in shared
// memory by a bitonic network (a rank by comparing all pairs takes len^2 / 128
// steps a thread: 373 us for this kernel in a batch of 12.4 M records, with the
// rows searched in global memory and the results written out of order; 126
// so).  The row is staged when it fits: it is at least as long as most segments.
constexpr int kMidThreads = 128;
constexpr int kMidCols = 3072;
__global__ void __launch_bounds__(kMidThreads) pair_mid(PairView o, const uint64_t* __restrict__ rec,
                                                        const int32_t* __restrict__ list,
                                                        const int32_t* __restrict__ cnt, int64_t* __restrict__ k_new) {
  __shared__ uint64_t s[kSegMid];
  __shared__ int32_t s_col[kMidCols];
  const int nl = *cnt, tid = threadIdx.x;
  for (int i = blockIdx.x; i < nl; i += gridDim.x) {
    const int32_t u = list[i];
    const int32_t a = o.off[u];
    const int len = o.off[u + 1] - a;
    const int64_t c0 = o.rp[u], ncol = o.rp[u + 1] - c0;
    int P = 1;
    while (P < len) P <<= 1;
    const bool scol = ncol <= kMidCols && ncol <= 32 * (int64_t)len;  // as in pair_tile
    if (scol)
      for (int x = tid; x < (int)ncol; x += kMidThreads) s_col[x] = ld_stream(o.col + c0 + x);
    for (int x = tid; x < P; x += kMidThreads) s[x] = x < len ? rec[a + x] : ~0ull;
    __syncthreads();
    bitonic_sort<kMidThreads>(s, P);
    PairSum acc;
    put_sorted(o, u, a, len, s, tid, kMidThreads, acc, scol ? s_col : nullptr);
    segment_out<kMidThreads>(o, u, acc, k_new);
  }
}

// Segments of kSegMid + 1 .. kSegLarge records: a CTA each, a bitonic network
// in shared memory, padded to a power of two with the largest key.
constexpr int kLargeThreads = 512;
__global__ void __launch_bounds__(kLargeThreads) pair_large(PairView o, const uint64_t* __restrict__ rec,
                                                            const int32_t* __restrict__ list,
                                                            const int32_t* __restrict__ cnt,
                                                            int64_t* __restrict__ k_new) {
  __shared__ uint64_t s[kSegLarge];
  const int nl = *cnt, tid = threadIdx.x;
  for (int i = blockIdx.x; i < nl; i += gridDim.x) {
    const int32_t u = list[i];
    const int32_t a = o.off[u];
    const int len = o.off[u + 1] - a;
    int P = 1;
    while (P < len) P <<= 1;
    for (int x = tid; x < P; x += kLargeThreads) s[x] = x < len ? rec[a + x] : ~0ull;
    __syncthreads();
    bitonic_sort<kLargeThreads>(s, P);
    PairSum acc;
    put_sorted(o, u, a, len, s, tid, kLargeThreads, acc);
    segment_out<kLargeThreads>(o, u, acc, k_new);
  }
}

// Longer segments: a CTA each, a stable LSD radix sort by sink in global
// memory (8-bit digits; x and y swap per digit), then as above.
constexpr int kHugeThreads = 512;
__global__ void __launch_bounds__(kHugeThreads) pair_huge(PairView o, uint64_t* rec, uint64_t* tmp,
                                                          const int32_t* __restrict__ list,
                                                          const int32_t* __restrict__ cnt, int bits,
                                                          int64_t* __restrict__ k_new) {
  constexpr int NW = kHugeThreads / 32;
  __shared__ uint32_t base[256], wcnt[NW][256];
  const int nl = *cnt, tid = threadIdx.x, wid = tid >> 5;
  for (int i = blockIdx.x; i < nl; i += gridDim.x) {
    const int32_t u = list[i];
    const int32_t a = o.off[u];
    const int len = o.off[u + 1] - a;
    uint64_t *x = rec + a, *y = tmp + a;
    for (int b = 32; b < 32 + bits; b += 8) {
      if (tid < 256) base[tid] = 0;
      for (int q = tid; q < NW * 256; q += kHugeThreads) (&wcnt[0][0])[q] = 0;
      __syncthreads();
      for (int e = tid; e < len; e += kHugeThreads) atomicAdd(&base[(uint32_t)(x[e] >> b) & 255u], 1u);
      __syncthreads();
      if (wid == 0) {  // exclusive scan of the 256 digit counts
        uint32_t run = 0;
        for (int q = 0; q < 8; q++) {
          const uint32_t c = base[q * 32 + lane_id()];
          const uint32_t inc = warp_incl_scan(c);
          base[q * 32 + lane_id()] = run + inc - c;
          run += __shfl_sync(0xffffffffu, inc, 31);
        }
      }
      __syncthreads();
      for (int e0 = 0; e0 < len; e0 += kHugeThreads) {
        const int e = e0 + tid;
        const bool ok = e < len;
        const uint64_t key = ok ? x[e] : 0;
        const uint32_t d = ok ? (uint32_t)(key >> b) & 255u : 256u;
        const unsigned peers = __match_any_sync(0xffffffffu, d);
        const int rk = __popc(peers & lanemask_lt());
        if (ok && rk == 0) wcnt[wid][d] = __popc(peers);
        __syncthreads();
        if (tid < 256) {  // thread t owns digit t: the warps' places, then the next round's base
          uint32_t run = base[tid];
          for (int q = 0; q < NW; q++) {
            const uint32_t c = wcnt[q][tid];
            wcnt[q][tid] = run;
            run += c;
          }
          base[tid] = run;
        }
        __syncthreads();
        if (ok) y[wcnt[wid][d] + rk] = key;
        __syncthreads();
        for (int q = tid; q < NW * 256; q += kHugeThreads) (&wcnt[0][0])[q] = 0;
        __syncthreads();
      }
      uint64_t* t = x;
      x = y;
      y = t;
    }
    PairSum acc;
    put_sorted(o, u, a, len, x, tid, kHugeThreads, acc);
    segment_out<kHugeThreads>(o, u, acc, k_new);
  }
}

// ---- segments above kSegHuge (merge_long) ----
//
// Their records are copied to one array, keyed by (place in the list of these
// sources, sink), sorted by the device-wide radix sort, and a record a thread
// becomes a pair: the last of a run of equal sinks takes the run's weights as a
// difference of their prefix sums, so neither a long segment nor a long run of one
// pair is ever one thread's or one CTA's work.
// 1 M records on one source: the merge takes 1.2 ms so and 9.7 with a CTA's radix
// sort in global memory (0.26 when they are spread); 1 M records of one pair 1.1 and
// 87.  A CTA's sort is the faster one to
// about 30 K records (20 K: 0.33 against 0.39 ms; 65 K: 0.76 and 0.47).

__global__ void long_sizes(const int32_t* __restrict__ list, int64_t n_long, const int32_t* __restrict__ off,
                           int64_t* __restrict__ len) {
  for (int64_t i = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; i <= n_long; i += (int64_t)gridDim.x * blockDim.x)
    len[i] = i < n_long ? off[list[i] + 1] - off[list[i]] : 0;
}

__global__ void long_keys(const int32_t* __restrict__ list, int64_t n_long, const int64_t* __restrict__ first,
                          const int32_t* __restrict__ off, const uint64_t* __restrict__ rec, int64_t T,
                          uint64_t* __restrict__ key, uint32_t* __restrict__ val) {
  for (int64_t x = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; x < T; x += (int64_t)gridDim.x * blockDim.x) {
    int64_t lo = 0, hi = n_long - 1;  // last segment that starts at or before x
    while (lo < hi) {
      const int64_t mid = (lo + hi + 1) >> 1;
      if (first[mid] <= x) lo = mid; else hi = mid - 1;
    }
    const uint64_t r = rec[off[list[lo]] + (x - first[lo])];
    key[x] = (uint64_t)lo << 32 | r >> 32;
    val[x] = (uint32_t)r;
  }
}

// Weights and deletes of the sorted records, to be scanned.
__global__ void long_terms(const uint32_t* __restrict__ val, int64_t T, int64_t* __restrict__ ws,
                           int32_t* __restrict__ ds) {
  for (int64_t x = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; x <= T; x += (int64_t)gridDim.x * blockDim.x) {
    ws[x] = x < T ? (int64_t)val[x] : 0;
    ds[x] = x < T && val[x] == 0 ? 1 : 0;
  }
}

// The pairs, a warp per kLongChunk sorted records; the sums of a chunk within one
// segment are added once.
constexpr int kLongChunk = 1024;
__global__ void __launch_bounds__(256) long_pairs(PairView o, const int32_t* __restrict__ list,
                                                  const int64_t* __restrict__ first, const uint64_t* __restrict__ key,
                                                  const int64_t* __restrict__ ws, const int32_t* __restrict__ ds,
                                                  int64_t T, int64_t* __restrict__ k_new) {
  const int lane = lane_id();
  const int64_t nw = ((int64_t)gridDim.x * blockDim.x) >> 5;
  for (int64_t c0 = ((blockIdx.x * (int64_t)blockDim.x + threadIdx.x) >> 5) * kLongChunk; c0 < T; c0 += nw * kLongChunk) {
    const int64_t c1 = c0 + kLongChunk < T ? c0 + kLongChunk : T;
    PairSum acc;
    auto add = [&](int32_t u, unsigned long long m2, unsigned long long in, unsigned heads) {
      GraphState& gs = o.gs[graph_of(o.gid, u)];
      if (m2) {
        atomicAdd((unsigned long long*)&k_new[u], m2);
        atomicAdd((unsigned long long*)&gs.m2, m2);
      }
      if (in) atomicAdd((unsigned long long*)&gs.in_cur, in);
      if (heads) atomicAdd((unsigned long long*)o.npairs, (unsigned long long)heads);
    };
    const bool one = key[c0] >> 32 == key[c1 - 1] >> 32;  // the chunk lies in one segment
    for (int64_t x0 = c0; x0 < c1; x0 += 32) {
      const int64_t x = x0 + lane;
      if (x < c1) {
        const uint64_t kx = key[x];
        const int64_t i = (int64_t)(kx >> 32);
        const int32_t u = list[i];
        const uint32_t v = (uint32_t)kx;
        const bool head = x + 1 == T || key[x + 1] != kx;
        int64_t W = 0;
        bool isdel = false;
        if (head) {
          int64_t lo = first[i], hi = x;  // first record of the run
          while (lo < hi) {
            const int64_t mid = (lo + hi) >> 1;
            if (key[mid] < kx) lo = mid + 1; else hi = mid;
          }
          W = ws[x + 1] - ws[lo];
          isdel = ds[x + 1] != ds[lo];
        }
        put_searched(o, o.off[u] + (x - first[i]), u, v, W, isdel, head, acc);
        if (!one) {
          add(u, (unsigned long long)acc.m2, (unsigned long long)acc.in, (unsigned)acc.heads);
          acc = PairSum();
        }
      }
    }
    if (one) {
      const unsigned long long m2 = warp_sum((unsigned long long)acc.m2), in = warp_sum((unsigned long long)acc.in);
      const unsigned heads = __reduce_add_sync(0xffffffffu, (unsigned)acc.heads);
      if (lane == 0) add(list[key[c0] >> 32], m2, in, heads);
    }
  }
}

// The entries every pair adds or removes, again (the scan took them).
__global__ void pair_net(const uint8_t* __restrict__ pflag, int64_t R, int32_t* __restrict__ net) {
  for (int64_t p = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; p <= R; p += (int64_t)gridDim.x * blockDim.x) {
    const uint8_t f = p < R ? pflag[p] : 0;
    net[p] = f & kPairAdded ? 1 : f & kPairRemoved ? -1 : 0;
  }
}

// sum_i e_{i->C(i)} and 2m of G_{t-1} per graph (kept by the previous update:
// prev[g], prev[G + g]); with_in: the former is tracked through the merge.
__global__ void seed_sums(GraphState* __restrict__ gs, int G, const int64_t* __restrict__ prev, int with_in) {
  for (int g = blockIdx.x * blockDim.x + threadIdx.x; g < G; g += gridDim.x * blockDim.x) {
    gs[g].in_cur += with_in ? prev[g] : 0;
    gs[g].m2 += prev[G + g];
  }
}

// Sums over every entry of a graph, entry-linear: a warp takes a range of entries
// whatever rows they belong to (a warp a row, as these once were, takes 4 ms for a
// row of 400,000 entries).
//
// k of a graph whose degrees no update of this context has computed (a loaded
// checkpoint), zeroed before, and its 2m into *m2.
__global__ void __launch_bounds__(256) row_degrees(int64_t n, int64_t m, const int64_t* __restrict__ rp,
                                                   const int32_t* __restrict__ w, int64_t per_warp,
                                                   unsigned long long* __restrict__ k,
                                                   unsigned long long* __restrict__ m2) {
  const int lane = lane_id();
  const int64_t gw = (blockIdx.x * (int64_t)blockDim.x + threadIdx.x) >> 5;
  const int64_t W0 = gw * per_warp, W1 = W0 + per_warp < m ? W0 + per_warp : m;
  if (W0 >= W1) return;
  RowWalk rw;
  rw.start(rp, n, W0);
  unsigned long long acc = 0, tot = 0;  // of row cur, a lane's share
  int64_t cur = -1;
  auto flush = [&]() {
    acc = warp_sum(acc);
    if (lane == 0 && acc) atomicAdd(&k[cur], acc);
    acc = 0;
  };
  for (int64_t c0 = W0; c0 < W1; c0 += 32) {
    const bool valid = c0 + lane < W1;
    const int64_t r = rw.row(rp, n, c0, valid);
    const unsigned long long x = valid ? (unsigned long long)ld_stream(w + c0 + lane) : 0ull;
    tot += x;
    const int64_t r0 = __shfl_sync(0xffffffffu, r, 0);
    const bool one = __all_sync(0xffffffffu, !valid || r == r0);
    if (cur >= 0 && !(one && r0 == cur)) flush();
    if (one) {
      cur = r0;
      acc += x;
    } else {  // several rows: a run each
      const unsigned peers = __match_any_sync(0xffffffffu, (unsigned long long)(valid ? r : -1));
      const int64_t sum = group_sum_exact(peers, (int64_t)x);
      if (valid && (int)(__ffs(peers) - 1) == lane) atomicAdd(&k[r], (unsigned long long)sum);
      cur = -1;
    }
  }
  if (cur >= 0) flush();
  tot = warp_sum(tot);
  if (lane == 0 && tot) atomicAdd(m2, tot);
}

// sum_i e_{i->C(i)} under labels L (when no update kept it: labels set by the
// caller, a loaded checkpoint; one graph).  *nnz: the entries.
__global__ void __launch_bounds__(256) in_weight(int64_t n, const int64_t* __restrict__ rp,
                                                 const int32_t* __restrict__ col, const int32_t* __restrict__ w,
                                                 const int32_t* __restrict__ L, GraphState* __restrict__ gs,
                                                 const int32_t* __restrict__ n_long) {
  if (*n_long) return;  // the rows are not merged yet
  constexpr int U = 4;
  const int lane = lane_id();
  const int64_t m = rp[n], warps = ((int64_t)gridDim.x * blockDim.x) >> 5;
  const int64_t per_warp = (((m + warps - 1) / warps) + 32 * U - 1) / (32 * U) * (32 * U);
  const int64_t gw = (blockIdx.x * (int64_t)blockDim.x + threadIdx.x) >> 5;
  const int64_t W0 = gw * per_warp, W1 = W0 + per_warp < m ? W0 + per_warp : m;
  if (W0 >= W1) return;
  RowWalk rw;
  rw.start(rp, n, W0);
  unsigned long long acc = 0;
  for (int64_t c0 = W0; c0 < W1; c0 += 32 * U) {
    int32_t y[U], x[U];
#pragma unroll
    for (int q = 0; q < U; q++) {
      const int64_t e = c0 + q * 32 + lane;
      y[q] = e < W1 ? ld_stream(col + e) : -1;
      x[q] = e < W1 ? ld_stream(w + e) : 0;
    }
#pragma unroll
    for (int q = 0; q < U; q++) y[q] = y[q] >= 0 ? L[y[q]] : -1;
#pragma unroll
    for (int q = 0; q < U; q++) {
      const int64_t c = c0 + q * 32;
      if (c < W1 && L[rw.row(rp, n, c, c + lane < W1)] == y[q]) acc += (unsigned long long)x[q];  // (c < W1: uniform)
    }
  }
  acc = warp_sum(acc);
  if (lane == 0 && acc) atomicAdd((unsigned long long*)&gs[0].in_cur, acc);
}

// ---- tiled merge ----
//
// The merge as one merge of two sorted sequences: the old entries, in CSR
// order, and the pairs, where pair q comes before entry epos[q].  Pair q is
// item q + epos[q] of the merged sequence.  With S(q) the entries added minus
// removed by the pairs before q, an old entry e lands at e + S over the pairs
// with epos <= e, and an added pair q at epos[q] + S(q); neither depends on
// the row, so the sequence is cut into tiles of kMergeTile items whatever
// rows they cover.
constexpr int kMergeTile = 2048;
constexpr int kMergeThreads = 256;
constexpr int kMergeItems = kMergeTile / kMergeThreads;

// Row u's start in the new CSR.
__global__ void new_rows(const int64_t* __restrict__ rp_o, const int32_t* __restrict__ off,
                         const int32_t* __restrict__ S, int64_t n, int64_t* __restrict__ rp_n) {
  for (int64_t u = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; u <= n; u += (int64_t)gridDim.x * blockDim.x)
    rp_n[u] = rp_o[u] + S[off[u]];
}

// Pairs before merged item t * kMergeTile.  *npair: the pairs there are (fewer
// than the batch's records when bad records took no place; the update then
// fails, but stays within its buffers).  While segments are left to merge_long
// (*n_long), their pairs hold nothing yet: no pairs, and merge_tile copies the old
// entries, which the next merge overwrites (a test in merge_tile for an early return
// cost it 37 us of 660 at 73 M entries and 12.4 M pairs).
__global__ void merge_split(const int64_t* __restrict__ epos, const int32_t* __restrict__ npair, int64_t nt,
                            int32_t* __restrict__ sq, const int32_t* __restrict__ n_long) {
  const int64_t P = *n_long ? 0 : *npair;
  const int lane = lane_id();
  const int64_t nw = ((int64_t)gridDim.x * blockDim.x) >> 5;
  // a warp a tile: 32 probes a step, so that the chain is log32 of the pairs
  for (int64_t t = (blockIdx.x * (int64_t)blockDim.x + threadIdx.x) >> 5; t <= nt; t += nw) {
    const int64_t d = t * kMergeTile;
    int64_t lo = 0, hi = P < d ? P : d;  // first q with q + epos[q] >= d
    while (lo < hi) {
      const int64_t step = (hi - lo + 31) / 32, q = lo + lane * step;
      const unsigned below = __ballot_sync(0xffffffffu, q < hi && q + epos[q] < d);  // a prefix of the lanes
      const int k = __popc(below);
      if (k == 0) {
        hi = lo;
      } else {
        const int64_t last = lo + (k - 1) * step;  // below d
        lo = last + 1;
        hi = last + step < hi ? last + step : hi;
      }
    }
    if (lane == 0) sq[t] = (int32_t)lo;
  }
}

// One tile.  The work beyond the copy is per pair: a pair marks the entry it
// changes (or whose successors it shifts) in shared memory, one block scan
// turns the marks into shifts, and a tile without pairs is a plain shifted
// copy.  Bound by the 16 bytes an entry: 80 M entries and 84 k pairs take
// 233 us (5.5 TB/s), 73 M entries and 12.4 M pairs 375 us.  With the per-entry
// searches (row of an entry, its place among the pairs) and row sums that ran
// here before, it was issue-bound: 1059 and 1534 us.
//
// NL: also the entry labels (label of every entry's column under lab; NULL: the
// column itself) of the new graph, for an update that will need them.  80 M
// entries and 84 K pairs: 480 us, where the copy alone takes 233 and the gather
// alone 316; both count against the rate of L2 sectors (one a gathered label,
// 5/8 of one for the streams of an entry), so what is saved is the second read of
// the columns and a launch.
template <bool NL>
__global__ void __launch_bounds__(kMergeThreads) merge_tile(
    int64_t nnz, const int32_t* __restrict__ col_o, const int32_t* __restrict__ w_o,
    const int32_t* __restrict__ sq, const int64_t* __restrict__ epos, const uint64_t* __restrict__ pkey,
    const int32_t* __restrict__ pdelta, const uint8_t* __restrict__ pflag, const int32_t* __restrict__ S,
    int32_t* __restrict__ col_n, int32_t* __restrict__ w_n, const int32_t* __restrict__ lab,
    int32_t* __restrict__ nlab) {
  __shared__ int32_t s_sh[kMergeTile + kMergeThreads];  // shift marks, then shifts (padded: one word a thread's run)
  __shared__ int32_t s_adj[kMergeTile];                 // weight change of an entry; INT32_MIN: removed
  auto at = [](int i) { return i + i / kMergeItems; };
  const int tid = threadIdx.x;
  const int64_t t = blockIdx.x;
  const int32_t q0 = sq[t], q1 = sq[t + 1];
  const int64_t e0 = t * kMergeTile - q0;
  const int64_t e1x = (t + 1) * kMergeTile - q1;
  const int64_t e1 = e1x < nnz ? e1x : nnz;
  const int ne = e1 > e0 ? (int)(e1 - e0) : 0, np = q1 - q0;
  const int32_t shift0 = S[q0];
  int32_t c[kMergeItems], w[kMergeItems];
#pragma unroll
  for (int x = 0; x < kMergeItems; x++) {
    const int j = x * kMergeThreads + tid;
    if (j < ne) {
      c[x] = ld_stream(col_o + e0 + j);
      w[x] = ld_stream(w_o + e0 + j);
    }
  }
  int32_t l[kMergeItems];
  if constexpr (NL) {
#pragma unroll
    for (int x = 0; x < kMergeItems; x++)
      if (x * kMergeThreads + tid < ne) l[x] = lab ? lab[c[x]] : c[x];
  }
  // the last pair before the tile may stand for the tile's first entry
  const bool lead = q0 > 0 && ne > 0 && epos[q0 - 1] == e0 && (pflag[q0 - 1] & kPairPresent);
  if (np == 0 && !lead) {
#pragma unroll
    for (int x = 0; x < kMergeItems; x++) {
      const int j = x * kMergeThreads + tid;
      if (j < ne) {
        st_stream(col_n + e0 + shift0 + j, c[x]);
        st_stream(w_n + e0 + shift0 + j, w[x]);
        if constexpr (NL) st_stream(nlab + e0 + shift0 + j, l[x]);
      }
    }
    return;
  }
  for (int j = tid; j < kMergeTile; j += kMergeThreads) {
    s_sh[at(j)] = 0;
    s_adj[j] = 0;
  }
  __syncthreads();
  if (lead && tid == 0) s_adj[0] = (pflag[q0 - 1] & kPairRemoved) ? INT32_MIN : pdelta[q0 - 1];
  for (int j = tid; j < np; j += kMergeThreads) {
    const int32_t q = q0 + j;
    const uint32_t f = pflag[q];
    if (f & (kPairAdded | kPairPresent)) {
      const int64_t ep = epos[q];
      const int rel = (int)(ep - e0);  // 0 .. ne
      const int32_t d = pdelta[q];
      if (f & kPairAdded) {
        const int64_t pos = ep + S[q];
        const int32_t v = (int32_t)(pkey[q] & 0xffffffffu);
        st_stream(col_n + pos, v);
        st_stream(w_n + pos, d);
        if constexpr (NL) st_stream(nlab + pos, lab ? lab[v] : v);
        if (rel < ne) atomicAdd(&s_sh[at(rel)], 1);
      } else if (rel < ne) {
        if (f & kPairRemoved) {
          s_adj[rel] = INT32_MIN;
          atomicAdd(&s_sh[at(rel)], -1);  // its successors move; the entry itself is gone
        } else {
          s_adj[rel] = d;
        }
      }
    }
  }
  __syncthreads();
  int32_t m[kMergeItems], sum = 0, all;
#pragma unroll
  for (int x = 0; x < kMergeItems; x++) {
    m[x] = s_sh[at(tid * kMergeItems + x)];
    sum += m[x];
  }
  int32_t run = block_excl_scan<int32_t, kMergeThreads>(sum, &all) + shift0;
#pragma unroll
  for (int x = 0; x < kMergeItems; x++) {
    run += m[x];
    s_sh[at(tid * kMergeItems + x)] = run;
  }
  __syncthreads();
#pragma unroll
  for (int x = 0; x < kMergeItems; x++) {
    const int j = x * kMergeThreads + tid;
    if (j < ne) {
      const int32_t d = s_adj[j];
      if (d != INT32_MIN) {
        const int64_t pos = e0 + j + s_sh[at(j)];
        st_stream(col_n + pos, c[x]);
        st_stream(w_n + pos, w[x] + d);
        if constexpr (NL) st_stream(nlab + pos, l[x]);
      }
    }
  }
}

}  // namespace

int validate_batch(dcd_ctx* c, const dcd_edge* ins, int64_t n_ins, const dcd_edge* del, int64_t n_del, bool* ok) {
  cudaStream_t s = c->stream;
  uint32_t* err = &c->dsc.get()->err;
  *ok = true;
  if (n_ins + n_del == 0) return DCD_OK;
  DCD_TRY_CUDA(cudaMemsetAsync(err, 0, sizeof(uint32_t), s));
  ::dcd::count_launch(), validate_records<<<grid_for(n_ins + n_del, 256), 256, 0, s>>>(ins, n_ins, del, n_del, c->n,
                                                                                       err);
  DCD_LAUNCH_CHECK();
  DCD_TRY_CUDA(cudaMemcpyAsync(c->hscratch, err, sizeof(uint32_t), cudaMemcpyDeviceToHost, s));
  DCD_TRY_CUDA(cudaStreamSynchronize(s));
  *ok = !(*reinterpret_cast<uint32_t*>(c->hscratch) & kErrBadRecord);
  return DCD_OK;
}

namespace {

PairView pair_view(dcd_ctx* c, const int32_t* labels0, const MergeOut& m) {
  const int cur = c->cur;
  DevScalars* d = c->dsc.get();
  return PairView{m.pair_ptr.get(), c->rp[cur].get(), c->col[cur].get(), c->w[cur].get(),
                  m.track_in ? labels0 : nullptr, c->G > 1 ? c->gid.get() : nullptr, m.pkey.get(), m.pw.get(),
                  m.pflag.get(), m.pdelta.get(), m.epos.get(), m.S.get(), c->gs.get(), &d->npairs, &d->err};
}

// G_t's rows from G_{t-1}'s and the pairs (of no use yet while segments are left to merge_long).
int merge_rows(dcd_ctx* c, const int32_t* labels0, bool static_start, MergeOut* out, EntryLabels* nlab) {
  cudaStream_t s = c->stream;
  const int64_t n = c->n, R = out->npairs, n_ins = c->n_ins;
  DevScalars* d = c->dsc.get();
  const int T = 256;
  const int cur = c->cur, nxt = 1 - c->cur;
  const int64_t* rp_o = c->rp[cur].get();
  const int32_t* col_o = c->col[cur].get();
  const int32_t* w_o = c->w[cur].get();
  const int32_t* gid = c->G > 1 ? c->gid.get() : nullptr;
  const int32_t* off = out->pair_ptr.get();
  Buf<int64_t>& epos = out->epos;
  Buf<int32_t>& S = out->S;
  Buf<int32_t> stmp;
  DCD_TRY(stmp.alloc(&c->mem, scan_tmp_count(R + 1)));
  DCD_TRY(exclusive_scan<int32_t>(S.get(), S.get(), R + 1, nullptr, stmp.get(), s));

  // ---- new row pointers, merge ----
  const int64_t cap = c->nnz + 2 * n_ins;
  DCD_TRY(c->rp[nxt].ensure(&c->mem, n + 1));
  DCD_TRY(c->col[nxt].ensure(&c->mem, cap));
  DCD_TRY(c->w[nxt].ensure(&c->mem, cap));
  int64_t* rp_n = c->rp[nxt].get();
  ::dcd::count_launch(), new_rows<<<grid_for(n + 1, T), T, 0, s>>>(rp_o, off, S.get(), n, rp_n);
  DCD_LAUNCH_CHECK();
  const int64_t nt = cdiv(c->nnz + R, (int64_t)kMergeTile);
  if (nt > 0) {
    Buf<int32_t> split;
    DCD_TRY(split.alloc(&c->mem, nt + 1));
    ::dcd::count_launch(), merge_split<<<grid_for((nt + 1) * 32, T), T, 0, s>>>(epos.get(), off + n, nt, split.get(),
                                                                              &d->n_long);
    DCD_LAUNCH_CHECK();
    if (nlab && nlab->buf.n < (size_t)cap) DCD_TRY(nlab->buf.alloc(&c->mem, cap));
    ::dcd::count_launch(), (nlab ? merge_tile<true> : merge_tile<false>)<<<(unsigned)nt, kMergeThreads, 0, s>>>(
        c->nnz, col_o, w_o, split.get(), epos.get(), out->pkey.get(), out->pdelta.get(), out->pflag.get(), S.get(),
        c->col[nxt].get(), c->w[nxt].get(), static_start ? nullptr : labels0, nlab ? nlab->buf.get() : nullptr);
    DCD_LAUNCH_CHECK();
    if (nlab) nlab->ready = true;
  }
  if (!static_start && !c->in_valid && c->cfg.alg == DCD_ALG_LOUVAIN) {
    ::dcd::count_launch(), in_weight<<<wave_grid(in_weight, cap, T), T, 0, s>>>(n, rp_n, c->col[nxt].get(),
                                                                                c->w[nxt].get(), labels0, c->gs.get(),
                                                                                &d->n_long);
    DCD_LAUNCH_CHECK();
  }
  return DCD_OK;
}

}  // namespace

int merge_batch(dcd_ctx* c, const int32_t* labels0, bool static_start, MergeOut* out, EntryLabels* nlab) {
  cudaStream_t s = c->stream;
  const int64_t n = c->n;
  const int64_t n_ins = c->n_ins, n_del = c->n_del, nr = n_ins + n_del;
  const int64_t R = 2 * nr;
  DevScalars* d = c->dsc.get();
  const int T = 256;
  const int cur = c->cur, nxt = 1 - c->cur;
  const int64_t* rp_o = c->rp[cur].get();
  const int32_t* col_o = c->col[cur].get();
  const int32_t* w_o = c->w[cur].get();
  const int32_t* gid = c->G > 1 ? c->gid.get() : nullptr;

  // ---- degrees and sums of G_{t-1} ----
  if (!c->k_valid) {
    DCD_TRY(c->kdeg[cur].ensure(&c->mem, n));
    DCD_TRY(c->in_prev.ensure(&c->mem, 2 * (size_t)c->G));
    DCD_TRY_CUDA(cudaMemsetAsync(c->in_prev.get(), 0, 2 * c->G * sizeof(int64_t), s));
    DCD_TRY_CUDA(cudaMemsetAsync(c->kdeg[cur].get(), 0, n * sizeof(int64_t), s));
    if (c->nnz > 0) {  // a loaded checkpoint: one graph
      const int grid = wave_grid(row_degrees, c->nnz, T);
      const int64_t per_warp = cdiv(cdiv(c->nnz, (int64_t)grid * (T / 32)), 32) * 32;
      ::dcd::count_launch(), row_degrees<<<grid, T, 0, s>>>(
          n, c->nnz, rp_o, w_o, per_warp, reinterpret_cast<unsigned long long*>(c->kdeg[cur].get()),
          reinterpret_cast<unsigned long long*>(c->in_prev.get() + c->G));
      DCD_LAUNCH_CHECK();
    }
    c->k_valid = true;
  }
  DCD_TRY(c->kdeg[nxt].ensure(&c->mem, n));
  out->k = &c->kdeg[nxt];
  // sum_i e_{i->C(i)} under the start labels on G_t: zero for a static start
  // (singletons, no self-loops); from the previous update's value plus the
  // batch's change when the context kept it (in_valid); else summed over
  // every entry of G_t
  const bool from_prev = !static_start && c->in_valid;
  DCD_TRY_CUDA(cudaMemsetAsync(c->gs.get(), 0, c->G * sizeof(GraphState), s));

  // ---- records by source ----
  Buf<int2> rank;
  Buf<uint64_t> rec2;
  Buf<int32_t> stmp;
  Buf<uint64_t>& rec = out->rec;
  Buf<int32_t>& big = out->big;
  out->npairs = R;
  DCD_TRY(out->pair_ptr.alloc(&c->mem, n + 4));  // + 3: the counts of the long segments' lists
  DCD_TRY(out->pkey.alloc(&c->mem, R));
  DCD_TRY(out->pw.alloc(&c->mem, R));
  DCD_TRY(out->pflag.alloc(&c->mem, R));
  DCD_TRY(out->pdelta.alloc(&c->mem, R));
  DCD_TRY(stmp.alloc(&c->mem, scan_tmp_count(n + 1)));
  DCD_TRY(out->epos.alloc(&c->mem, R));
  DCD_TRY(out->S.alloc(&c->mem, R + 1));
  Buf<int32_t>& S = out->S;
  int32_t* off = out->pair_ptr.get();
  int32_t* big_cnt = off + n + 1;
  DCD_TRY_CUDA(cudaMemsetAsync(off, 0, (n + 4) * sizeof(int32_t), s));
  DCD_TRY_CUDA(cudaMemsetAsync(S.get() + R, 0, sizeof(int32_t), s));
  if (R > 0) {
    DCD_TRY(rank.alloc(&c->mem, nr));
    DCD_TRY(rec.alloc(&c->mem, R));
    if (nr > kSegLarge) DCD_TRY(rec2.alloc(&c->mem, R));
    DCD_TRY(big.alloc(&c->mem, 3 * n));
    ::dcd::count_launch(), rec_count<<<grid_for(nr, T), T, 0, s>>>(c->ins.get(), n_ins, c->del.get(), n_del, n, off,
                                                                    rank.get(), &d->err);
    DCD_LAUNCH_CHECK();
    DCD_TRY(exclusive_scan<int32_t>(off, off, n + 1, nullptr, stmp.get(), s));
    ::dcd::count_launch(), rec_scatter<<<grid_for(nr, T), T, 0, s>>>(c->ins.get(), n_ins, c->del.get(), n_del, n, off,
                                                                      rank.get(), rec.get());
    DCD_LAUNCH_CHECK();
  }
  out->track_in = from_prev;
  const PairView o = pair_view(c, labels0, *out);
  if (R > 0) {
    // sources a CTA: about 64 records for its 128 threads (pair_tile)
    const int ns = R >= 2 * n || n < pair_wide() ? 32 : 2 * R >= n ? 64 : 128;
    auto* tile = ns == 32 ? pair_tile<32> : ns == 64 ? pair_tile<64> : pair_tile<128>;
    ::dcd::count_launch(), tile<<<(unsigned)cdiv(n, ns), kPairThreads, 0, s>>>(
        o, n, rec.get(), c->kdeg[cur].get(), out->k->get(), big.get(), big_cnt, &d->n_long);
    // a segment holds at most one record per batch record: the classes the
    // batch is too small for are not launched
    if (nr > kSegSmall)
      ::dcd::count_launch(), pair_mid<<<grid_for(nr, kSegSmall, 16), kMidThreads, 0, s>>>(
          o, rec.get(), big.get(), big_cnt, out->k->get());
    if (nr > kSegMid)
      ::dcd::count_launch(), pair_large<<<grid_for(nr, kSegMid, 4), kLargeThreads, 0, s>>>(
          o, rec.get(), big.get() + n, big_cnt + 1, out->k->get());
    if (nr > kSegLarge)
      ::dcd::count_launch(), pair_huge<<<grid_for(nr, kSegLarge, 2), kHugeThreads, 0, s>>>(
          o, rec.get(), rec2.get(), big.get() + 2 * n, big_cnt + 2, bits_for(n - 1), out->k->get());
    DCD_LAUNCH_CHECK();
  } else {
    DCD_TRY_CUDA(cudaMemcpyAsync(out->k->get(), c->kdeg[cur].get(), n * sizeof(int64_t), cudaMemcpyDeviceToDevice, s));
  }
  ::dcd::count_launch(), seed_sums<<<cdiv(c->G, 128), 128, 0, s>>>(c->gs.get(), c->G, c->in_prev.get(),
                                                                    from_prev ? 1 : 0);
  DCD_LAUNCH_CHECK();
  return merge_rows(c, labels0, static_start, out, nlab);
}

int merge_long(dcd_ctx* c, const int32_t* labels0, bool static_start, int64_t n_long, MergeOut* out,
               EntryLabels* nlab) {
  cudaStream_t s = c->stream;
  const int64_t n = c->n, R = out->npairs;
  DevScalars* d = c->dsc.get();
  const int T = 256;
  const int32_t* off = out->pair_ptr.get();
  const int32_t* list = out->big.get() + 3 * n - n_long;
  Buf<int64_t> first, ws;
  Buf<int64_t> ltmp;
  DCD_TRY(first.alloc(&c->mem, n_long + 1));
  DCD_TRY(ltmp.alloc(&c->mem, scan_tmp_count(n_long + 1)));
  ::dcd::count_launch(), long_sizes<<<grid_for(n_long + 1, T), T, 0, s>>>(list, n_long, off, first.get());
  DCD_LAUNCH_CHECK();
  DCD_TRY(exclusive_scan<int64_t>(first.get(), first.get(), n_long + 1, nullptr, ltmp.get(), s));
  DCD_TRY_CUDA(cudaMemcpyAsync(c->hscratch, first.get() + n_long, sizeof(int64_t), cudaMemcpyDeviceToHost, s));
  DCD_TRY_CUDA(cudaStreamSynchronize(s));
  const int64_t recs = c->hscratch[0];
  Buf<uint64_t> k0, k1;
  Buf<uint32_t> v0, v1, stmp;
  Buf<int64_t> wtmp;
  Buf<int32_t> ds;
  DCD_TRY(k0.alloc(&c->mem, recs));
  DCD_TRY(k1.alloc(&c->mem, recs));
  DCD_TRY(v0.alloc(&c->mem, recs));
  DCD_TRY(v1.alloc(&c->mem, recs));
  DCD_TRY(stmp.alloc(&c->mem, sort_tmp_words(recs) + scan_tmp_count(recs + 1)));
  ::dcd::count_launch(), long_keys<<<grid_for(recs, T), T, 0, s>>>(list, n_long, first.get(), off, out->rec.get(), recs,
                                                                   k0.get(), v0.get());
  DCD_LAUNCH_CHECK();
  const int ranges[4] = {0, bits_for(n - 1), 32, 32 + bits_for(n_long - 1)};
  bool in1 = false;
  DCD_TRY(sort_pairs<uint32_t>(k0.get(), v0.get(), k1.get(), v1.get(), recs, ranges, 2, stmp.get(), &in1, s));
  DCD_TRY(ws.alloc(&c->mem, recs + 1));
  DCD_TRY(ds.alloc(&c->mem, recs + 1));
  DCD_TRY(wtmp.alloc(&c->mem, scan_tmp_count(recs + 1)));
  ::dcd::count_launch(), long_terms<<<grid_for(recs + 1, T), T, 0, s>>>(in1 ? v1.get() : v0.get(), recs, ws.get(),
                                                                        ds.get());
  DCD_LAUNCH_CHECK();
  DCD_TRY(exclusive_scan<int64_t>(ws.get(), ws.get(), recs + 1, nullptr, wtmp.get(), s));
  DCD_TRY(exclusive_scan<int32_t>(ds.get(), ds.get(), recs + 1, nullptr, reinterpret_cast<int32_t*>(stmp.get()), s));
  ::dcd::count_launch(), long_pairs<<<grid_for(cdiv(recs, kLongChunk) * 32, T), T, 0, s>>>(
      pair_view(c, labels0, *out), list, first.get(), in1 ? k1.get() : k0.get(), ws.get(), ds.get(), recs,
      out->k->get());
  ::dcd::count_launch(), pair_net<<<grid_for(R + 1, T), T, 0, s>>>(out->pflag.get(), R, out->S.get());
  DCD_LAUNCH_CHECK();
  DCD_TRY_CUDA(cudaMemsetAsync(&d->n_long, 0, sizeof(int32_t), s));
  return merge_rows(c, labels0, static_start, out, nlab);
}

}  // namespace dcd
