// screen.cu -- Delta-screening (Algorithm 2, Sec. III-E) and the deletion
// rule, on G_t with the inherited labels C_{t-1}; then R_t.
//
// Per source i of the batch (its (source, sink) pairs are a contiguous range):
//   inserts: j* = argmax over the insert sinks j of S(i -> C(j)) (S = 0 when
//     C(j) = C(i); ties to the smaller C(j), then the smaller j -- the paper
//     fixes no tie rule); gain1 = S(i -> C(j*)), gain2 = S(j* -> C(i)); when
//     gain1 >= gain2 and gain1 > 0: mark i, j*, Gamma(i), flag C(j*).
//   deletes (not in the paper; reading): for each deleted pair (i, j) whose
//     edge was in G_{t-1}: mark i and j; if C(i) = C(j) also mark Gamma(i).
// R_t = marked vertices plus the members of flagged communities.  Screening
// changes no label.
//
// GPU schedule (same decisions, reordered work):
//   A  per source, binned by degree as the local move's vertices: sum row i by
//      community, S(i -> C(j)) of every insert pair (kept per pair), j*;
//      deletes.
//   B  per source: gain2.  An insert (i, j*) is also the insert (j*, i), so j*
//      is a source too and its phase A has S(j* -> C(i)) at the reverse pair:
//      a search of j*'s pairs replaces a second sum of row j*.  Marks i, j*,
//      flags C(j*), and lists the sources whose Gamma(i) is marked.
//   C  marks Gamma(i) and builds R_t, in the direction that reads less: the
//      rows of the listed sources (push), or, when they hold a fair part of
//      all entries, the rows of the vertices that are not in R_t yet, each only
//      up to its first listed neighbour (pull).
#include <type_traits>

#include "agg.cuh"
#include "bins.cuh"
#include "hub.cuh"
#include "prims.cuh"
#include "pull.cuh"
#include "rows.cuh"
#include "state.cuh"

namespace dcd {

namespace {

constexpr uint8_t kPairIns = 1, kPairDel = 2, kPairPresent = 4;

struct SV {
  const int64_t* rp;
  const int32_t* col;
  const int32_t* w;
  const int64_t* k;
  const int32_t* L;
  const int64_t* a;
  const uint64_t* pkey;
  const uint8_t* pflag;
  const int32_t* pair_ptr;
  int64_t m2;                   // 2m when the context holds one graph
  const int32_t* gid;           // graph of each vertex (several graphs)
  const GraphState* gs;
  __device__ __forceinline__ int64_t m2_of(int64_t v) const { return gid ? gs[gid[v]].m2 : m2; }
  uint8_t* mark;
  uint8_t* cflag;
  const int32_t* src;  // the sources, bin after bin
  // phase A's outputs per position in src: j* (-1: no insert) and whether an
  // intra-community delete marks Gamma(i); and per pair S(i -> C(j)), low
  // words, then (128-bit gains) high words
  int32_t* jstar;
  uint8_t* intra;
  long long* gain_lo;
  long long* gain_hi;
  // first-pass proposals (may be NULL): phase A sums a source's row by
  // community under C_{t-1} on G_t, the state the first local-move pass of
  // level 0 reads, so it also takes that pass's choice for the source (the
  // best neighbouring community, the S > 0 rule and the singleton guard) and
  // stores it in pre[source]; sources it does not sum keep -1
  const int32_t* size;
  int32_t* pre;
  const int32_t* nlab;  // labels in entry order (may be NULL)
};

// (S, D, j) order of the j* choice: larger gain, then smaller C(j), then smaller j.
template <typename ST>
__device__ __forceinline__ bool better3(ST s1, int32_t d1, int32_t j1, ST s2, int32_t d2, int32_t j2) {
  return s1 > s2 || (s1 == s2 && (d1 < d2 || (d1 == d2 && j1 < j2)));
}

// The j* choice over the SEG-lane segment of the calling lane (all lanes call).
template <int SEG, typename ST>
__device__ __forceinline__ void seg_argmax3(ST& S, int32_t& D, int32_t& J) {
#pragma unroll
  for (int o = SEG / 2; o > 0; o >>= 1) {
    const ST s2 = shfl_xor_st(S, o);
    const int32_t d2 = __shfl_xor_sync(0xffffffffu, D, o), j2 = __shfl_xor_sync(0xffffffffu, J, o);
    if (better3(s2, d2, j2, S, D, J)) {
      S = s2;
      D = d2;
      J = j2;
    }
  }
}

__device__ __forceinline__ void st_pair_gain(const SV& g, int64_t q, long long x) { g.gain_lo[q] = x; }
__device__ __forceinline__ void st_pair_gain(const SV& g, int64_t q, i128 x) {
  g.gain_lo[q] = (long long)(unsigned long long)x;
  g.gain_hi[q] = (long long)(unsigned long long)((unsigned __int128)x >> 64);
}
template <typename ST>
__device__ __forceinline__ ST ld_pair_gain(const SV& g, int64_t q);
template <>
__device__ __forceinline__ long long ld_pair_gain<long long>(const SV& g, int64_t q) {
  return g.gain_lo[q];
}
template <>
__device__ __forceinline__ i128 ld_pair_gain<i128>(const SV& g, int64_t q) {
  return (i128)(((unsigned __int128)(unsigned long long)g.gain_hi[q] << 64) | (unsigned long long)g.gain_lo[q]);
}

// Pairs [p0, p1) of source u by NT cooperating threads: marks the endpoints of
// deletes; returns bit 0: an intra-community delete, bit 1: an insert.
__device__ __forceinline__ unsigned scan_pairs(const SV& g, int32_t u, int32_t C, int64_t p0, int64_t p1, int tid,
                                               int NT) {
  unsigned f = 0;
  for (int64_t q = p0 + tid; q < p1; q += NT) {
    const uint8_t x = g.pflag[q];
    if (x & kPairIns) f |= 2;
    if ((x & kPairDel) && (x & kPairPresent)) {
      const int32_t j = (int32_t)(g.pkey[q] & 0xffffffffu);
      g.mark[j] = 1;
      g.mark[u] = 1;
      if (g.L[j] == C) f |= 1;
    }
  }
  return f;
}

// The insert pairs among [p0, p1) by NT cooperating threads: S(u -> C(j)) into
// the pair gains, and each thread's best (S, C(j), j).  lookup(D): the weight
// of row u into community D != C.
template <typename ST, typename F>
__device__ __forceinline__ void best_sink(const SV& g, int32_t C, int64_t p0, int64_t p1, int tid, int NT, int64_t m2,
                                          int64_t ku, int64_t eC, int64_t aC, F lookup, ST& S, int32_t& D, int32_t& J) {
  S = gain_lowest<ST>();
  D = J = INT_MAX;
  for (int64_t q = p0 + tid; q < p1; q += NT) {
    if (!(g.pflag[q] & kPairIns)) continue;
    const int32_t j = (int32_t)(g.pkey[q] & 0xffffffffu);
    const int32_t Dj = g.L[j];
    const ST x = (Dj == C) ? ST(0) : gain<ST>(m2, ku, lookup(Dj), eC, g.a[Dj], aC);
    st_pair_gain(g, q, x);
    if (better3(x, Dj, j, S, D, J)) {
      S = x;
      D = Dj;
      J = j;
    }
  }
}

// The same for a source that gains nowhere (stays, agg.cuh): 0 stands for its
// gains.  Phase B compares a pair's reverse gain with one above 0, for which all
// values up to 0 are alike.
template <typename ST>
__device__ __forceinline__ void no_sink(const SV& g, int64_t p0, int64_t p1, int tid, int NT) {
  for (int64_t q = p0 + tid; q < p1; q += NT)
    if (g.pflag[q] & kPairIns) st_pair_gain(g, q, ST(0));
}

// ---- phase A ----
//
// The kernels follow the local move's for the same row lengths (louvain.cu says
// why each is built as it is); what they add is a pass over the source's
// pairs before the row (deletes; a source without inserts needs no row) and
// one over its inserts after.  A source's kernel is chosen by its row or its
// pairs, whichever is longer: a vertex that loses 60,000 edges has no row left, and
// one lane walked over its pairs for 9 ms (0.15 so, 0.08 when as many are spread).
// Bound like them by the latency of dependent loads; on the LFR 2M step (2 M
// sources, 74 M entries, 12.4 M pairs) the bins
// run side by side in about 0.6 ms.  With four classes of sources (a warp with
// lane compares to 32 entries, a warp table to 256, a CTA with an 8192-slot
// table to 4096: two CTAs an SM for a row of 300) it took 1.9 ms, on R-MAT 22
// 2.8 ms for the last class alone (now 0.8).

// Rows of at most 32 entries: S lanes read a row (32 / S rows at a time), then
// a lane chooses for a source, from a list of the row's foreign entries.
template <typename ST, int S, int Q, int CAP>
__global__ void __launch_bounds__(256) scr_vert(SV g, int64_t off, int64_t cnt, int per) {
  using VT = typename TblVal<ST>::type;
  using Ent = ListEnt<VT>;
  constexpr int P = 32 / S, ROW = S * Q;
  constexpr bool kFree = ROW > CAP;  // rows may outgrow a lane's list
  static_assert(!kFree || ROW <= 4 * S, "list_best takes at most four entries a lane");
  extern __shared__ __align__(16) unsigned char smem[];
  const int lane = lane_id(), sub = lane / S, sl = lane % S, wib = threadIdx.x >> 5;
  const unsigned smask = ((1u << S) - 1u) << (sub * S);
  Ent* const ent = reinterpret_cast<Ent*>(smem + (size_t)wib * vert_bytes<S, Q, CAP, VT>());
  Ent* const row = ent + CAP * 32 + sub * (ROW + 2);
  const int64_t nw = ((int64_t)gridDim.x * blockDim.x) >> 5;
  for (int64_t wb = ((blockIdx.x * (int64_t)blockDim.x + threadIdx.x) >> 5) * per; wb < cnt; wb += nw * per) {
    const int nb = cnt - wb < per ? (int)(cnt - wb) : per;
    const bool own = lane < nb;
    int32_t u_l = 0, C_l = 0, p0 = 0, p1 = 0, J_l = -1, D_l = INT_MAX;
    int64_t b_l = 0, k_l = 0, aC_l = 0;
    int d_l = 0, n_l = 0;
    unsigned f_l = 0;
    if (own) {
      u_l = g.src[off + wb + lane];
      C_l = g.L[u_l];
      p0 = g.pair_ptr[u_l];
      p1 = g.pair_ptr[u_l + 1];
      b_l = g.rp[u_l];
      d_l = (int)(g.rp[u_l + 1] - b_l);
      k_l = g.k[u_l];
      aC_l = g.a[C_l];
      f_l = scan_pairs(g, u_l, C_l, p0, p1, 0, 1);
      if (!(f_l & 2)) d_l = 0;
    }
    const int steps = __any_sync(0xffffffffu, d_l > 0) ? (nb + P - 1) / P : 0;
    for (int t = 0; t < steps; t++) {
      const int at_l = t * P + sub;
      const int d = __shfl_sync(0xffffffffu, d_l, at_l);
      const int64_t b = __shfl_sync(0xffffffffu, b_l, at_l);
      const int32_t C = __shfl_sync(0xffffffffu, C_l, at_l);
      int32_t lab[Q], wt[Q];
#pragma unroll
      for (int q = 0; q < Q; q++) {
        const int e = q * S + sl;
        lab[q] = -1;
        wt[q] = 0;
        if (e < d) {
          lab[q] = ld_stream((g.nlab ? g.nlab : g.col) + b + e);
          wt[q] = ld_stream(g.w + b + e);
        }
      }
#pragma unroll
      for (int q = 0; q < Q; q++) lab[q] = lab[q] < 0 ? C : g.nlab ? lab[q] : g.L[lab[q]];
      int n = 0;
      int at[Q];
#pragma unroll
      for (int q = 0; q < Q; q++) {
        const unsigned bal = __ballot_sync(0xffffffffu, lab[q] != C) & smask;
        at[q] = n + __popc(bal & lanemask_lt());
        n += __popc(bal);
      }
      if (!kFree || !__any_sync(0xffffffffu, n > CAP)) {
#pragma unroll
        for (int q = 0; q < Q; q++)
          if (lab[q] != C) {
            Ent x{};
            x.lab = lab[q];
            x.w = (VT)wt[q];
            ent[at[q] * 32 + at_l] = x;
          }
        const int pick = __shfl_sync(0xffffffffu, n, (lane & (P - 1)) * S);
        if (lane / P == t) n_l = pick;
      } else if constexpr (kFree) {
        // a list is too long for its lane: the segments choose together
        VT sum = 0;
#pragma unroll
        for (int q = 0; q < Q; q++)
          if (lab[q] != C) {
            Ent x{};
            x.lab = lab[q];
            x.w = (VT)wt[q];
            row[at[q]] = x;
            sum += (VT)wt[q];
          }
        const int nmax = (int)__reduce_max_sync(0xffffffffu, (unsigned)n);
        for (int j = n + sl; j < nmax + (nmax & 1); j += S) row[j].lab = -2;
        __syncwarp();
        const int64_t ku = __shfl_sync(0xffffffffu, k_l, at_l), eC = ku - seg_total<S>(sum);
        const int64_t aC = __shfl_sync(0xffffffffu, aC_l, at_l);
        const int32_t u = __shfl_sync(0xffffffffu, u_l, at_l);
        const int64_t m2 = g.m2_of(u);
        if (g.pre) {
          ST Sb = gain_lowest<ST>();
          int32_t D = INT_MAX;
          int64_t eD;
          list_best<SV, ST, S, (ROW + S - 1) / S, VT>(g, row, n, nmax, ku, eC, aC, m2, sl, Sb, D, eD);
          const int32_t pick = __shfl_sync(0xffffffffu, Sb > 0 ? D : INT_MAX, (lane & (P - 1)) * S);
          if (lane / P == t) D_l = pick;
        }
        const int32_t q0 = __shfl_sync(0xffffffffu, p0, at_l), q1 = __shfl_sync(0xffffffffu, p1, at_l);
        ST Sj;
        int32_t Dj, Jj;
        best_sink<ST>(g, C, q0, d > 0 ? q1 : q0, sl, S, m2, ku, eC, aC,
                      [&](int32_t D) {
                        VT e = 0;
                        for (int j = 0; j < n; j++)
                          if (row[j].lab == D) e += row[j].w;
                        return (int64_t)e;
                      },
                      Sj, Dj, Jj);
        seg_argmax3<S>(Sj, Dj, Jj);
        const int32_t jj = __shfl_sync(0xffffffffu, Sj > 0 ? Jj : -1, (lane & (P - 1)) * S);
        if (lane / P == t) {
          J_l = jj;
          n_l = -1;
        }
        __syncwarp();
      }
    }
    __syncwarp();
    if (own && n_l >= 0 && (f_l & 2)) {
      Ent* const my = ent + lane;
      VT tot = 0;
      for (int j = 0; j < n_l; j++) tot += my[j * 32].w;
      const int64_t eC = k_l - (int64_t)tot, m2 = g.m2_of(u_l);
      const bool open = !stays<ST>(m2, k_l, eC, aC_l);
      if (!open) n_l = 0;
      // the lane's list folded by community, in place
      int nd = 0;
      for (int j = 0; j < n_l; j++) {
        const Ent x = my[j * 32];
        int i = 0;
        while (i < nd && my[i * 32].lab != x.lab) i++;
        if (i < nd) my[i * 32].w += x.w;
        else my[nd++ * 32] = x;
      }
      if (g.pre) {
        ST Sb = gain_lowest<ST>();
        int32_t D = INT_MAX;
        for (int i = 0; i < nd; i++) {
          const Ent x = my[i * 32];
          const ST y = gain<ST>(m2, k_l, (int64_t)x.w, eC, g.a[x.lab], aC_l);
          if (better(y, x.lab, Sb, D)) {
            Sb = y;
            D = x.lab;
          }
        }
        if (Sb > 0) D_l = D;
      }
      if (open) {
        ST Sj;
        int32_t Dj, Jj;
        best_sink<ST>(g, C_l, p0, p1, 0, 1, m2, k_l, eC, aC_l,
                      [&](int32_t D) {
                        for (int i = 0; i < nd; i++)
                          if (my[i * 32].lab == D) return (int64_t)my[i * 32].w;
                        return (int64_t)0;
                      },
                      Sj, Dj, Jj);
        if (Sj > 0) J_l = Jj;
      } else {
        no_sink<ST>(g, p0, p1, 0, 1);
      }
    }
    if (own) {
      g.jstar[off + wb + lane] = J_l;
      g.intra[off + wb + lane] = (uint8_t)(f_l & 1);
      if (g.pre && (f_l & 2)) g.pre[u_l] = move_proposal<long long>(1, D_l, C_l, g.size);
    }
    __syncwarp();
  }
}

// Rows of 33 to 256 entries: S lanes a source, the row's sums in the segment's
// table in shared memory.
template <typename ST, int S, int Q>
__global__ void __launch_bounds__(256) scr_seg(SV g, int64_t off, int64_t cnt) {
  static_assert(S == 16 || S == 32, "segments of 16 or 32 lanes");
  using VT = typename TblVal<ST>::type;
  constexpr int P = 32 / S, ROW = S * Q, CAP = seg_cap(ROW);
  constexpr uint32_t mask = CAP - 1;
  extern __shared__ __align__(16) unsigned char smem[];
  const int lane = lane_id(), sub = lane / S, sl = lane % S, wib = threadIdx.x >> 5;
  const unsigned smask = S == 32 ? 0xffffffffu : (((1u << S) - 1u) << (sub * S));
  unsigned char* base = smem + ((size_t)wib * P + sub) * row_tbl_bytes<ROW, VT>();
  int32_t* keys = reinterpret_cast<int32_t*>(base);
  VT* vals = reinterpret_cast<VT*>(base + (size_t)CAP * 4);
  uint16_t* slots = reinterpret_cast<uint16_t*>(base + (size_t)CAP * (4 + sizeof(VT)));
  for (int s = sl; s < CAP; s += S) {
    keys[s] = -1;
    vals[s] = 0;
  }
  __syncwarp();
  const int64_t nw = ((int64_t)gridDim.x * blockDim.x) >> 5;
  for (int64_t wb = ((blockIdx.x * (int64_t)blockDim.x + threadIdx.x) >> 5) * P; wb < cnt; wb += nw * P) {
    const int64_t i = wb + sub;
    const bool has = i < cnt;
    const int32_t u = has ? g.src[off + i] : 0;
    const int32_t C = g.L[u];
    const int64_t p0 = has ? g.pair_ptr[u] : 0, p1 = has ? g.pair_ptr[u + 1] : 0;
    const int64_t b = g.rp[u];
    const unsigned mine = scan_pairs(g, u, C, p0, p1, sl, S);
    const bool intra = (__ballot_sync(0xffffffffu, mine & 1) & smask) != 0;
    const bool ins = (__ballot_sync(0xffffffffu, mine & 2) & smask) != 0;
    const int d = ins ? (int)(g.rp[u + 1] - b) : 0;
    const int dmax = S == 32 ? d : (int)__reduce_max_sync(0xffffffffu, (unsigned)d);
    int32_t J = -1;
    if (dmax > 0) {
      int32_t lab[Q], wt[Q];
#pragma unroll
      for (int q = 0; q < Q; q++) {
        const int e = q * S + sl;
        lab[q] = -1;
        wt[q] = 0;
        if (e < d) {
          lab[q] = ld_stream((g.nlab ? g.nlab : g.col) + b + e);
          wt[q] = ld_stream(g.w + b + e);
        }
      }
      if (!g.nlab) {
#pragma unroll
        for (int q = 0; q < Q; q++) lab[q] = lab[q] >= 0 ? g.L[lab[q]] : -1;
      }
      VT eCl = 0;
      int nd = 0;
#pragma unroll
      for (int q = 0; q < Q; q++) eCl += lab[q] == C ? (VT)wt[q] : VT(0);
      const int64_t eC = seg_total<S>(eCl);
      const int64_t ku = g.k[u], aC = g.a[C], m2 = g.m2_of(u);
      const bool open = !stays<ST>(m2, ku, eC, aC);
#pragma unroll
      for (int q = 0; q < Q; q++) {
        if (q * S < dmax && __any_sync(0xffffffffu, open)) {
          bool claimed = false;
          uint32_t s = 0;
          if (lab[q] >= 0 && lab[q] != C && open) {
            s = probe_claim(keys, mask, lab[q], claimed);
            atomicAdd(&vals[s], (VT)wt[q]);
          }
          const unsigned bal = __ballot_sync(0xffffffffu, claimed) & smask;
          if (claimed) slots[nd + __popc(bal & lanemask_lt())] = (uint16_t)s;
          nd += __popc(bal);
        }
      }
      __syncwarp();
      if (g.pre) {  // the local move's choice over the table's communities
        ST Sb = gain_lowest<ST>();
        int32_t D = INT_MAX;
        for (int j = sl; j < nd; j += S) {
          const uint32_t s = slots[j];
          const int32_t key = keys[s];
          const ST x = gain<ST>(m2, ku, (int64_t)vals[s], eC, g.a[key], aC);
          if (better(x, key, Sb, D)) {
            Sb = x;
            D = key;
          }
        }
        seg_argmax<S>(Sb, D);
        if (sl == 0 && ins) g.pre[u] = move_proposal(Sb, D, C, g.size);
      }
      ST Sj;
      int32_t Dj, Jj;
      if (!open) no_sink<ST>(g, p0, p1, sl, S);
      best_sink<ST>(g, C, p0, ins && open ? p1 : p0, sl, S, m2, ku, eC, aC,
                    [&](int32_t D) { return tbl_get(keys, vals, mask, D); }, Sj, Dj, Jj);
      seg_argmax3<S>(Sj, Dj, Jj);
      if (Sj > 0) J = Jj;
      __syncwarp();
      for (int j = sl; j < nd; j += S) {
        const uint32_t s = slots[j];
        keys[s] = -1;
        vals[s] = 0;
      }
      __syncwarp();
    }
    if (sl == 0 && has) {
      g.jstar[off + i] = J;
      g.intra[off + i] = intra ? 1 : 0;
    }
  }
}

// Rows of 257 to 4096 entries: a CTA of T threads a source, Q entries a thread.
template <typename ST, int T, int Q>
__global__ void __launch_bounds__(T) scr_cta(SV g, int64_t off, int64_t cnt) {
  using VT = typename TblVal<ST>::type;
  constexpr int NW = T / 32, ROW = T * Q, CAP = seg_cap(ROW);
  constexpr uint32_t mask = CAP - 1;
  extern __shared__ __align__(16) unsigned char smem[];
  __shared__ ST redS[NW], preS[NW];
  __shared__ int32_t redD[NW], redJ[NW], preD[NW];
  __shared__ VT redC[NW];
  __shared__ int32_t s_nd;
  int32_t* keys = reinterpret_cast<int32_t*>(smem);
  VT* vals = reinterpret_cast<VT*>(smem + (size_t)CAP * 4);
  uint16_t* slots = reinterpret_cast<uint16_t*>(smem + (size_t)CAP * (4 + sizeof(VT)));
  const int tid = threadIdx.x, lane = lane_id(), wid = tid >> 5;
  for (int s = tid; s < CAP; s += T) {
    keys[s] = -1;
    vals[s] = 0;
  }
  if (tid == 0) s_nd = 0;
  __syncthreads();
  for (int64_t i = blockIdx.x; i < cnt; i += gridDim.x) {
    const int32_t u = g.src[off + i];
    const int32_t C = g.L[u];
    const int64_t p0 = g.pair_ptr[u], p1 = g.pair_ptr[u + 1];
    const int64_t b = g.rp[u];
    const unsigned mine = scan_pairs(g, u, C, p0, p1, tid, T);
    const bool intra = __syncthreads_or(mine & 1) != 0, ins = __syncthreads_or(mine & 2) != 0;
    if (!ins) {
      if (tid == 0) {
        g.jstar[off + i] = -1;
        g.intra[off + i] = intra ? 1 : 0;
      }
      continue;
    }
    const int d = (int)(g.rp[u + 1] - b);
    int32_t lab[Q], wt[Q];
#pragma unroll
    for (int q = 0; q < Q; q++) {
      const int e = q * T + tid;
      lab[q] = -1;
      wt[q] = 0;
      if (e < d) {
        lab[q] = ld_stream((g.nlab ? g.nlab : g.col) + b + e);
        wt[q] = ld_stream(g.w + b + e);
      }
    }
    if (!g.nlab) {
#pragma unroll
      for (int q = 0; q < Q; q++) lab[q] = lab[q] >= 0 ? g.L[lab[q]] : -1;
    }
    VT eCl = 0;
#pragma unroll
    for (int q = 0; q < Q; q++) eCl += lab[q] == C ? (VT)wt[q] : VT(0);
    const int64_t ew = seg_total<32>(eCl);
    if (lane == 0) redC[wid] = (VT)ew;
    const int64_t ku = g.k[u], aC = g.a[C], m2 = g.m2_of(u);
    __syncthreads();
    int64_t eC = 0;
#pragma unroll
    for (int x = 0; x < NW; x++) eC += (int64_t)redC[x];
    if (stays<ST>(m2, ku, eC, aC)) {  // uniform
      no_sink<ST>(g, p0, p1, tid, T);
      if (tid == 0) {
        g.jstar[off + i] = -1;
        g.intra[off + i] = intra ? 1 : 0;
        if (g.pre) g.pre[u] = C;
      }
      __syncthreads();
      continue;
    }
#pragma unroll
    for (int q = 0; q < Q; q++) {
      if (q * T < d) {
        bool claimed = false;
        uint32_t s = 0;
        if (lab[q] >= 0 && lab[q] != C) {
          s = probe_claim(keys, mask, lab[q], claimed);
          atomicAdd(&vals[s], (VT)wt[q]);
        }
        const unsigned bal = __ballot_sync(0xffffffffu, claimed);
        int at = 0;
        if (lane == 0 && bal) at = atomicAdd(&s_nd, __popc(bal));
        at = __shfl_sync(0xffffffffu, at, 0);
        if (claimed) slots[at + __popc(bal & lanemask_lt())] = (uint16_t)s;
      }
    }
    __syncthreads();
    const int nd = s_nd;
    if (g.pre) {  // the local move's choice over the table's communities
      ST Sb = gain_lowest<ST>();
      int32_t D = INT_MAX;
      for (int j = tid; j < nd; j += T) {
        const uint32_t s = slots[j];
        const int32_t key = keys[s];
        const ST x = gain<ST>(m2, ku, (int64_t)vals[s], eC, g.a[key], aC);
        if (better(x, key, Sb, D)) {
          Sb = x;
          D = key;
        }
      }
      warp_argmax(Sb, D);
      if (lane == 0) {
        preS[wid] = Sb;
        preD[wid] = D;
      }
    }
    ST Sj;
    int32_t Dj, Jj;
    best_sink<ST>(g, C, p0, p1, tid, T, m2, ku, eC, aC, [&](int32_t D) { return tbl_get(keys, vals, mask, D); }, Sj, Dj,
                  Jj);
    seg_argmax3<32>(Sj, Dj, Jj);
    if (lane == 0) {
      redS[wid] = Sj;
      redD[wid] = Dj;
      redJ[wid] = Jj;
    }
    __syncthreads();
    if (wid == 0) {
      Sj = lane < NW ? redS[lane] : gain_lowest<ST>();
      Dj = lane < NW ? redD[lane] : INT_MAX;
      Jj = lane < NW ? redJ[lane] : INT_MAX;
      seg_argmax3<32>(Sj, Dj, Jj);
      if (lane == 0) {
        g.jstar[off + i] = Sj > 0 ? Jj : -1;
        g.intra[off + i] = intra ? 1 : 0;
      }
      if (g.pre) {
        ST Sb = lane < NW ? preS[lane] : gain_lowest<ST>();
        int32_t D = lane < NW ? preD[lane] : INT_MAX;
        warp_argmax(Sb, D);
        if (lane == 0) g.pre[u] = move_proposal(Sb, D, C, g.size);
      }
    }
    for (int j = tid; j < nd; j += T) {
      const uint32_t s = slots[j];
      keys[s] = -1;
      vals[s] = 0;
    }
    if (tid == 0) s_nd = 0;
    __syncthreads();
  }
}

// Hub sources (rows above 4096 entries): the rows were summed into per-hub
// global tables by hub_agg (many CTAs per row); one CTA per source then
// reads its deletes and evaluates its insert sinks by table lookups.
template <typename ST, int T>
__global__ void __launch_bounds__(T) scr_hub(SV g, int64_t off, int64_t cnt, HubTables t) {
  constexpr int NW = T / 32;
  __shared__ ST redS[NW];
  __shared__ int32_t redD[NW], redJ[NW];
  const int tid = threadIdx.x, lane = lane_id(), wid = tid >> 5;
  for (int64_t h = blockIdx.x; h < cnt; h += gridDim.x) {
    const int32_t u = g.src[off + h];
    const int32_t C = g.L[u];
    const int64_t p0 = g.pair_ptr[u], p1 = g.pair_ptr[u + 1];
    const unsigned mine = scan_pairs(g, u, C, p0, p1, tid, T);
    const bool intra = __syncthreads_or(mine & 1) != 0;
    const uint32_t mask = (uint32_t)(t.toff[h + 1] - t.toff[h]) - 1;
    const int32_t* keys = t.keys + t.toff[h];
    const unsigned long long* vals = t.vals + t.toff[h];
    const int64_t eC = tbl_get(keys, vals, mask, C);
    ST Sj;
    int32_t Dj, Jj;
    best_sink<ST>(g, C, p0, p1, tid, T, g.m2_of(u), g.k[u], eC, g.a[C],
                  [&](int32_t D) { return tbl_get(keys, vals, mask, D); }, Sj, Dj, Jj);
    seg_argmax3<32>(Sj, Dj, Jj);
    if (lane == 0) {
      redS[wid] = Sj;
      redD[wid] = Dj;
      redJ[wid] = Jj;
    }
    __syncthreads();
    if (wid == 0) {
      Sj = lane < NW ? redS[lane] : gain_lowest<ST>();
      Dj = lane < NW ? redD[lane] : INT_MAX;
      Jj = lane < NW ? redJ[lane] : INT_MAX;
      seg_argmax3<32>(Sj, Dj, Jj);
      if (lane == 0) {
        g.jstar[off + h] = Sj > 0 ? Jj : -1;
        g.intra[off + h] = intra ? 1 : 0;
      }
    }
    __syncthreads();
  }
}

// ---- phase B ----

// The pair (u, v) (the last of equal ones, which carries the gain); it exists.
__device__ __forceinline__ int64_t find_pair(const SV& g, int32_t u, int32_t v) {
  int64_t lo = g.pair_ptr[u], hi = g.pair_ptr[u + 1];  // first pair with a larger sink
  while (lo < hi) {
    const int64_t mid = (lo + hi) >> 1;
    if ((int32_t)(g.pkey[mid] & 0xffffffffu) <= v) lo = mid + 1; else hi = mid;
  }
  return lo - 1;
}

constexpr int kGammaChunk = 256;  // entries of a row a work item marks

// A source per lane: gain1 >= gain2 decides; jstar holds only sinks of
// gain1 > 0.  82 us for 2 M sources, where sorting the sources by j* and
// summing row j* again took 0.6 ms (R-MAT 22: 1.6 ms), 25 launches and two
// host round trips.  The sources whose neighbourhood is marked set listed[] and
// become work items (u << 32 | chunk).
constexpr int kDecideThreads = 256;
template <typename ST>
__global__ void __launch_bounds__(kDecideThreads) scr_decide(SV g, int64_t nsrc, uint8_t* __restrict__ listed,
                                                  int64_t* __restrict__ items, int32_t* __restrict__ item_cnt,
                                                  unsigned long long* __restrict__ gamma_deg) {
  __shared__ int32_t s_at;
  const int lane = lane_id();
  const int64_t stride = (int64_t)gridDim.x * kDecideThreads;
  unsigned long long deg = 0;
  for (int64_t base = blockIdx.x * (int64_t)kDecideThreads; base < nsrc; base += stride) {
    const int64_t i = base + threadIdx.x;
    int nch = 0;
    int32_t u = 0;
    if (i < nsrc) {
      u = g.src[i];
      const int32_t j = g.jstar[i];
      bool gamma = g.intra[i] != 0;
      if (j >= 0) {
        const ST g1 = ld_pair_gain<ST>(g, find_pair(g, u, j)), g2 = ld_pair_gain<ST>(g, find_pair(g, j, u));
        if (g1 >= g2) {
          gamma = true;
          g.mark[j] = 1;
          g.cflag[g.L[j]] = 1;
        }
      }
      if (gamma) {
        g.mark[u] = 1;
        listed[u] = 1;
        const int64_t d = g.rp[u + 1] - g.rp[u];
        deg += (unsigned long long)d;
        nch = (int)((d + kGammaChunk - 1) / kGammaChunk);
      }
    }
    if (!__syncthreads_or(nch)) continue;
    int total;
    const int excl = block_excl_scan<int, kDecideThreads>(nch, &total);
    if (threadIdx.x == 0) s_at = atomicAdd(item_cnt, total);  // once a CTA and step: all on one word
    __syncthreads();
    const int32_t at = s_at + excl;
    for (int x = 0; x < nch; x++) items[at + x] = (int64_t)u << 32 | (uint32_t)x;
    __syncthreads();
  }
  deg = warp_sum(deg);
  if (lane == 0 && deg) atomicAdd(gamma_deg, deg);
}

// ---- phase C ----
//
// Pull reads a vertex's row up to its first listed neighbour.  With the listed
// sources holding a share s of all entries it expects 1 / s entries a vertex
// (an entry's neighbour is listed with probability about s), so from a quarter
// on it reads a few entries of the vertices that are left, where push stores
// into every neighbour of every listed source: on the LFR 2M step with 74 M
// entries, nearly all of them in listed rows, push took 605-640 us.
__device__ __forceinline__ bool pulls(unsigned long long gamma_deg, int64_t nnz) {
  return 4 * (int64_t)gamma_deg >= nnz;
}

__global__ void __launch_bounds__(256) scr_push(SV g, int64_t nnz, const int64_t* __restrict__ items,
                                                const int32_t* __restrict__ item_cnt,
                                                const unsigned long long* __restrict__ gamma_deg) {
  if (pulls(*gamma_deg, nnz)) return;
  constexpr int U = kGammaChunk / 32;
  const int64_t nw = ((int64_t)gridDim.x * blockDim.x) >> 5;
  const int64_t cnt = *item_cnt;
  for (int64_t i = (blockIdx.x * (int64_t)blockDim.x + threadIdx.x) >> 5; i < cnt; i += nw) {
    const int64_t it = items[i];
    const int32_t u = (int32_t)(it >> 32);
    const int64_t b = g.rp[u] + (int64_t)(uint32_t)it * kGammaChunk;
    const int64_t rest = g.rp[u + 1] - b;
    const int len = rest < kGammaChunk ? (int)rest : kGammaChunk;
    int32_t y[U];
#pragma unroll
    for (int q = 0; q < U; q++) y[q] = q * 32 + (int)lane_id() < len ? ld_stream(g.col + b + q * 32 + lane_id()) : -1;
#pragma unroll
    for (int q = 0; q < U; q++)
      if (y[q] >= 0) g.mark[y[q]] = 1;
  }
}

// R_t.  Pull: the vertices of a warp that are not in R_t yet are taken 8 lanes
// each, up to kPullFirst entries; who is still undecided is left to pull_rest.
struct Listed {
  const uint8_t* listed;
  __device__ __forceinline__ bool operator()(int32_t x) const { return listed[x] != 0; }
};
__global__ void __launch_bounds__(256) build_rset(int64_t n, int64_t nnz, const int64_t* __restrict__ rp,
                                                  const int32_t* __restrict__ col, const uint8_t* __restrict__ mark,
                                                  const uint8_t* __restrict__ cflag, const uint8_t* __restrict__ listed,
                                                  const unsigned long long* __restrict__ gamma_deg,
                                                  const int32_t* __restrict__ L, uint8_t* __restrict__ r,
                                                  PullRest rest, unsigned long long* __restrict__ count) {
  const bool pull = listed && pulls(*gamma_deg, nnz);
  unsigned long long c = 0;
  const int lane = lane_id(), grp = lane >> 3, gl = lane & 7;
  const int64_t stride = (int64_t)gridDim.x * blockDim.x;
  for (int64_t base = (blockIdx.x * (int64_t)blockDim.x) + (threadIdx.x & ~31); base < n; base += stride) {
    const int64_t v = base + lane;
    uint8_t x = v < n ? (uint8_t)(mark[v] | cflag[L[v]]) : (uint8_t)1;
    if (pull) {
      int64_t b = 0;
      int64_t d = 0;
      if (!x) {
        b = rp[v];
        d = rp[v + 1] - b;
      }
      unsigned todo = __ballot_sync(0xffffffffu, !x && d > 0);
      while (todo) {
        // the next four of them, a group of 8 lanes each
        unsigned left = todo;
        int who = -1;
#pragma unroll
        for (int k = 0; k < 4; k++) {
          const int f = left ? __ffs(left) - 1 : -1;
          if (k == grp) who = f;
          if (f >= 0) left &= left - 1;
        }
        const int64_t bb = __shfl_sync(0xffffffffu, b, who < 0 ? 0 : who);
        const int64_t dw = __shfl_sync(0xffffffffu, d, who < 0 ? 0 : who);
        const int lim = who < 0 ? 0 : (int)(dw < kPullFirst ? dw : kPullFirst);
        bool hit = false;
        for (int e0 = 0; e0 < kPullFirst; e0 += 8) {
          const bool go = !hit && e0 < lim;
          if (!__any_sync(0xffffffffu, go)) break;
          const bool h = go && e0 + gl < lim && listed[col[bb + e0 + gl]];
          hit |= (__ballot_sync(0xffffffffu, h) >> (grp * 8) & 0xffu) != 0;
        }
        const unsigned hits = __ballot_sync(0xffffffffu, hit && gl == 0);
#pragma unroll
        for (int k = 0; k < 4; k++) {
          const int f = __shfl_sync(0xffffffffu, who, k * 8);
          if (f == lane && (hits >> (k * 8) & 1u)) x = 1;
        }
        todo = left;
      }
      pull_defer(rest, !x && d > kPullFirst, v, d);
    }
    if (v < n) {
      r[v] = x;
      c += x;
    }
  }
  c = warp_sum(c);
  if (lane == 0 && c) atomicAdd(count, c);
}

// ---- host side ----

template <typename ST, int S, int Q, int CAP>
int launch_scr_vert(cudaStream_t s, const SV& sv, int64_t off, int64_t cnt) {
  constexpr int T = 256, P = 32 / S;
  constexpr size_t smem = 8 * vert_bytes<S, Q, CAP, typename TblVal<ST>::type>();
  DCD_TRY_CUDA(cudaFuncSetAttribute(scr_vert<ST, S, Q, CAP>, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)smem));
  const int64_t warps = (int64_t)wave_grid(scr_vert<ST, S, Q, CAP>, INT64_MAX / 2, T, smem) * (T / 32);
  int per = 32;
  while (per > P && cdiv(cnt, per) < 2 * warps) per /= 2;
  count_launch(), scr_vert<ST, S, Q, CAP><<<wave_grid(scr_vert<ST, S, Q, CAP>, cdiv(cnt, per) * 32, T, smem), T, smem,
                                            s>>>(sv, off, cnt, per);
  return DCD_OK;
}

template <typename ST, int S, int Q>
int launch_scr_seg(cudaStream_t s, const SV& sv, int64_t off, int64_t cnt) {
  constexpr int T = 256, P = 32 / S;
  constexpr size_t smem = (size_t)8 * P * row_tbl_bytes<S * Q, typename TblVal<ST>::type>();
  DCD_TRY_CUDA(cudaFuncSetAttribute(scr_seg<ST, S, Q>, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)smem));
  count_launch(), scr_seg<ST, S, Q><<<wave_grid(scr_seg<ST, S, Q>, cdiv(cnt, P) * 32, T, smem), T, smem, s>>>(sv, off,
                                                                                                            cnt);
  return DCD_OK;
}

template <typename ST, int T, int Q>
int launch_scr_cta(cudaStream_t s, const SV& sv, int64_t off, int64_t cnt) {
  constexpr size_t smem = row_tbl_bytes<T * Q, typename TblVal<ST>::type>();
  DCD_TRY_CUDA(cudaFuncSetAttribute(scr_cta<ST, T, Q>, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)smem));
  count_launch(), scr_cta<ST, T, Q><<<wave_grid(scr_cta<ST, T, Q>, cnt * T, T, smem), T, smem, s>>>(sv, off, cnt);
  return DCD_OK;
}

template <typename ST>
int screen_rows(dcd_ctx* c, const SV& sv, const Csr<int32_t>& g, const SourceBins& sb) {
  const BinPlan& plan = sb.plan;
  HubBufs hb;
  const int64_t hubs = sb.cnt[plan.nb - 1], hub_off = sb.total - hubs;
  if (hubs) DCD_TRY(hub_setup(c, sv.src + hub_off, hubs, g.rp, &hb));
  // the bins write disjoint slices of the per-source outputs: side by side
  SideBySide par(c, sb.total);
  DCD_TRY(par.fork());
  int64_t off = 0;
  for (int x = 0; x < plan.nb; x++) {
    const int64_t cnt = sb.cnt[x];
    if (!cnt) continue;
    cudaStream_t s;
    DCD_TRY(par.on(x, &s));
    switch (plan.var[x]) {
      case kLmSeg16: DCD_TRY((launch_scr_vert<ST, 4, 4, 16>(s, sv, off, cnt))); break;
      case kLmSeg32: DCD_TRY((launch_scr_vert<ST, 8, 4, kCap32>(s, sv, off, cnt))); break;
      case kLmSeg64: DCD_TRY((launch_scr_seg<ST, 16, 4>(s, sv, off, cnt))); break;
      case kLmWarp128: DCD_TRY((launch_scr_seg<ST, 32, 4>(s, sv, off, cnt))); break;
      case kLmWarp256: DCD_TRY((launch_scr_seg<ST, 32, 8>(s, sv, off, cnt))); break;
      case kLmCta512: DCD_TRY((launch_scr_cta<ST, 128, 4>(s, sv, off, cnt))); break;
      case kLmCta1k: DCD_TRY((launch_scr_cta<ST, 256, 4>(s, sv, off, cnt))); break;
      case kLmCta2k: DCD_TRY((launch_scr_cta<ST, 512, 4>(s, sv, off, cnt))); break;
      case kLmCta4k: DCD_TRY((launch_scr_cta<ST, 512, 8>(s, sv, off, cnt))); break;
      default:
        count_launch(), hub_agg<int32_t, ST><<<hub_grid(c, hb), kHubThreads, 0, s>>>(sv, hb.t);
        count_launch(), scr_hub<ST, 512><<<(unsigned)(cnt < 4 * c->sms ? cnt : 4 * c->sms), 512, 0, s>>>(sv, off, cnt,
                                                                                                        hb.t);
        break;
    }
    DCD_LAUNCH_CHECK();
    off += cnt;
  }
  return par.join();
}

}  // namespace

int source_counts(dcd_ctx* c, const int64_t* rp, const int32_t* pair_ptr, SourceBins* sb) {
  cudaStream_t s = c->stream;
  DevScalars* d = c->dsc.get();
  sb->plan = default_bin_plan();
  DCD_TRY_CUDA(cudaMemsetAsync(&d->bcnt[0], 0, 3 * kMaxBins * sizeof(int64_t), s));
  DCD_TRY_CUDA(cudaMemsetAsync(&d->act_deg, 0, 2 * sizeof(int64_t), s));
  count_launch(), bin_count<<<grid_for(c->n, 256), 256, 0, s>>>(rp, c->n, WantSource{pair_ptr}, d, sb->plan, nullptr);
  DCD_LAUNCH_CHECK();
  return DCD_OK;
}

int screen_batch(dcd_ctx* c, const Csr<int32_t>& g, const int32_t* labels0, const int64_t* k, const int64_t* a,
                 const MergeOut& mo, const SourceBins& sb, const int32_t* nlab, uint8_t* rset, const int32_t* size,
                 int32_t* pre) {
  cudaStream_t s = c->stream;
  DevScalars* d = c->dsc.get();
  const int64_t n = g.n;
  const int T = 256;
  // byte flags of vertices and communities, one clearing for all
  Buf<uint8_t> flags;
  DCD_TRY(flags.alloc(&c->mem, 3 * n));
  uint8_t *mark = flags.get(), *cflag = mark + n, *listed = cflag + n;
  DCD_TRY_CUDA(cudaMemsetAsync(mark, 0, 3 * n, s));
  DCD_TRY_CUDA(cudaMemsetAsync(&d->r_screen, 0, 4 * sizeof(int64_t), s));  // r_screen, gamma_deg, gamma_items, rest
  unsigned long long* gamma_deg = reinterpret_cast<unsigned long long*>(&d->gamma_deg);
  int32_t* item_cnt = reinterpret_cast<int32_t*>(&d->gamma_items);
  const bool may_pull = sb.total > 0 && 4 * sb.deg >= g.nnz;  // else pull cannot be taken
  PullBufs rest_bufs;
  PullRest rest{};
  if (may_pull) DCD_TRY(rest_bufs.alloc(&c->mem, n, g.nnz, d->rest_cnt, &rest));
  if (sb.total > 0) {
    const int64_t nsrc = sb.total, item_cap = nsrc + sb.deg / kGammaChunk;
    Buf<int32_t> src, cursor, jstar;
    Buf<uint8_t> intra;
    Buf<long long> gains;
    Buf<int64_t> items;
    DCD_TRY(src.alloc(&c->mem, nsrc));
    DCD_TRY(cursor.alloc(&c->mem, kMaxBins));
    DCD_TRY_CUDA(cudaMemsetAsync(cursor.get(), 0, kMaxBins * sizeof(int32_t), s));
    launch_bin_scatter(s, g.rp, n, WantSource{mo.pair_ptr.get()}, d, cursor.get(), src.get(), sb.plan);
    DCD_LAUNCH_CHECK();
    int64_t m2max = 0;
    for (int x = 0; x < c->G; x++) m2max = c->hgs[x].m2 > m2max ? c->hgs[x].m2 : m2max;
    const bool wide = m2max >= ((int64_t)1 << 31);
    DCD_TRY(jstar.alloc(&c->mem, nsrc));
    DCD_TRY(intra.alloc(&c->mem, nsrc));
    DCD_TRY(gains.alloc(&c->mem, (wide ? 2 : 1) * mo.npairs));
    DCD_TRY(items.alloc(&c->mem, item_cap));
    const SV sv{g.rp, g.col, g.w, k, labels0, a, mo.pkey.get(), mo.pflag.get(), mo.pair_ptr.get(), c->hgs[0].m2,
                c->G > 1 ? c->gid.get() : nullptr, c->gs.get(), mark, cflag, src.get(), jstar.get(), intra.get(),
                gains.get(), wide ? gains.get() + mo.npairs : nullptr, size, pre, nlab};
    if (wide) DCD_TRY(screen_rows<i128>(c, sv, g, sb));
    else DCD_TRY(screen_rows<long long>(c, sv, g, sb));
    trace("screen: phase A");
    if (wide)
      count_launch(), scr_decide<i128><<<grid_for(nsrc, T), T, 0, s>>>(sv, nsrc, listed, items.get(), item_cnt,
                                                                       gamma_deg);
    else
      count_launch(), scr_decide<long long><<<grid_for(nsrc, T), T, 0, s>>>(sv, nsrc, listed, items.get(), item_cnt,
                                                                            gamma_deg);
    count_launch(), scr_push<<<wave_grid(scr_push, item_cap * 32, T), T, 0, s>>>(sv, g.nnz, items.get(), item_cnt,
                                                                                 gamma_deg);
    DCD_LAUNCH_CHECK();
  }
  unsigned long long* count = reinterpret_cast<unsigned long long*>(&d->r_screen);
  count_launch(), build_rset<<<grid_for(n, T), T, 0, s>>>(n, g.nnz, g.rp, g.col, mark, cflag,
                                                          may_pull ? listed : nullptr, gamma_deg, labels0, rset,
                                                          rest, count);
  if (may_pull)
    count_launch(), pull_rest<<<4 * c->sms, kPullThreads, 0, s>>>(g.rp, g.col, rest, Listed{listed}, rset, count);
  DCD_LAUNCH_CHECK();
  return DCD_OK;
}

}  // namespace dcd
