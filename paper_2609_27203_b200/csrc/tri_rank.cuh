// Fused triangle aggregate  h(x, count) :- e(x,y), e(y,z), e(z,x)  over a degree-ordered copy of the graph, under logsumexp and
// sum-product.
//
// triangle.cuh finds every directed triangle three times, once from each of its corners, and walks 8.4e8 list entries on
// an R-MAT 18 graph to do so.  Here the nodes are numbered by degree and a triangle v -> a -> b -> v is found from its lowest
// corner v, of whose lists only the higher part is walked (at most sqrt(2 m) entries whatever the hubs; a few hundred on R-MAT
// graphs): 1.2e8 entries for the same graph.  Its
// term goes to all three corners.  The tags make that cheap: the term's weight exp(w_va + w_ab + w_bv) is the product of three
// numbers kept with the edges, and the sums are plain sums in fp64 (for sum-product the tags are such numbers already).
// Usable while no product of two or three can leave the normal fp32 range, in whatever order a corner sees its factors: |w| <=
// kTriRankMaxTag under logsumexp, w = 0 or kTriRankMinNum <= |w| <= kTriRankMaxNum under sum-product.
//
// Two launches, one per group of corners, so that no sum is formed by atomics in an order that varies:
//   by a:  mark out(a) in a shared-memory bitmap; for every lower v with v -> a walk the higher b with b -> v: a marked b closes
//          a triangle.  S[a] is the block's sum; v's part is a sum per edge (v,a), written in v's own order.
//   by b:  the same over the reversed graph (mark in(b), for every lower v with b -> v walk the higher a with v -> a): S[b].
// A corner a with little to walk is handled by one warp that searches out(a) instead (k_tri_rank_small).  k_tri_rank_groups then
// adds up each node's parts: its units' sums of both launches and its edges' sums.
//
// R-MAT 18 (3.9 M edges, 39 M triangles): 5.47 -> 1.03 ms per evaluation, 0.83 ms of it the two bitmap launches (bound by instruction
// issue: 75 % of the slots; 0.88 with a chain of reads ahead of every item's list), 0.11 the searched corners; the first one on a new
// relation, which orders the graph, 5.82 -> 2.42.
#pragma once
#include "common.cuh"

namespace xlog {

constexpr int64_t kTriRankMaxNodes = (int64_t)1 << 19;       // 128 KB of bitmap and places
constexpr uint32_t kTriRankMinEdges = 1u << 17;  // below, the plain kernels are as fast and need no second copy of the graph
// Ordering a graph costs 0.25 ms and 0.16 ms per million edges once; it is ordered where that is back by the second evaluation.
// Which way a graph goes depends on the graph alone, so that its results repeat bit for bit.  Entries to walk: per edge the
// shorter of the two lists that the plain kernels meet.  First / later evaluation, ms, plain and ordered:
//   R-MAT 15, 0.16 M edges, 33 entries an edge   0.46 / 0.37 and 0.53 / 0.16     16, 0.96 M, 106   1.50 / 1.38 and 0.89 / 0.32
//   even, 2,000 nodes, 0.20 M edges, 92 an edge  0.40 / 0.32 and 0.49 / 0.15     60,000 nodes, 1.0 M, 14   0.54 / 0.42 and 0.68 / 0.16
// and, below the line, even, 100,000 nodes, 0.14 M, 0.8   0.28 / 0.18 and 0.53 / 0.11     250,000 nodes, 1.0 M, 3   0.56 / 0.41 and 0.87 / 0.26
constexpr uint64_t kTriRankPerEdge = 32, kTriRankEntries = 10000000;      // entries per edge; entries and five times the edges
constexpr uint32_t kTriRankHub = 1u << 15;       // a list that the plain kernels are slow with: wheel of 70,000 nodes 1.17 / 1.08 and 0.89 / 0.34
constexpr float kTriRankMaxTag = 28.f;           // exp(3 * 28) and exp(-3 * 28) are normal fp32 numbers
constexpr float kTriRankMaxNum = 0x1p42f, kTriRankMinNum = 0x1p-42f;      // as are 2^126 and 2^-126
constexpr int kTriRankBlock = 512;
// corners with fewer entries to walk are searched, a warp each; a block's bitmap costs about as much as 500 searches in a row
// (all kernels, us, at limits of 2048 / 1024 / 512: R-MAT 18 1186 / 1203 / 1212, R-MAT 16 367 / 304 / 284, R-MAT 14 271 / 200 / 173)
constexpr uint32_t kTriRankSmall = 512;
constexpr int kTriRankSweeps = 2;                // sweeps of 32 list entries a warp reads before it tests them (both launches, us: 1 907, 2 878, 3 909, 4 962)

enum { kTrkEdges = 0, kTrkNodes = 1, kTrkLoops = 2, kTrkAbsMax = 3, kTrkUnitsA = 4, kTrkUnitsB = 5, kTrkWalkA = 6, kTrkWalkB = 7,
       kTrkAbsMin = 8, kTrkPlain = 9, kTrkLongest = 10, kTrkTotals = 11 };      // kTrkAbsMin: complement of the smallest |tag| that is not zero (0: none)

// One orientation of the ordered graph: lists of neighbours in ascending rank; entries [off[v], split[v]) rank lower than v.
struct TriRankLists {
  const uint32_t* off;
  const uint32_t* split;
  const uint32_t* nbr;
  const float* e;                    // the edge's number
  const uint32_t* other;             // the place of the same edge in the other orientation's lists (may be null)
};

// degree of every corner, of the other nodes 0
static __global__ void __launch_bounds__(256) k_trk_degrees(const uint32_t* __restrict__ out_off, int64_t out_domain, const uint32_t* __restrict__ in_off, int64_t in_domain,
                                                            uint32_t n_nodes, uint32_t* __restrict__ deg, uint32_t* __restrict__ node) {
  for (uint32_t v = blockIdx.x * blockDim.x + threadIdx.x; v < n_nodes; v += gridDim.x * blockDim.x) {
    const uint32_t o = v < out_domain ? out_off[v + 1] - out_off[v] : 0u, i = v < in_domain ? in_off[v + 1] - in_off[v] : 0u;
    deg[v] = o && i ? o + i : 0u;
    node[v] = v;
  }
}
// rank of every node among the corners, in order of degree (node: the nodes sorted by degree); the others get n_nodes
static __global__ void __launch_bounds__(256) k_trk_ranks(const uint32_t* __restrict__ node, uint32_t n_nodes, uint32_t corners, uint32_t* __restrict__ rank) {
  const uint32_t skip = n_nodes - corners;
  for (uint32_t i = blockIdx.x * blockDim.x + threadIdx.x; i < n_nodes; i += gridDim.x * blockDim.x) rank[node[i]] = i >= skip ? i - skip : n_nodes;
}
// What decides whether the graph is ordered, in one read of its nodes and edges: corners (nodes with edges in and out), longest
// list, edges between corners, loops, the range of |tag|, and the entries that the plain kernels would walk (per edge the shorter
// of the two lists that are met).
static __global__ void __launch_bounds__(256) k_trk_check(const int32_t* __restrict__ src, const int32_t* __restrict__ dst, const float* __restrict__ w, uint32_t n,
                                                          const uint32_t* __restrict__ out_off, int64_t out_domain, const uint32_t* __restrict__ in_off, int64_t in_domain,
                                                          uint32_t n_nodes, unsigned long long* __restrict__ totals) {
  __shared__ unsigned long long s_walk;
  __shared__ uint32_t s_kept, s_loops, s_top, s_low, s_corners, s_longest;
  if (threadIdx.x == 0) { s_walk = 0; s_kept = s_loops = s_top = s_low = s_corners = s_longest = 0; }
  __syncthreads();
  uint32_t kept = 0, loops = 0, top = 0, low = 0, corners = 0, longest = 0;
  for (uint32_t v = blockIdx.x * blockDim.x + threadIdx.x; v < n_nodes; v += gridDim.x * blockDim.x) {
    const uint32_t o = v < out_domain ? out_off[v + 1] - out_off[v] : 0u, i = v < in_domain ? in_off[v + 1] - in_off[v] : 0u;
    corners += o && i;
    longest = max(longest, max(o, i));
  }
  unsigned long long walk = 0;
  for (uint32_t e = blockIdx.x * blockDim.x + threadIdx.x; e < n; e += gridDim.x * blockDim.x) {
    const int32_t s = src[e], d = dst[e];
    const uint32_t si = s < in_domain ? in_off[s + 1] - in_off[s] : 0u, dn = d < out_domain ? out_off[d + 1] - out_off[d] : 0u;
    kept += si && dn;                               // the source has edges out, the target has edges in: this one
    walk += min(si, dn);
    loops += s == d;
    const uint32_t t = __float_as_uint(fabsf(w[e]));
    top = max(top, t);
    if (t) low = max(low, ~t);
  }
  kept = __reduce_add_sync(0xffffffffu, kept); loops = __reduce_add_sync(0xffffffffu, loops); top = __reduce_max_sync(0xffffffffu, top); low = __reduce_max_sync(0xffffffffu, low);
  corners = __reduce_add_sync(0xffffffffu, corners); longest = __reduce_max_sync(0xffffffffu, longest);
#pragma unroll
  for (int d = 16; d; d >>= 1) walk += __shfl_xor_sync(0xffffffffu, walk, d);
  if (lane_id() == 0) { atomicAdd(&s_walk, walk); atomicAdd(&s_kept, kept); atomicAdd(&s_loops, loops); atomicMax(&s_top, top); atomicMax(&s_low, low); atomicAdd(&s_corners, corners); atomicMax(&s_longest, longest); }
  __syncthreads();
  if (threadIdx.x == 0) {
    atomicAdd(totals + kTrkEdges, (unsigned long long)s_kept);
    if (s_loops) atomicAdd(totals + kTrkLoops, (unsigned long long)s_loops);
    atomicAdd(totals + kTrkPlain, s_walk);
    atomicMax(totals + kTrkAbsMax, (unsigned long long)s_top);
    atomicMax(totals + kTrkAbsMin, (unsigned long long)s_low);
    if (s_corners) atomicAdd(totals + kTrkNodes, (unsigned long long)s_corners);
    atomicMax(totals + kTrkLongest, (unsigned long long)s_longest);
  }
}
// the edges between corners first: key = rank of the source, of the others n_nodes
static __global__ void __launch_bounds__(256) k_trk_edges(const int32_t* __restrict__ src, const int32_t* __restrict__ dst, uint32_t n,
                                                          const uint32_t* __restrict__ rank, uint32_t n_nodes, uint32_t* __restrict__ key, uint32_t* __restrict__ edge) {
  for (uint32_t e = blockIdx.x * blockDim.x + threadIdx.x; e < n; e += gridDim.x * blockDim.x) {
    const uint32_t s = rank[src[e]];
    key[e] = s < n_nodes && rank[dst[e]] < n_nodes ? s : n_nodes;
    edge[e] = e;
  }
}
static __global__ void __launch_bounds__(256) k_trk_keys(const uint32_t* __restrict__ edge, uint32_t n, const int32_t* __restrict__ col, const uint32_t* __restrict__ rank, uint32_t* __restrict__ key) {
  for (uint32_t i = blockIdx.x * blockDim.x + threadIdx.x; i < n; i += gridDim.x * blockDim.x) key[i] = rank[col[edge[i]]];
}
// lists of one orientation from the edges in its order; place[e] (optional) = where edge e went
template <bool EXP>
__global__ void __launch_bounds__(256) k_trk_lists(const uint32_t* __restrict__ edge, uint32_t n, const int32_t* __restrict__ nbr_col, const float* __restrict__ w,
                                                   const uint32_t* __restrict__ rank, uint32_t* __restrict__ nbr, float* __restrict__ num, uint32_t* __restrict__ place) {
  for (uint32_t i = blockIdx.x * blockDim.x + threadIdx.x; i < n; i += gridDim.x * blockDim.x) {
    const uint32_t e = edge[i];
    nbr[i] = rank[nbr_col[e]];
    num[i] = EXP ? expf(w[e]) : w[e];
    if (place) place[e] = i;
  }
}
static __global__ void __launch_bounds__(256) k_trk_gather(const uint32_t* __restrict__ edge, uint32_t n, const uint32_t* __restrict__ place, uint32_t* __restrict__ other) {
  for (uint32_t i = blockIdx.x * blockDim.x + threadIdx.x; i < n; i += gridDim.x * blockDim.x) other[i] = place[edge[i]];
}
// first entry that ranks higher than v in each of v's two lists
static __global__ void __launch_bounds__(256) k_trk_splits(const uint32_t* __restrict__ off0, const uint32_t* __restrict__ nbr0, uint32_t* __restrict__ split0,
                                                           const uint32_t* __restrict__ off1, const uint32_t* __restrict__ nbr1, uint32_t* __restrict__ split1, uint32_t n_nodes) {
  for (uint32_t i = blockIdx.x * blockDim.x + threadIdx.x; i < 2 * n_nodes; i += gridDim.x * blockDim.x) {
    const uint32_t v = i < n_nodes ? i : i - n_nodes;
    const uint32_t* __restrict__ off = i < n_nodes ? off0 : off1;
    const uint32_t* __restrict__ nbr = i < n_nodes ? nbr0 : nbr1;
    uint32_t lo = off[v], hi = off[v + 1];
    while (lo < hi) { const uint32_t mid = (lo + hi) >> 1; if (nbr[mid] < v) lo = mid + 1; else hi = mid; }
    (i < n_nodes ? split0 : split1)[v] = lo;
  }
}

// Items of a unit: enough that marking the corner's list (`marked` entries) is a small part of the unit's walk; for a hub, whose
// items are many and walk an entry or two each, enough units that the blocks of one corner fill the device (wheels of 70,000 and
// 400,000 nodes, ms per evaluation, an eighth / a 64th of the list: 0.94 / 0.34 and 5.37 / 1.63; the plain kernels 1.08 and 5.48).
__device__ __forceinline__ uint32_t trk_unit_items(uint32_t marked) { return marked >= kTriRankHub ? marked / 64u : max(256u, marked / 8u); }

// Entries that every corner a walks in the lists of its lower neighbours, work[a] (zero on entry): each v adds the length of its
// higher list in I to its higher neighbours in M, which are the corners that it is a lower neighbour of.  Eight lanes a v, whose
// higher lists are short whatever the hubs; a warp a corner took 5 ms to go through the 400,000 neighbours of a wheel's hub.
static __global__ void __launch_bounds__(256) k_trk_work(TriRankLists I, TriRankLists M, uint32_t n_nodes, uint32_t* __restrict__ work) {
  const uint32_t sub = threadIdx.x % 8;
  for (uint32_t v = (blockIdx.x * blockDim.x + threadIdx.x) / 8; v < n_nodes; v += gridDim.x * blockDim.x / 8) {
    const uint32_t n = I.off[v + 1] - I.split[v], e1 = M.off[v + 1];
    if (n) for (uint32_t i = M.split[v] + sub; i < e1; i += 8) atomicAdd(work + M.nbr[i], n);
  }
}
// units of the bitmap kernel (0: the corner is searched); *walk += all of work
static __global__ void __launch_bounds__(256) k_trk_units(TriRankLists I, TriRankLists M, uint32_t n_nodes, const uint32_t* __restrict__ work, uint32_t* __restrict__ units,
                                                          unsigned long long* __restrict__ walk) {
  __shared__ unsigned long long s_sum;
  if (threadIdx.x == 0) s_sum = 0;
  __syncthreads();
  unsigned long long sum = 0;
  for (uint32_t a = blockIdx.x * blockDim.x + threadIdx.x; a <= n_nodes; a += gridDim.x * blockDim.x) {
    uint32_t u = 0;
    if (a < n_nodes) {
      const uint32_t n = work[a], per = trk_unit_items(M.off[a + 1] - M.off[a]);
      if (n >= kTriRankSmall) u = (I.split[a] - I.off[a] + per - 1) / per;
      sum += n;
    }
    units[a] = u;
  }
#pragma unroll
  for (int d = 16; d; d >>= 1) sum += __shfl_xor_sync(0xffffffffu, sum, d);
  if (lane_id() == 0 && sum) atomicAdd(&s_sum, sum);
  __syncthreads();
  if (threadIdx.x == 0 && s_sum) atomicAdd(walk, s_sum);
}
static __global__ void __launch_bounds__(256) k_trk_unit_fill(TriRankLists I, TriRankLists M, uint32_t n_nodes, const uint32_t* __restrict__ unit_off, uint2* __restrict__ unit) {
  for (uint32_t a = blockIdx.x * blockDim.x + threadIdx.x; a < n_nodes; a += gridDim.x * blockDim.x) {
    const uint32_t per = trk_unit_items(M.off[a + 1] - M.off[a]);
    for (uint32_t u = unit_off[a], i = I.off[a]; u < unit_off[a + 1]; ++u, i += per) unit[u] = make_uint2(a, i);
  }
}

struct TriRankPass {
  TriRankLists I;                    // the corner's neighbours (lower ones are the v), and the v's lists that are walked
  TriRankLists M;                    // the corner's list that is marked
  uint32_t n_nodes;
  const uint32_t* unit_off;
  const uint2* unit;
  uint32_t n_units;
  double* unit_sum;                  // per unit, then per searched corner at n_units + a
  uint32_t* unit_cnt;
  double* edge_sum;                  // per edge (v, corner), at its place in v's list of the other orientation (null: not wanted)
  uint32_t* edge_cnt;
};

// One block per unit, the corners of highest degree (the longest units) first.  A warp takes an item (a lower neighbour v) and
// walks v's higher neighbours, kTriRankSweeps sweeps of them in flight; hits multiply and add where they fall.
template <bool EDGES>
__global__ void __launch_bounds__(kTriRankBlock) k_tri_rank(const __grid_constant__ TriRankPass P) {
  extern __shared__ uint32_t trk_smem[];
  __shared__ double s_sum[kTriRankBlock / 32];
  __shared__ uint32_t s_cnt[kTriRankBlock / 32];
  const uint32_t words = (P.n_nodes + 31) / 32;
  uint32_t* bits = trk_smem;
  uint32_t* before = trk_smem + words;             // per word: place in the marked list of the first entry marked in it
  const unsigned lane = lane_id(), wid = warp_id();
  const uint32_t u = P.n_units - 1 - blockIdx.x;
  const uint2 un = P.unit[u];
  const uint32_t a = un.x, m0 = P.M.off[a], m1 = P.M.off[a + 1];
  for (uint32_t i = threadIdx.x; i < words; i += kTriRankBlock) bits[i] = 0u;
  __syncthreads();
  for (uint32_t i = m0 + threadIdx.x; i < m1; i += kTriRankBlock) {
    const uint32_t z = P.M.nbr[i];
    atomicOr(bits + (z >> 5), 1u << (z & 31));
    if (i == m0 || (P.M.nbr[i - 1] >> 5) != (z >> 5)) before[z >> 5] = i;
  }
  __syncthreads();
  const uint32_t it0 = un.y, it1 = min(it0 + trk_unit_items(m1 - m0), P.I.split[a]);
  double sum = 0.0;
  uint32_t cnt = 0;
  // a warp takes one in sixteen of the unit's items (neighbours have lists of like length), and a lane each fetches the next 32 items' bounds
  for (uint32_t b0 = it0 + wid; b0 < it1; b0 += kTriRankBlock) {
    const uint32_t ib = b0 + lane * (kTriRankBlock / 32);
    uint32_t first = 0, end = 0;
    float e = 0.f;
    if (ib < it1) { const uint32_t v = P.I.nbr[ib]; e = P.I.e[ib]; first = P.I.split[v]; end = P.I.off[v + 1]; }
#pragma unroll 1
    for (uint32_t j = 0, it = b0; it < it1 && j < 32; ++j, it += kTriRankBlock / 32) {
      const uint32_t w0 = __shfl_sync(0xffffffffu, first, j), w1 = __shfl_sync(0xffffffffu, end, j);
      const float ev = __shfl_sync(0xffffffffu, e, j);
      double isum = 0.0;
      uint32_t icnt = 0;
      for (uint32_t i0 = w0; i0 < w1; i0 += 32 * kTriRankSweeps) {
        uint32_t z[kTriRankSweeps], wd[kTriRankSweeps];
#pragma unroll
        for (int k = 0; k < kTriRankSweeps; ++k) { const uint32_t i = i0 + k * 32 + lane; z[k] = i < w1 ? P.I.nbr[i] : 0xffffffffu; }
#pragma unroll
        for (int k = 0; k < kTriRankSweeps; ++k) wd[k] = z[k] != 0xffffffffu ? bits[z[k] >> 5] : 0u;
#pragma unroll
        for (int k = 0; k < kTriRankSweeps; ++k)
          if ((wd[k] >> (z[k] & 31)) & 1u) {
            const uint32_t at = before[z[k] >> 5] + __popc(wd[k] & ((1u << (z[k] & 31)) - 1u));
            isum += (double)((ev * P.M.e[at]) * P.I.e[i0 + k * 32 + lane]);
            ++icnt;
          }
      }
      sum += isum; cnt += icnt;
      if (EDGES) {
        icnt = __reduce_add_sync(0xffffffffu, icnt);
        if (icnt)
#pragma unroll
          for (int d = 16; d; d >>= 1) isum += __shfl_xor_sync(0xffffffffu, isum, d);
        if (lane == 0) { const uint32_t o = P.I.other[it]; P.edge_sum[o] = isum; P.edge_cnt[o] = icnt; }
      }
    }
  }
  cnt = __reduce_add_sync(0xffffffffu, cnt);
#pragma unroll
  for (int d = 16; d; d >>= 1) sum += __shfl_xor_sync(0xffffffffu, sum, d);
  if (lane == 0) { s_sum[wid] = sum; s_cnt[wid] = cnt; }
  __syncthreads();
  if (threadIdx.x == 0) {
    double t = 0.0;
    uint32_t c = 0;
    for (int w = 0; w < kTriRankBlock / 32; ++w) { t += s_sum[w]; c += s_cnt[w]; }
    P.unit_sum[u] = t; P.unit_cnt[u] = c;
  }
}

// The corners without units, a warp each: 32 items at a time, their entries laid out in a line over the lanes, every entry
// searched in the corner's list (in shared memory where it has at most kTriRankListed entries).  The values of one item are
// neighbours in that line: a segmented scan per step brings them together in a fixed order.
constexpr uint32_t kTriRankListed = 512;
template <bool EDGES>
__global__ void __launch_bounds__(256) k_tri_rank_small(const __grid_constant__ TriRankPass P) {
  __shared__ uint32_t s_list[8][kTriRankListed];
  __shared__ double s_item[8][32];
  __shared__ uint32_t s_hits[8][32];
  const uint32_t nwarps = (gridDim.x * blockDim.x) >> 5;
  const unsigned lane = lane_id(), wid = warp_id();
  for (uint32_t a = (blockIdx.x * blockDim.x + threadIdx.x) >> 5; a < P.n_nodes; a += nwarps) {
    if (P.unit_off[a + 1] != P.unit_off[a]) continue;
    const uint32_t m0 = P.M.off[a], nm = P.M.off[a + 1] - m0, i1 = P.I.split[a];
    const bool listed = nm <= kTriRankListed;
    __syncwarp();
    if (listed && i1 > P.I.off[a]) for (uint32_t i = lane; i < nm; i += 32) s_list[wid][i] = P.M.nbr[m0 + i];
    __syncwarp();
    double sum = 0.0;
    uint32_t cnt = 0;
    for (uint32_t ib = P.I.off[a]; ib < i1; ib += 32) {
      const uint32_t it = ib + lane;
      uint32_t w0 = 0, n = 0;
      float ev = 0.f;
      if (it < i1) { const uint32_t v = P.I.nbr[it]; ev = P.I.e[it]; w0 = P.I.split[v]; n = P.I.off[v + 1] - w0; }
      if (EDGES) { s_item[wid][lane] = 0.0; s_hits[wid][lane] = 0u; }
      const uint32_t incl = warp_scan_incl(n), total = __shfl_sync(0xffffffffu, incl, 31);
      const uint32_t from = w0 + n - incl;             // entry p of the line is entry from + p of its item's list
      __syncwarp();
      for (uint32_t p0 = 0; p0 < total; p0 += 32) {
        const uint32_t p = p0 + lane;
        uint32_t owner = 0;                            // first item whose inclusive prefix exceeds p
#pragma unroll
        for (int d = 16; d; d >>= 1) { const uint32_t x = __shfl_sync(0xffffffffu, incl, owner + d - 1); if (x <= p) owner += d; }
        const uint32_t i = __shfl_sync(0xffffffffu, from, owner) + p;
        const float e = __shfl_sync(0xffffffffu, ev, owner);
        double val = 0.0;
        uint32_t hit = 0;
        if (p < total) {
          const uint32_t z = P.I.nbr[i];
          uint32_t lo = 0, hi = nm;
          if (listed) while (lo < hi) { const uint32_t mid = (lo + hi) >> 1; if (s_list[wid][mid] < z) lo = mid + 1; else hi = mid; }
          else while (lo < hi) { const uint32_t mid = (lo + hi) >> 1; if (P.M.nbr[m0 + mid] < z) lo = mid + 1; else hi = mid; }
          if (lo < nm && (listed ? s_list[wid][lo] : P.M.nbr[m0 + lo]) == z) { hit = 1u; val = (double)((e * P.M.e[m0 + lo]) * P.I.e[i]); }
        }
        sum += val; cnt += hit;
        if (EDGES && __any_sync(0xffffffffu, hit)) {
#pragma unroll
          for (int d = 1; d < 32; d <<= 1) {
            const double ov = __shfl_up_sync(0xffffffffu, val, d);
            const uint32_t oh = __shfl_up_sync(0xffffffffu, hit, d), oo = __shfl_up_sync(0xffffffffu, owner, d);
            if ((int)lane >= d && oo == owner) { val += ov; hit += oh; }
          }
          const uint32_t next = __shfl_down_sync(0xffffffffu, owner, 1);
          if (hit && (lane == 31 || next != owner)) { s_item[wid][owner] += val; s_hits[wid][owner] += hit; }
          __syncwarp();
        }
      }
      if (EDGES && it < i1) { const uint32_t o = P.I.other[it]; P.edge_sum[o] = s_item[wid][lane]; P.edge_cnt[o] = s_hits[wid][lane]; }
      __syncwarp();
    }
    cnt = __reduce_add_sync(0xffffffffu, cnt);
#pragma unroll
    for (int d = 16; d; d >>= 1) sum += __shfl_xor_sync(0xffffffffu, sum, d);
    if (lane == 0) { P.unit_sum[P.n_units + a] = sum; P.unit_cnt[P.n_units + a] = cnt; }
  }
}

// Eight lanes a node of the relation: its parts from both launches and from its edges to higher corners, in a fixed order.  A chain of
// reads (rank, bounds, sums) and few of them a node: R-MAT 18 51 us, a warp a node 88.
constexpr int kTrkGroupLanes = 8;
template <bool LSE>
__global__ void __launch_bounds__(256) k_tri_rank_groups(TriRankPass A, TriRankPass B, const uint32_t* __restrict__ rank, int64_t domain, uint32_t* __restrict__ grp_cnt,
                                                         float* __restrict__ grp_tag, uint32_t* __restrict__ flag, uint32_t* __restrict__ max_cnt, uint32_t* __restrict__ err) {
  constexpr int G = kTrkGroupLanes;
  const int64_t step = (int64_t)gridDim.x * 256 / G;
  const unsigned sub = threadIdx.x % G;
  uint32_t top = 0;
  for (int64_t x0 = ((int64_t)blockIdx.x * 256 + threadIdx.x) / 32 * (32 / G); x0 < domain; x0 += step) {      // uniform over the warp
    const int64_t x = x0 + lane_id() / G;
    const uint32_t v = x < domain ? rank[x] : 0xffffffffu;
    double sum = 0.0;
    uint64_t cnt = 0;
    if (v < A.n_nodes) {
      const uint32_t e0 = A.M.split[v] + sub, e1 = A.M.off[v + 1];
#pragma unroll
      for (int p = 0; p < 2; ++p) {
        const TriRankPass& Q = p ? B : A;
        const uint32_t u0 = Q.unit_off[v], u1 = Q.unit_off[v + 1];
        for (uint32_t u = u0 + sub; u < u1; u += G) { sum += Q.unit_sum[u]; cnt += Q.unit_cnt[u]; }
        if (u0 == u1 && sub == 0) { sum += Q.unit_sum[Q.n_units + v]; cnt += Q.unit_cnt[Q.n_units + v]; }
      }
#pragma unroll 4
      for (uint32_t i = e0; i < e1; i += G) { sum += A.edge_sum[i]; cnt += A.edge_cnt[i]; }
    }
#pragma unroll
    for (int d = G / 2; d; d >>= 1) { sum += __shfl_xor_sync(0xffffffffu, sum, d); cnt += __shfl_xor_sync(0xffffffffu, cnt, d); }
    if (sub == 0 && x < domain) {
      if (cnt > 0x7fffffffull) { atomicOr(err, kErrCountOverflow); cnt = 0x7fffffffull; }
      grp_cnt[x] = (uint32_t)cnt;
      grp_tag[x] = cnt ? (LSE ? (float)log(sum) : (float)sum) : 0.f;
      flag[x] = cnt ? 1u : 0u;
      top = max(top, (uint32_t)cnt);
    }
  }
  top = __reduce_max_sync(0xffffffffu, top);
  if (lane_id() == 0 && top) atomicMax(max_cnt, top);
}

}  // namespace xlog
