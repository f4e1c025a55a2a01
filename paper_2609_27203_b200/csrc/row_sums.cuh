// Row-local fixpoint of the additive recursion  h(a, c) :- h(a, b), r(b, c)  (path sums under logsumexp or sum-product on an
// acyclic graph) when one value of a owns few enough keys to live in shared memory.
//
// As in row_fixpoint.cuh the rule never changes a, so the rounds of the delta form  Delta' = T(Delta), I' = I (+) Delta'  fall
// apart into one independent sequence per a and the whole stratum after its seed round is one launch: a block takes a
// value of a and keeps I, Delta and Delta' of that row in shared memory.  The oplus is not idempotent, so candidates are not
// applied where they fall: a round first marks the targets c of Delta's runs of r (shared-memory bitmap, first marker queues
// c), then every queued c collects its candidates from r's transposed run of c, in index order, testing Delta's bitmap per
// entry.  Each c's sum is thus formed by one thread (or one warp with a fixed tree, for long runs) in an order that depends
// on the graph alone: results repeat from run to run, and the accumulation is that of the reduce-by-key kernels
// ((max, sum) pairs for logsumexp, fp64 for sums).
//
// What bounds it: latency.  On the closure of a 1,000-node DAG (4,000 edges, 90 K tuples, 20 rounds) a row's round holds 13
// candidates: a chain of half a dozen dependent L1 / L2 reads and two block barriers.  The same rounds on the sorting route are
// 17 launches and two control reads each: 3.61 ms against 0.29 ms per evaluation, 0.09 ms of it this kernel (a thread per row in
// blocks of 128: 0.22 ms, of 512: 0.10; four lanes per row in blocks of 512, entries read four at a time: 0.086).
#pragma once
#include "common.cuh"
#include "row_fixpoint.cuh"

namespace xlog {

constexpr int kRowSumBlock = 512;
constexpr int kRowSumLanes = 4;                  // lanes to a delta row or target; runs longer than kRowSumLong take the whole warp
constexpr uint32_t kRowSumLong = 32;

// Totals of the launch, in the control words.
enum { kRsCandidates = 0, kRsUnique = 1, kRsNew = 2, kRsRounds = 3, kRsCapped = 4, kRsTotals = 5 };

struct RowSumRule {                  // h(a, c) :- h(a, b), r(b, c)
  const uint32_t* off;               // r over its first column b: targets z
  uint32_t domain;
  const int32_t* z;
  const uint32_t* in_off;            // r over its second column c: sources and tags, ascending sources
  uint32_t in_domain;
  const int32_t* in_b;
  const float* in_w;
};

struct RowSums {
  RowSumRule rules[kRowMaxRules];
  int n_rules;
  uint32_t n_rows;                   // values of a
  int c_bits;                        // log2 of the slots per row
  uint32_t z_max;
  uint32_t max_rounds;
  int times;                         // otimes is * instead of +
  const uint32_t* start;             // [2][n_rows + 1]: first row of every a in the relation and in the seed round's delta
  const uint32_t* keys;              // the relation after the seed round (a << c_bits | c, ascending)
  const float* tags;
  const uint32_t* dkeys;             // its delta
  const float* dtags;
  int32_t* table;                    // out: one order-mapped tag per slot, kMirrorEmptyMin where no tuple is
  unsigned long long* totals;
  uint32_t* err;
};

// shared memory: I, Delta, Delta' (4 B per slot each), two slot lists (2 B), four bitmaps
inline size_t row_sums_smem(int c_bits) { return ((size_t)16 << c_bits) + 16 * std::max<size_t>(((size_t)1 << c_bits) / 32, 1); }

// start[a] = first key of row a, for a in 0 .. n_rows, in the relation and in the delta
static __global__ void __launch_bounds__(256) k_row_starts(const uint32_t* __restrict__ keys, uint32_t n, const uint32_t* __restrict__ dkeys, uint32_t dn,
                                                          int c_bits, uint32_t n_rows, uint32_t* __restrict__ start) {
  const uint32_t i = blockIdx.x * blockDim.x + threadIdx.x;
  if (i >= 2 * (n_rows + 1)) return;
  const bool second = i > n_rows;
  const uint64_t want = (uint64_t)(second ? i - n_rows - 1 : i) << c_bits;
  const uint32_t* k = second ? dkeys : keys;
  uint32_t lo = 0, hi = second ? dn : n;
  while (lo < hi) { const uint32_t mid = lo + ((hi - lo) >> 1); if ((uint64_t)k[mid] < want) lo = mid + 1; else hi = mid; }
  start[i] = lo;
}

template <typename Op>
__global__ void __launch_bounds__(kRowSumBlock) k_row_sums(const __grid_constant__ RowSums P) {
  typedef typename Op::A A;
  extern __shared__ uint32_t rs_smem[];
  __shared__ uint32_t s_touched[2];                               // targets queued, by the parity of the round
  const uint32_t S = 1u << P.c_bits, W = max(S >> 5, 1u), smask = S - 1;
  float* sum = reinterpret_cast<float*>(rs_smem);                 // I
  float* d = sum + S;                                             // Delta
  float* dn = d + S;                                              // Delta'
  uint32_t* pres = rs_smem + 3 * S;                               // keys of I, of Delta, of Delta'; one being cleared for the next round
  uint32_t* has = pres + W;
  uint32_t* mark = has + W;
  uint32_t* spare = mark + W;
  uint16_t* list = reinterpret_cast<uint16_t*>(spare + W);        // slots of Delta, of Delta'
  uint16_t* next = list + S;
  constexpr int G = kRowSumLanes, kRowsPerBlock = kRowSumBlock / G;
  const unsigned lane = lane_id(), sub = lane % G;
  unsigned long long cand = 0, uniq = 0;
  uint32_t fresh = 0, rounds_seen = 0, capped = 0;
  for (uint32_t a = blockIdx.x; a < P.n_rows; a += gridDim.x) {
    const size_t base = (size_t)a << P.c_bits;
    const uint32_t i0 = P.start[a], i1 = P.start[a + 1], d0 = P.start[P.n_rows + 1 + a], d1 = P.start[P.n_rows + 2 + a];
    for (uint32_t i = threadIdx.x; i < W; i += kRowSumBlock) { pres[i] = 0u; has[i] = 0u; mark[i] = 0u; spare[i] = 0u; }
    __syncthreads();
    for (uint32_t i = i0 + threadIdx.x; i < i1; i += kRowSumBlock) {
      const uint32_t c = P.keys[i] & smask;
      sum[c] = P.tags[i];
      atomicOr(pres + (c >> 5), 1u << (c & 31));
    }
    for (uint32_t i = d0 + threadIdx.x; i < d1; i += kRowSumBlock) {
      const uint32_t c = P.dkeys[i] & smask;
      d[c] = P.dtags[i];
      list[i - d0] = (uint16_t)c;
      atomicOr(has + (c >> 5), 1u << (c & 31));
    }
    if (threadIdx.x == 0) s_touched[0] = s_touched[1] = 0;
    __syncthreads();
    uint32_t nd = d1 - d0, rounds = 0;
    while (nd) {
      if (rounds >= P.max_rounds) { capped = 1; break; }
      const uint32_t par = rounds & 1;
      ++rounds;
      // the targets of Delta's runs: G lanes per delta row, long runs by the whole warp.  The bitmap of the round before is
      // cleared on the side: it takes the marks of the next round.
      for (uint32_t i = threadIdx.x; i < W; i += kRowSumBlock) spare[i] = 0u;
      for (int q = 0; q < P.n_rules; ++q) {
        const RowSumRule& R = P.rules[q];
        auto touch = [&](uint32_t c) {
          if (c > P.z_max || c >= S) { atomicOr(P.err, kErrHeadRange); return; }
          const uint32_t bit = 1u << (c & 31);
          if (!(atomicOr(mark + (c >> 5), bit) & bit)) next[atomicAdd(&s_touched[par], 1u)] = (uint16_t)c;
        };
        for (uint32_t r0 = warp_id() * (32 / G); r0 < nd; r0 += kRowsPerBlock) {
          uint32_t lo = 0, dg = 0;
          if (r0 + lane / G < nd) {
            const uint32_t b = list[r0 + lane / G];
            if (b < R.domain) { lo = R.off[b]; dg = R.off[b + 1] - lo; }
          }
          if (sub == 0) cand += dg;
          if (dg <= kRowSumLong)
            for (uint32_t j = sub; j < dg; j += 4 * G) {       // four targets in flight
              int32_t c[4];
#pragma unroll
              for (int k = 0; k < 4; ++k) c[k] = j + k * G < dg ? R.z[lo + j + k * G] : -1;
#pragma unroll
              for (int k = 0; k < 4; ++k) if (c[k] >= 0) touch((uint32_t)c[k]);
            }
          unsigned big = __ballot_sync(0xffffffffu, sub == 0 && dg > kRowSumLong);
          while (big) {
            const int src = __ffs(big) - 1;
            big &= big - 1;
            const uint32_t L = __shfl_sync(0xffffffffu, lo, src), N = __shfl_sync(0xffffffffu, dg, src);
            for (uint32_t j = lane; j < N; j += 32) touch((uint32_t)R.z[L + j]);
          }
        }
      }
      __syncthreads();
      const uint32_t nt = s_touched[par];
      if (threadIdx.x == 0) { s_touched[par ^ 1] = 0; uniq += nt; }
      // every target collects its candidates (G lanes each, a fixed tree over the lanes); their sum is Delta', and I takes it in
      for (uint32_t r0 = warp_id() * (32 / G); r0 < nt; r0 += kRowsPerBlock) {
        const bool mine = r0 + lane / G < nt;
        const uint32_t c = mine ? next[r0 + lane / G] : 0u;
        A acc = Op::identity();
        for (int q = 0; q < P.n_rules; ++q) {
          const RowSumRule& R = P.rules[q];
          uint32_t lo = 0, dg = 0;
          if (mine && c < R.in_domain) { lo = R.in_off[c]; dg = R.in_off[c + 1] - lo; }
          auto take = [&](A& into, uint32_t b, float w) {
            if (b < S && ((has[b >> 5] >> (b & 31)) & 1u)) into = Op::combine(into, Op::lift(P.times ? d[b] * w : d[b] + w));
          };
          if (dg <= kRowSumLong)
            for (uint32_t j = sub; j < dg; j += 4 * G) {       // four entries in flight
              uint32_t b[4];
              float w[4];
#pragma unroll
              for (int k = 0; k < 4; ++k) {
                const bool in = j + k * G < dg;
                b[k] = in ? (uint32_t)R.in_b[lo + j + k * G] : 0xffffffffu;
                w[k] = in ? R.in_w[lo + j + k * G] : 0.f;
              }
#pragma unroll
              for (int k = 0; k < 4; ++k) take(acc, b[k], w[k]);
            }
          unsigned big = __ballot_sync(0xffffffffu, sub == 0 && dg > kRowSumLong);
          while (big) {
            const int src = __ffs(big) - 1;
            big &= big - 1;
            const uint32_t L = __shfl_sync(0xffffffffu, lo, src), N = __shfl_sync(0xffffffffu, dg, src);
            A part = Op::identity();
            for (uint32_t j = lane; j < N; j += 32) take(part, (uint32_t)R.in_b[L + j], R.in_w[L + j]);
#pragma unroll
            for (int s = 16; s; s >>= 1) part = Op::combine(part, shfl_down(part, s));
            part = shfl_idx(part, 0);
            if ((int)lane == src) acc = Op::combine(acc, part);
          }
        }
#pragma unroll
        for (int s = G / 2; s; s >>= 1) acc = Op::combine(acc, shfl_down(acc, s));      // lanes past the group bring garbage to lanes other than its first
        if (mine && sub == 0) {
          const float v = Op::lower(acc);
          const uint32_t bit = 1u << (c & 31);
          dn[c] = v;
          if (atomicOr(pres + (c >> 5), bit) & bit) sum[c] = Op::lower(Op::combine(Op::lift(sum[c]), Op::lift(v)));
          else { sum[c] = v; ++fresh; }
        }
      }
      __syncthreads();
      // Delta' is Delta now
      { float* t = d; d = dn; dn = t; uint16_t* l = list; list = next; next = l; uint32_t* h = has; has = mark; mark = spare; spare = h; }
      nd = nt;
    }
    rounds_seen = max(rounds_seen, rounds);
    __syncthreads();
    for (uint32_t i = threadIdx.x; i < S; i += kRowSumBlock) {
      int32_t v = kMirrorEmptyMin;
      if ((pres[i >> 5] >> (i & 31)) & 1u) { const float t = sum[i]; v = isnan(t) ? 0x7fc00000 : f2ord(t); }   // never the empty marker
      P.table[base + i] = v;
    }
    __syncthreads();
  }
#pragma unroll
  for (int s = 16; s; s >>= 1) cand += __shfl_down_sync(0xffffffffu, cand, s);
  fresh = __reduce_add_sync(0xffffffffu, fresh);
  if (lane == 0) {
    if (cand) atomicAdd(P.totals + kRsCandidates, cand);
    if (fresh) atomicAdd(P.totals + kRsNew, (unsigned long long)fresh);
  }
  if (threadIdx.x == 0) {
    if (uniq) atomicAdd(P.totals + kRsUnique, uniq);
    if (rounds_seen) atomicMax(P.totals + kRsRounds, (unsigned long long)rounds_seen);
    if (capped) atomicMax(P.totals + kRsCapped, 1ull);
  }
}

}  // namespace xlog
