// Row-local fixpoint for the rule shape  h(a, c) :- h(a, b), r(b, c)  (transitive closure, multi-source reachability)
// over a max / min semiring, when one value of a owns few enough keys to live in shared memory.
//
// The rule never changes a: the tuples of one a are derived from the tuples of that a and from r alone.  The rounds of
// Algorithm 1 therefore fall apart into one independent sequence of rounds per value of a, and the whole fixpoint of the
// stratum is ONE launch without any grid-wide step: a block takes a value of a, loads its row of the tag mirror (one slot
// per value of c, in the relation's own key order) into shared memory and runs that row's rounds there - delta list from
// the changed bits, tags of the delta set aside before the join (the join lowers the row while other warps still read
// the delta), candidates applied with shared-memory atomics, new keys settled against the row's bitmap of present keys -
// until the row's delta is empty, then writes the row back.  Round r of a row is exactly round r of the global
// semi-naive loop restricted to that a, so the counters add up to the global ones: candidates, new and improved keys are
// sums over rows and rounds, and the number of global rounds is the largest number of rounds any row needed.
//
// The same holds for several mutually recursive heads whose rules all have this shape with one shared first column,
//   h_i(a, c) :- h_j(a, b), r(b, c)      (odd / even walks),
// as long as the heads share one key layout: a block then holds one row per head, a round closes every head's changed
// bits into its delta first and then applies every rule from its source head's delta to its target head's row.
//
// Bound by the latency of a round (two barriers, a lookup and a candidate read one after the other) and by how many rows an SM
// holds.  Closing a round a lane per bit and laying the candidates out warp by warp, without a barrier: 1,000 nodes and 4,000
// edges 122 -> 97 us, 300 nodes 43 -> 35 us, 2,400 nodes 536 -> 392 us (before: a thread per bitmap word, one prefix over
// the whole block, ten steps of search per candidate).  Registers for 6 blocks an SM: with as many as the compiler
// likes 134, 31 and 567 us; for 8 blocks 88, 37 and 407 us, which is taken where it saves a wave of rows.
#pragma once
#include "common.cuh"
#include "join.cuh"

namespace xlog {

constexpr int kRowMaxBits = 13;                  // keys per value of a: at most 8192 (row, tags set aside and delta list: 80 KB)
constexpr int kRowBlock = 256;
constexpr int kRowBlocks = 6, kRowBlocksMany = 8;       // blocks an SM of one head's kernel is built for
constexpr int kRowUnroll = 2;                    // candidates a lane looks up at a time

// Totals of the launch, in the control words.
enum { kRowCandidates = 0, kRowChanged = 1, kRowNew = 2, kRowRounds = 3, kRowCapped = 4, kRowTotals = 5 };

constexpr int kRowMaxHeads = 4, kRowMaxRules = 8;

struct RowHead {
  int32_t* table;                  // tag mirror in the relation's key order: slot = a << c_bits | c
  uint32_t* changed;               // changed bitmap: what the seed round derived; left all zero
  uint32_t* present;               // keys the relation holds
  int is_max;                      // oplus: max (1) or min (0)
};

struct RowRule {                   // heads[dst](a, c) :- heads[src](a, b), r(b, c)
  int src, dst;
  const uint32_t* off;             // r's offsets over its probed column
  uint32_t domain;                 // off has domain + 1 entries
  const int32_t* z;                // r's other column, in index order
  const float* w;                  // its tags
};

struct RowFix {
  RowHead heads[kRowMaxHeads];
  RowRule rules[kRowMaxRules];
  int n_heads, n_rules;
  uint32_t n_rows;                 // values of a
  int c_bits;                      // log2 of the slots per row (at least 5: a row owns whole bitmap words), the same for every head
  uint32_t z_max;                  // largest value a head's second column may take
  uint32_t max_rounds;             // rounds a row may run before the iteration cap is reached
  unsigned long long* totals;      // kRowTotals counters, zeroed by the caller
  uint32_t* err;
};

// per head: row tags (4 B per slot), delta tags (4 B), delta slots (2 B), changed and present bits
inline size_t row_fix_smem(int c_bits, int n_heads) { return (size_t)n_heads * (((size_t)10 << c_bits) + ((size_t)2 << c_bits) / 8); }

template <int NH, int BLOCKS>
__global__ void __launch_bounds__(kRowBlock, BLOCKS) k_row_fixpoint(const __grid_constant__ RowFix P) {
  extern __shared__ uint32_t row_smem[];
  __shared__ uint32_t s_nd[2][NH];                                   // delta rows of every head in the running round, and in the next
  const uint32_t S = 1u << P.c_bits, W = S >> 5;
  const uint32_t per_head = 2 * S + 2 * W + S / 2;                   // words of shared memory per head
  const unsigned lane = lane_id();
  unsigned long long cand = 0;                    // the warp's
  uint32_t n_changed = 0, n_new = 0, max_rounds_seen = 0, capped = 0;
  for (uint32_t a = blockIdx.x; a < P.n_rows; a += gridDim.x) {
    const size_t base = (size_t)a << P.c_bits;
    uint32_t any = 0;
#pragma unroll
    for (int h = 0; h < NH; ++h) {
      uint32_t* chg = row_smem + h * per_head + 2 * S;
      uint32_t* pres = chg + W;
      for (uint32_t i = threadIdx.x; i < W; i += kRowBlock) {
        const uint32_t m = P.heads[h].changed[(base >> 5) + i];
        chg[i] = m;
        pres[i] = P.heads[h].present[(base >> 5) + i];
        any |= m;
      }
    }
    if (__syncthreads_or(any != 0u) == 0) continue;                            // nothing of this a changed in the seed round
#pragma unroll
    for (int h = 0; h < NH; ++h) {
      int32_t* row = reinterpret_cast<int32_t*>(row_smem + h * per_head);
      for (uint32_t i = threadIdx.x; i < S; i += kRowBlock) row[i] = P.heads[h].table[base + i];
      for (uint32_t i = threadIdx.x; i < W; i += kRowBlock) P.heads[h].changed[(base >> 5) + i] = 0u;
    }
    if (threadIdx.x < 2 * NH) s_nd[threadIdx.x / NH][threadIdx.x % NH] = 0;
    __syncthreads();
    uint32_t rounds = 0;
    for (uint32_t par = 0;; par ^= 1) {
      // close the round before, head by head: its changed keys are the delta now, the new ones among them enter the relation;
      // a warp takes its share of the words, up to 32 at a time, and writes the keys of a word a lane per bit
      for (int h = 0; h < NH; ++h) {
        int32_t* row = reinterpret_cast<int32_t*>(row_smem + h * per_head);
        float* dtag = reinterpret_cast<float*>(row_smem + h * per_head + S);
        uint32_t* chg = row_smem + h * per_head + 2 * S;
        uint32_t* pres = chg + W;
        uint16_t* didx = reinterpret_cast<uint16_t*>(pres + W);
        const uint32_t share = (W + kRowBlock / 32 - 1) / (kRowBlock / 32);      // at most 32
        const uint32_t i = warp_id() * share + lane;
        const uint32_t m = lane < share && i < W ? chg[i] : 0u;
        uint32_t some = __ballot_sync(0xffffffffu, m != 0u);
        if (some == 0u) continue;
        if (m) {
          n_new += __popc(m & ~pres[i]);
          pres[i] |= m;
          chg[i] = 0u;
        }
        const uint32_t upto = warp_scan_incl((uint32_t)__popc(m));
        uint32_t first = 0;
        if (lane == 31) first = atomicAdd(&s_nd[par][h], upto);
        first = __shfl_sync(0xffffffffu, first, 31) + upto - __popc(m);
        for (; some; some &= some - 1) {
          const int src = __ffs(some) - 1;
          const uint32_t mask = __shfl_sync(0xffffffffu, m, src), at = __shfl_sync(0xffffffffu, first, src) + __popc(mask & lanemask_lt());
          if ((mask >> lane) & 1u) {
            const uint32_t slot = ((warp_id() * share + src) << 5) + lane;
            didx[at] = (uint16_t)slot;
            dtag[at] = ord2f(row[slot]);
          }
        }
      }
      __syncthreads();
      uint32_t nd_all = 0;
#pragma unroll
      for (int h = 0; h < NH; ++h) nd_all += s_nd[par][h];
      if (nd_all == 0) break;
      if (threadIdx.x < NH) s_nd[par ^ 1][threadIdx.x] = 0;
      if (threadIdx.x == 0) n_changed += nd_all;
      if (rounds >= P.max_rounds) { capped = 1; break; }
      ++rounds;
      // the joins, rule by rule: a warp takes up to 32 delta rows, a lane looks up the run of one, and the candidates of all of
      // them lie in a line over the lanes, whatever the mix of short and long runs
      for (int q = 0; q < P.n_rules; ++q) {
        const RowRule& R = P.rules[q];
        const uint32_t nd = s_nd[par][R.src], batch = min(32u, (nd + kRowBlock / 32 - 1) / (kRowBlock / 32));
        const float* dtag = reinterpret_cast<const float*>(row_smem + R.src * per_head + S);
        const uint16_t* didx = reinterpret_cast<const uint16_t*>(row_smem + R.src * per_head + 2 * S + 2 * W);
        int32_t* row = reinterpret_cast<int32_t*>(row_smem + R.dst * per_head);
        uint32_t* chg = row_smem + R.dst * per_head + 2 * S;
        const bool is_max = P.heads[R.dst].is_max != 0;
        for (uint32_t r0 = warp_id() * batch; r0 < nd; r0 += batch * (kRowBlock / 32)) {
          const uint32_t r = r0 + lane;
          uint32_t lo = 0, dg = 0;
          float t = 0.f;
          if (lane < batch && r < nd) {
            const uint32_t b = didx[r];
            t = dtag[r];
            if (b < R.domain) { lo = R.off[b]; dg = R.off[b + 1] - lo; }
          }
          const uint32_t incl = warp_scan_incl(dg), total = __shfl_sync(0xffffffffu, incl, 31), from = lo + dg - incl;
          cand += total;
          for (uint32_t p0 = 0; p0 < total; p0 += 32 * kRowUnroll) {
            uint32_t c[kRowUnroll];
            float w[kRowUnroll];
#pragma unroll
            for (int u = 0; u < kRowUnroll; ++u) {
              const uint32_t p = p0 + u * 32 + lane;
              uint32_t owner = 0;                // first row whose inclusive prefix exceeds p
#pragma unroll
              for (int d = 16; d; d >>= 1) { const uint32_t x = __shfl_sync(0xffffffffu, incl, owner + d - 1); if (x <= p) owner += d; }
              const uint32_t e = __shfl_sync(0xffffffffu, from, owner) + p;
              w[u] = __shfl_sync(0xffffffffu, t, owner);
              c[u] = 0xffffffffu;
              if (p < total) { c[u] = (uint32_t)R.z[e]; w[u] += R.w[e]; }
            }
#pragma unroll
            for (int u = 0; u < kRowUnroll; ++u) {
              if (c[u] == 0xffffffffu) continue;
              if (c[u] > P.z_max || c[u] >= S) { atomicOr(P.err, kErrHeadRange); continue; }
              const int32_t v = f2ord(w[u]);
              const int32_t cur = row[c[u]];
              if (is_max ? v > cur : v < cur) {
                if (is_max) atomicMax(row + c[u], v); else atomicMin(row + c[u], v);
                atomicOr(chg + (c[u] >> 5), 1u << (c[u] & 31));
              }
            }
          }
        }
      }
      __syncthreads();
    }
    max_rounds_seen = max(max_rounds_seen, rounds);
    __syncthreads();
#pragma unroll
    for (int h = 0; h < NH; ++h) {
      const int32_t* row = reinterpret_cast<const int32_t*>(row_smem + h * per_head);
      const uint32_t* pres = row_smem + h * per_head + 2 * S + W;
      for (uint32_t i = threadIdx.x; i < S; i += kRowBlock) P.heads[h].table[base + i] = row[i];
      for (uint32_t i = threadIdx.x; i < W; i += kRowBlock) P.heads[h].present[(base >> 5) + i] = pres[i];
    }
    __syncthreads();
  }
  // totals: per warp, then one atomic per counter
  n_new = __reduce_add_sync(0xffffffffu, n_new);
  if (lane == 0 && n_new) atomicAdd(P.totals + kRowNew, (unsigned long long)n_new);
  if (lane == 0 && cand) atomicAdd(P.totals + kRowCandidates, cand);
  if (threadIdx.x == 0) {
    if (n_changed) atomicAdd(P.totals + kRowChanged, (unsigned long long)n_changed);
    if (max_rounds_seen) atomicMax(P.totals + kRowRounds, (unsigned long long)max_rounds_seen);
    if (capped) atomicMax(P.totals + kRowCapped, 1ull);
  }
}

}  // namespace xlog
