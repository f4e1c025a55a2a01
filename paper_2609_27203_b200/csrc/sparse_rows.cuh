// Row-local fixpoint of  h(a, c) :- h(a, b), r(b, c)  over a max / min semiring when the values of c are too many for a dense
// row in shared memory (row_fixpoint.cuh) but the rows themselves are short: ancestors in a forest, transitive closure of a
// sparse acyclic graph, any closure whose tuples per first column are few.
//
// The rounds of one a are independent of every other a's (row_fixpoint.cuh says why), so after the seed round a group of G
// lanes takes a value of a and runs that row's rounds to the end on an open-addressed hash table of T slots in shared
// memory: delta list with the tags set aside, candidates laid out in a line per G delta rows, one atomic max / min per
// candidate.  The groups of a warp run their rounds in lockstep, each at its own row; a group that finishes writes the row to
// a staging area and takes the next one.  A row of more tuples than its table has slots is left alone at the first candidate that finds
// no room and its a queued for the next launch, with longer tables and wider groups.  The rows that outgrow the last tier are few:
// the stratum goes on with them alone, round by round, and the finished rows join them at its end (k_sparse_keep, k_sparse_take).
// A first tier in which every eighth row outgrows its table (a second in which every 64th does), or a full staging area, sets
// the status word, and the stratum goes on as if nothing had been tried (the relation and its delta are only read here).
//
// What bounds it: instruction issue (half of the slots) and the latency of one dependent L2 read per row and round, over as
// many rows as shared memory holds at a time.  300,000 rows of 17 tuples and 13 rounds on average (5.06 M tuples, 28 rounds):
// 7.22 ms on the sorting route, 0.89 ms here, of which 0.47 in the first tier and 0.15 in the second (5 % of the rows).
// Rows of every length (the descendants in such forests, ms, sorting route or mirror / here): 9,000 nodes 2.80 / 3.16, 60,000 2.92 /
// 4.18, 300,000 6.64 / 7.70, a node in 1,024 going on alone for all of the rounds; one row of 1,500 tuples that is done in two
// rounds among 200,000: 2.63 / 0.42.
// r is therefore read through 16-byte entries (c, tag, where c's own run begins, its length), so that a round needs no
// look-up of offsets; a row's first key comes with its record, so that taking a row needs no chain of reads either; and rows
// leave unordered (k_sparse_emit ranks them, at full occupancy).  See the tiers in host_mirror_rows.cuh.
#pragma once
#include "common.cuh"
#include "join.cuh"

namespace xlog {

constexpr int kSparseBlock = 256;
constexpr uint32_t kSparseStage = 256;           // staging places a warp reserves at a time, or more if its rows need more

// Control words of the launches.
enum { kSpCandidates = 0, kSpUnique = 1, kSpChanged = 2, kSpNew = 3, kSpRounds = 4, kSpCapped = 5, kSpStatus = 6, kSpStaged = 7, kSpQueued = 8,
       kSpTicket = 11, kSpTotals = 14 };          // kSpQueued / kSpTicket: one word per tier

struct SparseRows {
  const void* keys;                  // the relation after the seed round (K, ascending: a << c_bits | c) and its tags
  const float* tags;
  const void* dkeys;                 // the seed round's delta, a subset of it
  const float* dtags;
  const uint4* rec;                  // per a: first and one past the last entry in the relation, its first c and tag bits
  const uint2* rec_run;              // and where that c's run of r begins, its length
  const uint2* drec;                 // per a: first and one past the last entry in the delta (null: the delta is the relation)
  uint32_t n_rows;
  int c_bits;
  uint32_t z_max;                    // largest value the head's second column may take
  uint32_t max_rounds;
  const uint32_t* off;               // r's offsets over its probed column
  uint32_t domain;
  const uint4* adj;                  // per row of r, in index order: c, tag bits, where c's run begins, its length
  uint32_t* row_pos;                 // out, per a: where its row starts in the staging area, and its length
  uint32_t* row_len;
  uint32_t* st_c;                    // staging area: c and tag
  float* st_t;
  uint32_t st_cap;
  const uint32_t* rows_in;           // the a to do (null: all n_rows), their number (at most max_in) in totals[kSpQueued + tier - 1]
  uint32_t max_in;
  uint32_t* rows_out;                // the a whose rows outgrew the table
  int tier;
  uint32_t max_queued;               // more rows than this in rows_out: give up
  unsigned long long* totals;
  uint32_t* err;
};

template <int T> struct __align__(16) SparseRow {
  uint32_t hkey[T];                  // hash table: c (kSparseEmpty: free), order-mapped tag
  int32_t hval[T];
  uint2 hrun[T];                     // r's run of c: first row, length
  float dtag[T];                     // tags of the delta, by place in the list
  uint16_t list[T];                  // slots of the delta
  uint32_t occ[T / 32], seen[T / 32], chg[T / 32];      // slots in use / hit by a candidate / changed in the running round
  uint32_t pad;                      // rows of neighbouring groups start in different banks
};
constexpr uint32_t kSparseEmpty = 0xffffffffu;   // no c: keys are below 2^31

// adj, see SparseRows
static __global__ void __launch_bounds__(256) k_sparse_adj(const int32_t* __restrict__ z, const float* __restrict__ w, uint32_t n, const uint32_t* __restrict__ off,
                                                           uint32_t domain, uint4* __restrict__ adj) {
  for (uint32_t i = blockIdx.x * blockDim.x + threadIdx.x; i < n; i += gridDim.x * blockDim.x) {
    const uint32_t c = (uint32_t)z[i];
    uint32_t lo = 0, hi = 0;
    if (c < domain) { lo = off[c]; hi = off[c + 1]; }
    adj[i] = make_uint4(c, __float_as_uint(w[i]), lo, hi - lo);
  }
}

// Row records of a sorted list of keys: rec (zero on entry) and run, or, where only the bounds are wanted, bounds (zero on entry).
template <typename K>
__global__ void __launch_bounds__(256) k_sparse_records(const K* __restrict__ keys, const float* __restrict__ tags, uint32_t n, int c_bits, const uint32_t* __restrict__ off,
                                                        uint32_t domain, uint4* __restrict__ rec, uint2* __restrict__ run, uint2* __restrict__ bounds) {
  for (uint32_t i = blockIdx.x * blockDim.x + threadIdx.x; i < n; i += gridDim.x * blockDim.x) {
    const K k = keys[i];
    const uint32_t a = (uint32_t)(k >> c_bits);
    const bool head = i == 0 || (uint32_t)(keys[i - 1] >> c_bits) != a, tail = i + 1 == n || (uint32_t)(keys[i + 1] >> c_bits) != a;
    if (bounds) {
      if (head) bounds[a].x = i;
      if (tail) bounds[a].y = i + 1;
      continue;
    }
    if (head) {
      const uint32_t c = (uint32_t)(k & (((K)1 << c_bits) - 1));
      uint32_t lo = 0, hi = 0;
      if (c < domain) { lo = off[c]; hi = off[c + 1]; }
      rec[a].x = i; rec[a].z = c; rec[a].w = __float_as_uint(tags[i]);
      run[a] = make_uint2(lo, hi - lo);
    }
    if (tail) rec[a].y = i + 1;
  }
}

// Slot of c in the table, inserted if absent (is_new); T if there is no room.  Tables fill to the last slot; in the longer ones the
// steps grow by one (1 + 2 + ... meets every slot of a power of two), or the last keys of a row would each look at most of the
// table.
template <int T>
__device__ __forceinline__ uint32_t sparse_slot(SparseRow<T>& R, uint32_t c, bool& is_new) {
  constexpr int LOG = T == 32 ? 5 : T == 64 ? 6 : T == 128 ? 7 : T == 256 ? 8 : T == 512 ? 9 : 10;
  static_assert((1 << LOG) == T, "table size");
  uint32_t h = (c * 0x9E3779B1u) >> (32 - LOG);
  is_new = false;
#pragma unroll 1
  for (int probe = 0; probe < T; ++probe) {
    uint32_t k = *reinterpret_cast<volatile uint32_t*>(&R.hkey[h]);
    if (k == kSparseEmpty) {
      k = atomicCAS(&R.hkey[h], kSparseEmpty, c);
      if (k == kSparseEmpty) { is_new = true; return h; }
    }
    if (k == c) return h;
    h = (h + (T <= 32 ? 1 : probe + 1)) & (T - 1);
  }
  return T;
}

template <typename K, int SINK, int G, int T>
__global__ void __launch_bounds__(kSparseBlock) k_sparse_rows(const __grid_constant__ SparseRows P) {
  constexpr int32_t kEmptyVal = SINK == kSinkMin ? kMirrorEmptyMin : kMirrorEmptyMax;
  constexpr int B = T / G;                         // slots per lane where the bitmaps are read
  static_assert(B <= 32 && 32 % B == 0, "a lane's slots lie in one bitmap word");
  constexpr uint32_t kMaskB = B == 32 ? 0xffffffffu : (1u << (B & 31)) - 1u;
  constexpr unsigned kGroups = 32 / G;
  constexpr int kBatch = kGroups >= 4 ? 4 : 1;     // groups that leave together
  extern __shared__ __align__(16) unsigned char sp_smem[];
  SparseRow<T>& R = reinterpret_cast<SparseRow<T>*>(sp_smem)[threadIdx.x / G];
  const unsigned lane = lane_id(), sub = lane % G, grp = lane / G;
  const unsigned gmask = (G == 32 ? 0xffffffffu : ((1u << (G & 31)) - 1u)) << (grp * G);
  const uint32_t bword = sub * B / 32, bshift = sub * B % 32;
  const K* keys = (const K*)P.keys;
  const K* dkeys = (const K*)P.dkeys;
  const K cmask = ((K)1 << P.c_bits) - 1;
  const uint32_t n_todo = P.rows_in ? min((uint32_t)P.totals[kSpQueued + P.tier - 1], P.max_in) : P.n_rows;
  // rows a warp draws at a time: one a group, fewer where there are few (neighbouring rows may all be long)
  const uint32_t per_draw = max(1u, min(kGroups, n_todo / (gridDim.x * (kSparseBlock / 32))));
  unsigned long long* const queued = P.totals + kSpQueued + P.tier;
  unsigned long long cand = 0;
  uint32_t uniq = 0, n_changed = 0, n_new = 0, max_rounds_seen = 0, capped = 0;
  uint32_t chunk = 0, chunk_end = 0;               // rows the warp has drawn and not begun (uniform)
  uint32_t stage = 0, stage_end = 0;               // staging room the warp holds (uniform)
  bool dry = false;                                // the warp's supply has run out (uniform)
  bool active = false, more = false, outgrown = false;      // the group has a row; the row has a delta; it does not fit the table
  uint32_t a = 0, rounds = 0, turns = 0;
  bool have_next = false;                          // the group has drawn the row after this one
  uint32_t next_a = 0;
  uint4 next_rec = make_uint4(0, 0, 0, 0);
  uint2 next_run = make_uint2(0, 0), next_dr = make_uint2(0, 0);
  uint32_t row_cand = 0, row_uniq = 0, row_changed = 0, row_new = 0;      // of the running row: dropped if it outgrows the table
  for (;;) {
    const bool cap = active && more && !outgrown && rounds >= P.max_rounds;
    const bool waits = !active || !more || outgrown || cap;      // nothing to do but leave, or take a row
    // every turn either runs a round of some row or lets a row go or come: the loop ends with the rows (`turns` only guards that)
    const unsigned waiting = __ballot_sync(0xffffffffu, waits && (active || have_next || !dry) && sub == 0);
    const bool running = __any_sync(0xffffffffu, !waits);
    if (!running && (waiting == 0u || ++turns > 4u * n_todo + 64u)) {
      if (waiting && lane == 0) { atomicOr(P.err, kErrInternal); atomicExch(P.totals + kSpStatus, 3ull); }
      break;
    }
    if ((int)__popc(waiting) >= kBatch || !running) {
      // ---- rows that are done, outgrown or capped leave
      const bool emit = active && waits && !outgrown && !cap;
      if (__any_sync(0xffffffffu, active && waits)) {
        if (cap) capped = 1;
        const uint32_t m = emit ? (R.occ[bword] >> bshift) & kMaskB : 0u;
        const uint32_t mine = __popc(m);
        // staging room: the groups of the warp that emit now, one after the other
        uint32_t incl = mine;
#pragma unroll
        for (int d = 1; d < 32; d <<= 1) { const uint32_t o = __shfl_up_sync(0xffffffffu, incl, d); if ((int)lane >= d) incl += o; }
        const uint32_t need = __shfl_sync(0xffffffffu, incl, 31);
        if (need > stage_end - stage) {
          const uint32_t take = max(need, kSparseStage);
          uint32_t got = 0;
          if (lane == 0) {
            const unsigned long long g0 = atomicAdd(P.totals + kSpStaged, (unsigned long long)take);
            got = g0 + take <= P.st_cap ? (uint32_t)g0 : kSparseEmpty;
            if (got == kSparseEmpty) atomicExch(P.totals + kSpStatus, 2ull);
          }
          stage = __shfl_sync(0xffffffffu, got, 0);
          stage_end = stage == kSparseEmpty ? kSparseEmpty : stage + take;
        }
        const bool room = stage != kSparseEmpty;
        const uint32_t first = __shfl_sync(0xffffffffu, incl - mine, grp * G), last = __shfl_sync(0xffffffffu, incl, grp * G + G - 1);
        if (emit && room) {
          uint32_t at = stage + incl - mine;
          for (uint32_t bits = m; bits; bits &= bits - 1, ++at) {
            const uint32_t s = sub * B + __ffs(bits) - 1;
            P.st_c[at] = R.hkey[s];
            P.st_t[at] = ord2f(R.hval[s]);
          }
          if (sub == 0) { P.row_pos[a] = stage + first; P.row_len[a] = last - first; }
        }
        if (room) stage += need; else { stage = stage_end = 0; }
        if (active && outgrown && sub == 0) {
          const unsigned long long q = atomicAdd(queued, 1ull);
          if (q < P.max_queued) P.rows_out[q] = a; else atomicExch(P.totals + kSpStatus, 1ull);
          P.row_len[a] = 0u;
        }
        if (emit) { max_rounds_seen = max(max_rounds_seen, rounds); cand += row_cand; uniq += row_uniq; n_changed += row_changed; n_new += row_new; }
        if (waits) active = false;
        __syncwarp();
      }
      // ---- idle groups take the row they have drawn, and draw another
      if (!dry || __any_sync(0xffffffffu, have_next && !active)) {
        if (chunk >= chunk_end && !dry) {
          uint32_t t = 0;
          if (lane == 0) {
            const bool stop = *reinterpret_cast<volatile unsigned long long*>(P.totals + kSpStatus) != 0ull;
            t = stop ? n_todo : (uint32_t)atomicAdd(P.totals + kSpTicket + P.tier, (unsigned long long)per_draw);
          }
          chunk = __shfl_sync(0xffffffffu, t, 0);
          chunk_end = min(chunk + per_draw, n_todo);
          if (chunk >= n_todo) { dry = true; chunk = chunk_end = 0; }
        }
        const unsigned idle = __ballot_sync(0xffffffffu, !active && sub == 0);
        const uint32_t mine = chunk + __popc(idle & ((1u << (grp * G)) - 1u));
        const bool fetch = !active && have_next;
        const bool draw = !active && mine < chunk_end;          // the row after the one taken now: its record is read ahead
        chunk = min(chunk + (uint32_t)__popc(idle), chunk_end);
        uint4 rec = make_uint4(0, 0, 0, 0);
        uint2 run = make_uint2(0, 0), dr = make_uint2(0, 0);
        bool fits = false;
        if (fetch) {
          a = next_a; rec = next_rec; run = next_run; dr = next_dr;
          fits = rec.y - rec.x <= (uint32_t)T;
          const uint32_t ev = (uint32_t)kEmptyVal;
          for (int i = sub; i < T / 4; i += G) {
            reinterpret_cast<uint4*>(R.hkey)[i] = make_uint4(kSparseEmpty, kSparseEmpty, kSparseEmpty, kSparseEmpty);
            reinterpret_cast<uint4*>(R.hval)[i] = make_uint4(ev, ev, ev, ev);
          }
          for (int i = sub; i < T / 32; i += G) { R.occ[i] = 0u; R.chg[i] = 0u; }
        }
        if (!active) have_next = draw;
        if (draw) {
          next_a = P.rows_in ? P.rows_in[mine] : mine;
          next_rec = P.rec[next_a];
          next_run = P.rec_run[next_a];
          next_dr = P.drec ? P.drec[next_a] : make_uint2(0, 0);
        }
        __syncwarp();
        if (fetch && fits)
          for (uint32_t i = rec.x + sub; i < rec.y; i += G) {
            const bool first = i == rec.x;
            const uint32_t c = first ? rec.z : (uint32_t)(keys[i] & cmask);
            const float t = first ? __uint_as_float(rec.w) : P.tags[i];
            uint2 r = run;
            if (!first) {
              r = make_uint2(0, 0);
              if (c < P.domain) { r.x = P.off[c]; r.y = P.off[c + 1] - r.x; }
            }
            bool is_new;
            const uint32_t s = sparse_slot<T>(R, c, is_new);
            R.hval[s] = f2ord(t);
            R.hrun[s] = r;
            atomicOr(&R.occ[s >> 5], 1u << (s & 31));
            if (!P.drec) atomicOr(&R.chg[s >> 5], 1u << (s & 31));
          }
        if (P.drec) {
          __syncwarp();
          if (fetch && fits)
            for (uint32_t i = dr.x + sub; i < dr.y; i += G) {
              bool is_new;
              const uint32_t s = sparse_slot<T>(R, (uint32_t)(dkeys[i] & cmask), is_new);
              atomicOr(&R.chg[s >> 5], 1u << (s & 31));
            }
        }
        if (fetch) {
          rounds = 0;
          row_cand = row_uniq = row_changed = row_new = 0;
          more = P.drec ? dr.y != dr.x : rec.y != rec.x;
          outgrown = !fits;
          active = true;
        }
        __syncwarp();
      }
    }
    // ---- one round of every group that has a delta: its list, in order of the slots
    const bool go = active && more && !outgrown && rounds < P.max_rounds;
    if (!__any_sync(0xffffffffu, go)) continue;
    const uint32_t dm = go ? (R.chg[bword] >> bshift) & kMaskB : 0u;
    uint32_t incl = __popc(dm);
#pragma unroll
    for (int d = 1; d < G; d <<= 1) { const uint32_t o = __shfl_up_sync(0xffffffffu, incl, d, G); if ((int)sub >= d) incl += o; }
    const uint32_t nd = __shfl_sync(0xffffffffu, incl, G - 1, G);
    const uint32_t occ_before = go ? __popc((R.occ[bword] >> bshift) & kMaskB) : 0u;
    {
      uint32_t at = incl - __popc(dm);
      for (uint32_t bits = dm; bits; bits &= bits - 1, ++at) {
        const uint32_t s = sub * B + __ffs(bits) - 1;
        R.list[at] = (uint16_t)s;
        R.dtag[at] = ord2f(R.hval[s]);
      }
    }
    __syncwarp();
    if (go) for (int i = sub; i < T / 32; i += G) { R.seen[i] = 0u; R.chg[i] = 0u; }
    __syncwarp();
    bool full = false, stop = false;                         // stop: some lane of the group found the table full; the round's rest is not looked at
    for (uint32_t r0 = 0; __any_sync(0xffffffffu, go && !stop && r0 < nd); r0 += G) {
      uint32_t lo = 0, dg = 0;
      float t = 0.f;
      if (go && !stop && r0 + sub < nd) {
        const uint2 run = R.hrun[R.list[r0 + sub]];
        t = R.dtag[r0 + sub];
        lo = run.x; dg = run.y;
      }
      uint32_t end = dg;
#pragma unroll
      for (int d = 1; d < G; d <<= 1) { const uint32_t o = __shfl_up_sync(0xffffffffu, end, d, G); if ((int)sub >= d) end += o; }
      const uint32_t total = __shfl_sync(0xffffffffu, end, G - 1, G);
      row_cand += dg;
      for (uint32_t p0 = 0; __any_sync(0xffffffffu, !stop && p0 < total); p0 += G) {
        const uint32_t p = p0 + sub;
        uint32_t owner = 0;                                  // first lane of the group whose inclusive prefix exceeds p
#pragma unroll
        for (int d = G / 2; d; d >>= 1) { const uint32_t v = __shfl_sync(0xffffffffu, end, owner + d - 1, G); if (v <= p) owner += d; }
        const uint32_t from = __shfl_sync(0xffffffffu, lo + dg - end, owner, G);        // the owner's run, less the candidates before it
        const float ot = __shfl_sync(0xffffffffu, t, owner, G);
        if (!stop && p < total) {
          const uint4 q = P.adj[from + p];
          const uint32_t c = q.x;
          const int32_t v = f2ord(ot + __uint_as_float(q.y));
          if (c > P.z_max) atomicOr(P.err, kErrHeadRange);
          else {
            bool is_new;
            const uint32_t s = sparse_slot<T>(R, c, is_new);
            if (s == (uint32_t)T) full = true;
            else {
              const uint32_t bit = 1u << (s & 31);
              if (is_new) { R.hrun[s] = make_uint2(q.z, q.w); atomicOr(&R.occ[s >> 5], bit); }
              atomicOr(&R.seen[s >> 5], bit);
              const int32_t old = SINK == kSinkMin ? atomicMin(&R.hval[s], v) : atomicMax(&R.hval[s], v);
              if (SINK == kSinkMin ? v < old : v > old) atomicOr(&R.chg[s >> 5], bit);
            }
          }
        }
        // once one candidate has found no room none is looked for any more
        const unsigned none = __ballot_sync(0xffffffffu, full);      // by every lane, stopped or not
        stop = (none & gmask) != 0u;
      }
    }
    __syncwarp();
    const uint32_t cm = go ? (R.chg[bword] >> bshift) & kMaskB : 0u;
    const unsigned any_full = __ballot_sync(0xffffffffu, full), any_more = __ballot_sync(0xffffffffu, cm != 0u);
    if (go) {
      outgrown = (any_full & gmask) != 0u;
      more = (any_more & gmask) != 0u;
      ++rounds;
      row_uniq += __popc((R.seen[bword] >> bshift) & kMaskB);
      row_changed += __popc(cm);
      row_new += __popc((R.occ[bword] >> bshift) & kMaskB) - occ_before;
    }
  }
#pragma unroll
  for (int s = 16; s; s >>= 1) cand += __shfl_down_sync(0xffffffffu, cand, s);
  uniq = __reduce_add_sync(0xffffffffu, uniq); n_changed = __reduce_add_sync(0xffffffffu, n_changed); n_new = __reduce_add_sync(0xffffffffu, n_new);
  max_rounds_seen = __reduce_max_sync(0xffffffffu, max_rounds_seen); capped = __reduce_or_sync(0xffffffffu, capped);
  if (lane == 0) {
    if (cand) atomicAdd(P.totals + kSpCandidates, cand);
    if (uniq) atomicAdd(P.totals + kSpUnique, (unsigned long long)uniq);
    if (n_changed) atomicAdd(P.totals + kSpChanged, (unsigned long long)n_changed);
    if (n_new) atomicAdd(P.totals + kSpNew, (unsigned long long)n_new);
    if (max_rounds_seen) atomicMax(P.totals + kSpRounds, (unsigned long long)max_rounds_seen);
    if (capped) atomicMax(P.totals + kSpCapped, 1ull);
  }
}

constexpr uint32_t kSparseLongest = 1024;       // slots of the last tier's table

// The staged rows to their places, in order of c: G lanes per row, off = exclusive scan of row_len.  A key's place is the number
// of smaller keys in its row: rows of up to 32 keys are ordered in registers by G lanes, longer ones by the warp in shared
// memory; both are written in line.
template <typename K>
__global__ void __launch_bounds__(256) k_sparse_emit(const uint32_t* __restrict__ row_pos, const uint32_t* __restrict__ row_len, const uint32_t* __restrict__ off,
                                                     uint32_t n_rows, int c_bits, const uint32_t* __restrict__ st_c, const float* __restrict__ st_t,
                                                     K* __restrict__ keys, float* __restrict__ tags) {
  constexpr int G = 8, R = 4;
  __shared__ uint2 s_row[256 / G][G * R + 1];
  __shared__ uint32_t s_long[256 / 32][kSparseLongest];
  uint2* row = s_row[threadIdx.x / G];
  uint32_t* lrow = s_long[warp_id()];
  const uint32_t sub = threadIdx.x % G;
  const uint32_t stride = gridDim.x * blockDim.x / G, last = (n_rows + stride - 1) / stride * stride;      // every lane of a warp takes part in every step
  for (uint32_t a = (blockIdx.x * blockDim.x + threadIdx.x) / G; a < last; a += stride) {
    const uint32_t n = a < n_rows ? row_len[a] : 0u, at = n ? row_pos[a] : 0u, to = n ? off[a] : 0u;
    const bool small = n <= G * R;
    uint32_t c[R], rank[R];
    float t[R];
#pragma unroll
    for (int r = 0; r < R; ++r) {
      const bool in = small && sub + r * G < n;
      c[r] = in ? st_c[at + sub + r * G] : 0xffffffffu;
      t[r] = in ? st_t[at + sub + r * G] : 0.f;
      rank[r] = 0;
    }
#pragma unroll
    for (int r = 0; r < R; ++r)
      if (__any_sync(0xffffffffu, small && r * G < n))
#pragma unroll
        for (int j = 0; j < G; ++j) {
          const uint32_t o = __shfl_sync(0xffffffffu, c[r], j, G);
#pragma unroll
          for (int q = 0; q < R; ++q) rank[q] += o < c[q] ? 1u : 0u;
        }
#pragma unroll
    for (int r = 0; r < R; ++r) if (small && sub + r * G < n) row[rank[r]] = make_uint2(c[r], __float_as_uint(t[r]));
    __syncwarp();
    if (small)
      for (uint32_t i = sub; i < n; i += G) { const uint2 e = row[i]; keys[to + i] = ((K)a << c_bits) | (K)e.x; tags[to + i] = __uint_as_float(e.y); }
    for (unsigned todo = __ballot_sync(0xffffffffu, !small && sub == 0); todo; todo &= todo - 1) {
      const int src = __ffs(todo) - 1;
      const uint32_t N = min(__shfl_sync(0xffffffffu, n, src), kSparseLongest), A = __shfl_sync(0xffffffffu, a, src), AT = __shfl_sync(0xffffffffu, at, src),
                     TO = __shfl_sync(0xffffffffu, to, src);
      __syncwarp();
      for (uint32_t i = lane_id(); i < N; i += 32) lrow[i] = st_c[AT + i];
      __syncwarp();
      for (uint32_t i = lane_id(); i < N; i += 32) {
        const uint32_t ci = lrow[i];
        uint32_t k = 0;
#pragma unroll 8
        for (uint32_t j = 0; j < N; ++j) k += lrow[j] < ci ? 1u : 0u;
        keys[TO + k] = ((K)A << c_bits) | (K)ci;
        tags[TO + k] = st_t[AT + i];
      }
    }
    __syncwarp();
  }
}

// The rows (of first column) on a list, marked; the tuples of marked rows in a list of keys, flagged; and copied to the places that
// a scan of the flags gives.
static __global__ void __launch_bounds__(256) k_sparse_mark(const uint32_t* __restrict__ rows, uint32_t n, uint32_t* __restrict__ mark) {
  for (uint32_t i = blockIdx.x * blockDim.x + threadIdx.x; i < n; i += gridDim.x * blockDim.x) mark[rows[i]] = 1u;
}
template <typename K>
__global__ void __launch_bounds__(256) k_sparse_keep(const K* __restrict__ keys, uint32_t n, int c_bits, const uint32_t* __restrict__ mark, uint32_t* __restrict__ flag) {
  for (uint32_t i = blockIdx.x * blockDim.x + threadIdx.x; i <= n; i += gridDim.x * blockDim.x) flag[i] = i < n ? mark[(uint32_t)(keys[i] >> c_bits)] : 0u;
}
template <typename K>
__global__ void __launch_bounds__(256) k_sparse_take(const K* __restrict__ keys, const float* __restrict__ tags, uint32_t n, const uint32_t* __restrict__ at,
                                                     K* __restrict__ out_keys, float* __restrict__ out_tags) {
  for (uint32_t i = blockIdx.x * blockDim.x + threadIdx.x; i < n; i += gridDim.x * blockDim.x)
    if (at[i] != at[i + 1]) { out_keys[at[i]] = keys[i]; out_tags[at[i]] = tags[i]; }
}

}  // namespace xlog
