// Small resident rounds (resident.cuh) run inside one thread-block cluster: the tag mirror of a key space of up to 2^17 keys fits the
// shared memory of eight SMs, so rounds whose deltas are small need no kernel boundary, no L2 atomics and no list in memory.
//
// CTA `owner(key)` of the cluster holds a key's slot twice, as of the start of the running round (read by every candidate's
// check) and as of its end (improved by atomics over distributed shared memory); the two swap roles each round, and the owner
// brings a slot that changed in the round before up to date when it takes its delta row.  One cluster barrier per round: after
// it a CTA turns its changed bits into its part of the next delta, in its own shared memory.  Round r here is round r of the
// resident loop; the books kept in the state block are the same.
//
// The kernel is the first node of the loop body: it takes over when the delta is small (at most kRcMaxRows rows and kRcMaxCand
// candidates) and runs rounds until the relation is finished or the next round would not be; it then writes the mirror and the
// changed bits back, and the body's join (nothing to do) and emit kernels close that round and go on grid-wide.  Eight SMs have a
// twentieth of the device's lanes, so candidates are what counts: a CTA may have kRcMaxCta of them in a round.  With rows of at
// most kRcMaxRun matches (the host looks, see host_mirror.cuh) the rows bound them well enough while they are few; above, the
// degrees of the changed keys are added up before their round is begun, at the price of one more barrier.
//
// What bounds it: a chain per round of two L2 reads (offsets, then columns; the barrier's acquire empties L1), one
// distributed-shared-memory read, the barrier (its release waits for the atomics under way) and the list: about 3 us on a grid
// of 90,601 nodes (595 rounds of 1,200 rows), where the two grid-wide launches took 12: 7.6 -> 1.8 ms per query; a grid of 1,600
// nodes 2.2 us a round.  Tried and dropped: an mbarrier per CTA instead of the hardware barrier (its cluster-scope release
// costs more than the barrier's), rows listed per warp without a block barrier (uneven warps), 1,024 threads.
#pragma once
#include <cuda_runtime.h>

#include "common.cuh"
#include "join.cuh"
#include "resident.cuh"

namespace xlog {

constexpr int kRcCtas = 8, kRcCtasLog = 3;       // the largest portable cluster
constexpr int kRcBlock = 512;                    // 1024: 3 % faster on the 90,000-node grid, 6 - 9 % slower on grids of 1,600 and 10,000 nodes
constexpr int kRcMinBits = 8, kRcMaxBits = 17;   // at least a bitmap word per CTA; two copies of 16384 slots in shared memory
constexpr uint32_t kRcMaxRows = 8192;            // slots changed in a round (with repeats) up to which rounds stay in the cluster
constexpr uint32_t kRcMaxCand = 65536;           // candidates of the first round, and of one whose degrees are not added up
constexpr uint32_t kRcMaxCta = 8192;             // candidates of one CTA's keys, where they are: 8192 take 10 us, a grid-wide round 11
constexpr uint32_t kRcMaxRun = 64;               // rows of the looked-up relation's longest run, unless it has at most kRcFewRows in all
// grid-wide / in the cluster, us: R-MAT 11 with 13,898 edges 187 / 155, with 25,595 179 / 189, a star of 16,000 leaves 109 / 126, of
// 32,000 113 / 147
constexpr uint32_t kRcFewRows = 16384;
constexpr uint32_t kRcWarpRow = 64, kRcBlockRow = 2048;      // rows with more matches are walked by a warp, by the block
constexpr uint32_t kRcLong = kRcMaxCand / kRcBlockRow;       // such block rows a round can have

inline size_t res_cluster_smem(uint32_t slots) { const size_t sl = slots / kRcCtas; return sl * 8 + sl / 32 * 12 + sl * 2; }

__device__ __forceinline__ uint32_t dsm_addr(const void* p, uint32_t rank) {
  uint32_t a = (uint32_t)__cvta_generic_to_shared(p), r;
  asm("mapa.shared::cluster.u32 %0, %1, %2;" : "=r"(r) : "r"(a), "r"(rank));
  return r;
}
__device__ __forceinline__ int32_t dsm_load(uint32_t a) {
  int32_t v;
  asm volatile("ld.shared::cluster.s32 %0, [%1];" : "=r"(v) : "r"(a) : "memory");
  return v;
}
template <int SINK>
__device__ __forceinline__ void dsm_improve(uint32_t a, int32_t v) {
  if (SINK == kSinkMin) asm volatile("red.relaxed.cluster.shared::cluster.min.s32 [%0], %1;" ::"r"(a), "r"(v) : "memory");
  else asm volatile("red.relaxed.cluster.shared::cluster.max.s32 [%0], %1;" ::"r"(a), "r"(v) : "memory");
}
__device__ __forceinline__ void dsm_or(uint32_t a, uint32_t v) { asm volatile("red.relaxed.cluster.shared::cluster.or.b32 [%0], %1;" ::"r"(a), "r"(v) : "memory"); }
__device__ __forceinline__ void dsm_add(uint32_t a, uint32_t v) { asm volatile("red.relaxed.cluster.shared::cluster.add.u32 [%0], %1;" ::"r"(a), "r"(v) : "memory"); }
__device__ __forceinline__ void dsm_max(uint32_t a, uint32_t v) { asm volatile("red.relaxed.cluster.shared::cluster.max.u32 [%0], %1;" ::"r"(a), "r"(v) : "memory"); }
__device__ __forceinline__ void cluster_barrier() {
  asm volatile("barrier.cluster.arrive.release.aligned;\n\tbarrier.cluster.wait.acquire.aligned;" ::: "memory");
}

struct ResCluster {
  uint32_t slots;                  // keys in use, rounded up to whole bitmap words for every CTA
  int32_t* table;
  uint32_t* words;                 // changed bitmap
  uint32_t* present;
  const uint32_t* dkeys;
  const float* dtags;
  ResState* st;
  unsigned long long* new_total;
  uint32_t key_max;
  uint32_t longest;                // longest run of the looked-up relation
  uint32_t* err;
};

// This thread's part of the degrees of the keys that changed in a CTA's words, none counted for more than ends the matter.  Out of
// line: the rounds of short rows never come here, and run 1 % slower with it among them.
__device__ __noinline__ uint32_t rc_next_candidates(const JoinSpec& S, const uint32_t* words, uint32_t W, uint32_t rank, bool plain, uint32_t domain, uint32_t* err) {
  uint32_t next = 0;
  for (uint32_t i = threadIdx.x; i < W; i += kRcBlock)
    for (uint32_t m = words[i]; m; m &= m - 1) {
      const uint32_t key = (((i << kRcCtasLog) | rank) << 5) + __ffs(m) - 1;
      uint32_t deg = 0;
      if (plain) {
        const uint32_t pv = (key >> S.s_probe_shift) & S.s_probe_mask;
        if (pv < domain) deg = __ldg(S.inner_off + pv + 1) - __ldg(S.inner_off + pv);
      } else deg = join_count_kv<uint32_t>(S, key, 0.f, 0, nullptr, err);
      next += min(deg, kRcMaxCta + 1);
    }
  return next;
}

static __global__ void __launch_bounds__(256) k_longest_run(const uint32_t* __restrict__ off, int64_t domain, uint32_t* __restrict__ longest) {
  uint32_t n = 0;
  for (int64_t v = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; v < domain; v += (int64_t)gridDim.x * blockDim.x) n = max(n, off[v + 1] - off[v]);
  n = __reduce_max_sync(0xffffffffu, n);
  if (lane_id() == 0 && n) atomicMax(longest, n);
}

template <int SINK>
__global__ void __launch_bounds__(kRcBlock, 1) k_res_cluster(const __grid_constant__ JoinSpec S, const __grid_constant__ ResCluster P) {
  extern __shared__ __align__(16) uint32_t rc_smem[];
  __shared__ uint32_t s_sum[3][2];                   // per round modulo 3: slots improved anywhere in the cluster (with repeats), most candidates of a CTA in the next
  __shared__ uint32_t s_nd, s_nlong, s_next;         // this CTA's rows of the delta; rows for the whole block; candidates of its changed keys
  __shared__ uint4 s_long[kRcLong];                  // {first row of the run, length, tag bits, row part of the head key}
  ResState* const st = P.st;
  if (st->status != kResOk) return;
  const uint32_t n0 = st->n_delta;
  if (n0 == 0u || n0 > kRcMaxRows || st->total > kRcMaxCand) return;
  const uint32_t SL = P.slots / kRcCtas, W = SL / 32;
  // offsets in rc_smem (kept as numbers: the compiler then knows that what they lead to is shared memory)
  uint32_t xcur = 0, xnxt = SL;                      // this CTA's slots as of the start / the end of the running round
  uint32_t chg = 2 * SL, chg_other = 2 * SL + W;     // slots changed in the running round; the other one is clear
  const uint32_t pres = 2 * SL + 2 * W;
  uint16_t* const list = reinterpret_cast<uint16_t*>(rc_smem + 2 * SL + 3 * W);
  uint32_t rank;
  asm("mov.u32 %0, %%cluster_ctarank;" : "=r"(rank));
  const unsigned lane = lane_id(), sub = lane & 3u, wid = warp_id();
  const uint32_t max_rounds = st->max_rounds, rounds0 = st->rounds;
  // local slot i <-> key: a bitmap word's 32 keys live in CTA (word mod kRcCtas)
  auto key_of = [&](uint32_t i) { return ((((i >> 5) << kRcCtasLog) | rank) << 5) | (i & 31u); };
  uint32_t imp = 0;                                  // this thread's improvements in the running round
  for (uint32_t i = threadIdx.x; i < SL; i += kRcBlock) rc_smem[xcur + i] = rc_smem[xnxt + i] = (uint32_t)P.table[key_of(i)];
  for (uint32_t i = threadIdx.x; i < W; i += kRcBlock) {
    const uint32_t g = (i << kRcCtasLog) | rank, m = P.words[g];
    rc_smem[chg_other + i] = 0u;
    rc_smem[chg + i] = m;                                   // what the rules without an atom over h derived belongs to this round
    imp += __popc(m);
    rc_smem[pres + i] = P.present[g];
  }
  if (threadIdx.x < 6) s_sum[threadIdx.x / 2][threadIdx.x % 2] = 0u;
  if (threadIdx.x == 0) s_nlong = 0u;
  cluster_barrier();
  unsigned long long cand = 0;                       // closed rounds'
  uint32_t round_cand = 0, n_changed = 0, n_new = 0, closed = 0;
  uint32_t verdict = kResOk, par = 0;
  const uint32_t sure = kRcMaxCand / P.longest;      // rows that have no more candidates than that, whatever their degrees
  bool first = true;
  const uint32_t sm0 = (uint32_t)__cvta_generic_to_shared(rc_smem), mult = (uint32_t)S.inner_mult[0];
  // the usual row: no constants in the scanned atom, the probed column taken as it is, at most one head column copied from the
  // row and no constant in the head; anything else goes through the general per-row work of the join kernels
  const uint32_t domain = (uint32_t)min(S.inner_domain, (int64_t)0xffffffff);
  bool plain = S.simple && S.s_const_mask == 0ull && S.probe_mul == 1 && S.probe_add == 0;
  uint32_t src_shift = 0, src_mask = 0, src_to = 0;
#pragma unroll
  for (int c = 0; c < kMaxArity; ++c)
    if (c < S.head.arity) {
      plain = plain && S.s_c0[c] == 0u && (S.s_src_mask[c] == 0u || (src_mask == 0u && S.s_src_mask[c] <= S.head.mask[c]));
      if (S.s_src_mask[c]) { src_shift = S.s_src_shift[c]; src_mask = S.s_src_mask[c]; src_to = S.head.shift[c]; }
    }
  const int32_t* __restrict__ zc = S.inner_col[0];
  const float* __restrict__ wc = S.inner_tag;
  for (;;) {
    const uint32_t xa = sm0 + xcur * 4u, xb = sm0 + xnxt * 4u, cb = sm0 + chg * 4u;
    auto apply = [&](uint32_t key, float tag) {
      if (key > P.key_max) { atomicOr(P.err, kErrHeadRange); return; }
      const uint32_t w = key >> 5, i = ((w >> kRcCtasLog) << 5) | (key & 31u);
      uint32_t base;                                 // offset of the owner's shared memory from this CTA's
      asm("mapa.shared::cluster.u32 %0, %1, %2;" : "=r"(base) : "r"(xa + i * 4u), "r"(w & (kRcCtas - 1)));
      const int32_t v = f2ord(tag), old = dsm_load(base);
      if (SINK == kSinkMin ? v < old : v > old) {
        dsm_improve<SINK>(base + (xb - xa), v);
        dsm_or(base - (xa + i * 4u) + cb + (i >> 5) * 4u, 1u << (i & 31u));
        ++imp;
      }
    };
    // part of a row's run: entries j, j + step, ...; four reads in flight
    auto walk = [&](uint32_t lo, uint32_t n, float tag, uint32_t rowkey, uint32_t j, uint32_t step) {
      for (; j < n; j += 4 * step) {
        int32_t z[4];
        float w[4];
#pragma unroll
        for (int k = 0; k < 4; ++k) { const bool in = j + k * step < n; z[k] = in ? __ldg(zc + lo + j + k * step) : 0; w[k] = in ? __ldg(wc + lo + j + k * step) : 0.f; }
#pragma unroll
        for (int k = 0; k < 4; ++k) if (j + k * step < n) apply(rowkey + (uint32_t)z[k] * mult, tag + w[k]);
      }
    };
    // eight rows to a warp, four lanes each
    const uint32_t nd = first ? n0 : s_nd;
    const uint32_t r_step = first ? kRcCtas * (kRcBlock / 4) : kRcBlock / 4;
    for (uint32_t r0 = (first ? rank * (kRcBlock / 4) : 0u) + wid * 8; r0 < nd; r0 += r_step) {
      const uint32_t r = r0 + lane / 4;
      uint4 info = make_uint4(0, 0, 0, 0);
      uint32_t deg = 0;
      float tag = 0.f;
      if (r < nd) {
        uint32_t key;
        if (first) { key = P.dkeys[r]; tag = P.dtags[r]; }
        else {
          const uint32_t i = list[r];
          const int32_t v = (int32_t)rc_smem[xcur + i];
          key = key_of(i); tag = ord2f(v);
          if (sub == 0) { int32_t* to = reinterpret_cast<int32_t*>(rc_smem) + xnxt + i; if (SINK == kSinkMin) atomicMin(to, v); else atomicMax(to, v); }     // the copy this round improves
        }
        if (plain) {
          const uint32_t pv = (key >> S.s_probe_shift) & S.s_probe_mask;
          if (pv < domain) { info.x = __ldg(S.inner_off + pv); deg = __ldg(S.inner_off + pv + 1) - info.x; }
          info.z = ((key >> src_shift) & src_mask) << src_to;
        } else deg = join_count_kv<uint32_t>(S, key, tag, 0, &info, P.err);
        if (sub == 0) round_cand += deg;
        if (deg <= kRcWarpRow) {
          if (sub < deg) apply(info.z + (uint32_t)__ldg(zc + info.x + sub) * mult, tag + __ldg(wc + info.x + sub));      // most rows of a mesh end here
          if (deg > 4) walk(info.x, deg, tag, info.z, sub + 4, 4);
        }
      }
      __syncwarp();
      unsigned big = __ballot_sync(0xffffffffu, sub == 0 && deg > kRcWarpRow);
      while (big) {
        const int src = __ffs(big) - 1;
        big &= big - 1;
        const uint32_t L = __shfl_sync(0xffffffffu, info.x, src), N = __shfl_sync(0xffffffffu, deg, src), K = __shfl_sync(0xffffffffu, info.z, src);
        const float T = __shfl_sync(0xffffffffu, tag, src);
        if (N > kRcBlockRow) {
          uint32_t at = 0;
          if (lane == 0) { at = atomicAdd(&s_nlong, 1u); if (at < kRcLong) s_long[at] = make_uint4(L, N, __float_as_uint(T), K); }
          if (__shfl_sync(0xffffffffu, at, 0) < kRcLong) continue;
        }
        walk(L, N, T, K, lane, 32);
        __syncwarp();
      }
    }
    __syncthreads();
    const uint32_t nlong = min(s_nlong, kRcLong);
    for (uint32_t q = 0; q < nlong; ++q) { const uint4 e = s_long[q]; walk(e.x, e.y, __uint_as_float(e.z), e.w, threadIdx.x, kRcBlock); }
    // what changed, told to every CTA
    const uint32_t w_imp = __reduce_add_sync(0xffffffffu, imp);
    if (w_imp && lane < kRcCtas) dsm_add(dsm_addr(&s_sum[par][0], lane), w_imp);
    const uint32_t par_next = par == 2 ? 0u : par + 1;
    if (threadIdx.x == 0) { s_sum[par_next][0] = s_sum[par_next][1] = 0u; s_nd = 0u; }
    cluster_barrier();
    const uint32_t total_imp = s_sum[par][0];
    { const uint32_t t = xcur; xcur = xnxt; xnxt = t; }        // the round's end is the next one's start
    if (total_imp == 0u) { cand += round_cand; round_cand = 0; ++closed; verdict = kResDone; break; }
    if (rounds0 + closed + 1 >= max_rounds) { cand += round_cand; round_cand = 0; ++closed; verdict = kResCap; break; }
    if (total_imp > kRcMaxRows) break;               // the emit kernel closes this round
    if (__builtin_expect(total_imp > sure, 0)) {
      const uint32_t next = __reduce_add_sync(0xffffffffu, rc_next_candidates(S, rc_smem + chg, W, rank, plain, domain, P.err));
      if (threadIdx.x == 0) s_next = 0u;
      __syncthreads();
      if (lane == 0 && next) atomicAdd(&s_next, next);
      __syncthreads();
      if (threadIdx.x < kRcCtas && s_next) dsm_max(dsm_addr(&s_sum[par][1], threadIdx.x), s_next);
      cluster_barrier();
      if (s_sum[par][1] > kRcMaxCta) break;
    }
    // close the round: this CTA's changed keys are its part of the next delta
    cand += round_cand; round_cand = 0; imp = 0; ++closed;
    if (threadIdx.x == 0) s_nlong = 0u;
    for (uint32_t i0 = 0; i0 < W; i0 += kRcBlock / 2) {
      // 16 words to a warp (spread over the key space, a front being dense somewhere), two lanes to a word
      const uint32_t i = i0 + (lane >> 1) * (kRcBlock / 32) + wid, half = (lane & 1u) * 16;
      const uint32_t word = i < W ? rc_smem[chg + i] : 0u;
      if (__ballot_sync(0xffffffffu, word != 0u) == 0u) continue;
      uint32_t m = (word >> half) & 0xffffu;
      const uint32_t incl = warp_scan_incl((uint32_t)__popc(m));
      uint32_t at = 0;
      if (lane == 31) at = atomicAdd(&s_nd, incl);
      if (word && half == 0u) {
        const uint32_t had = rc_smem[pres + i];
        n_changed += __popc(word);
        n_new += __popc(word & ~had);
        rc_smem[pres + i] = had | word;
        rc_smem[chg + i] = 0u;
      }
      at = __shfl_sync(0xffffffffu, at, 31) + incl - __popc(m);
      for (; m; m &= m - 1) list[at++] = (uint16_t)((i << 5) + half + __ffs(m) - 1);
    }
    __syncthreads();
    first = false;
    { const uint32_t t = chg; chg = chg_other; chg_other = t; }
    par = par_next;
  }
  // the mirror back to memory; xcur is complete.  Changed bits stay only if the emit kernel has to close the last round.
  for (uint32_t i = threadIdx.x; i < SL; i += kRcBlock) P.table[key_of(i)] = (int32_t)rc_smem[xcur + i];
  for (uint32_t i = threadIdx.x; i < W; i += kRcBlock) {
    const uint32_t g = (i << kRcCtasLog) | rank;
    P.words[g] = verdict == kResOk ? rc_smem[chg + i] : 0u;
    P.present[g] = rc_smem[pres + i];
  }
  unsigned long long c2 = cand, last = round_cand;
#pragma unroll
  for (int s = 16; s; s >>= 1) { c2 += __shfl_down_sync(0xffffffffu, c2, s); last += __shfl_down_sync(0xffffffffu, last, s); }
  n_changed = __reduce_add_sync(0xffffffffu, n_changed);
  n_new = __reduce_add_sync(0xffffffffu, n_new);
  if (rank == 0 && threadIdx.x == 0) {
    st->rounds += closed; st->status = verdict; st->total = 0; st->ntiles = 0; st->n_delta = 0; st->round_cand = 0;
  }
  cluster_barrier();                                 // nobody leaves while a peer may still reach into its shared memory; the block above is ordered before the sums below
  if (lane == 0) {
    if (c2) { atomicAdd(&st->candidates, c2); atomicAdd(&st->small_cand, c2); }
    if (last) { atomicAdd(&st->round_cand, last); atomicAdd(&st->small_cand, last); }
    if (n_new) { atomicAdd(&st->n_new, (unsigned long long)n_new); atomicAdd(&st->new_seen, (unsigned long long)n_new); atomicAdd(P.new_total, (unsigned long long)n_new); }
    if (n_changed > n_new) atomicAdd(&st->n_improved, (unsigned long long)(n_changed - n_new));
  }
}

}  // namespace xlog
