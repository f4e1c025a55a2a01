// A two-atom rule whose groups are products of two runs:   h(p', c0 + k1 * a + k2 * b) :- d(m p + s, a), e(m' p + s', b)
// (the digit sum is  sum(p, a + b) :- digit(2p, a), digit(2p + 1, b)).
//
// Both atoms are met on p, so the group of p is the product of one run of d and one run of e, and when the head's second column
// takes at most 32 values ("slots") and so does d's, a run is at most a row a lane and a warp needs no candidate in memory: a
// lane holds the tag of the e row that would land in its slot from row part 0, each row of d moves those tags along by its own
// part (one read of shared memory), and each lane folds what comes by.  The sorting route writes every candidate, sorts, and reduces by key.
//
//   k_group_rule      a warp per p: aggregates and the mask of slots that have any; counts of rows and candidates per block
//   k_group_emit      the same blocks: the counts of the blocks before are the offset, rows go out in key order.  The host
//                     needs no count in between: the rows have room for every slot.
//   k_group_backward  a warp per p: the group's head rows, one per lane, found next to those of the p before; weights are
//                     summed in registers per row of d and of e, and meet memory once per row
//
// 65,536 pairs of digits (6.55 million candidates, 1.25 million rows): evaluation 390 -> 119 us, gradient 338 -> 81 us; 64 pairs:
// 164 -> 70 us and 106 -> 35 us, all of it launches and the wait for the counts.  The kernels take 41, 20 and 49 us and are bound
// by instruction issue (10 rows of d a group, an exponential and a dozen instructions each; the memory of it would take 5 us);
// candidates found by a search over the lanes instead of two runs laid against each other: 213 and 168 us.
#pragma once
#include "common.cuh"
#include "join.cuh"

namespace xlog {

constexpr int kGroupSlots = 32;
constexpr uint32_t kGroupEmpty = 0xffffdeadu;    // no sum or product has this pattern: the arithmetic's one NaN is 0x7fffffff
constexpr int kGroupBlock = 256;

struct GroupRule {
  uint32_t n_groups;                             // p in [0, n_groups)
  int64_t mul0, add0, mul1, add1;                // runs: d's first column is mul0 * p + add0, e's is mul1 * p + add1
  const uint32_t *off0, *off1;                   // their offsets
  int64_t domain0, domain1;
  uint32_t mask0;                                // d's second column: key & mask0
  const float* tag0;
  const int32_t* col1;                           // e's second column and tags, in the order of off1
  const float* tag1;
  int64_t top_c0, top_mul;                       // head's first column: top_c0 + top_mul * p
  int64_t c0, mulp, k0;                          // row part of the second: c0 + mulp * p + k0 * a
  uint32_t k1;                                   // and e's part: k1 * b
  int shift;                                     // bits of the head's second column
  uint32_t top_mask;
  uint32_t slots;                                // values of the second column, <= kGroupSlots
  uint32_t per_warp;                             // groups a warp takes, one after another
  uint32_t* mask;                                // per group: the slots that have rows
  float* agg;                                    // [group][slots]
  ulonglong2* sums;                              // per block: rows, candidates
  uint32_t* err;
};

// A warp's groups, 32 at a time: lane i works out the runs of group p0 + i.
__device__ __forceinline__ uint4 group_runs(const GroupRule& P, uint32_t p, uint32_t end) {
  uint4 r = make_uint4(0, 0, 0, 0);
  if (p < end) {
    const int64_t x = P.mul0 * p + P.add0, y = P.mul1 * p + P.add1;
    if (x >= 0 && x < P.domain0 && y >= 0 && y < P.domain1) r = make_uint4(P.off0[x], P.off0[x + 1], P.off1[y], P.off1[y + 1]);
    if (r.x == r.y || r.z == r.w) r = make_uint4(0, 0, 0, 0);
  }
  return r;
}
__device__ __forceinline__ uint4 group_runs_of(uint4 r, int i) {
  return make_uint4(__shfl_sync(0xffffffffu, r.x, i), __shfl_sync(0xffffffffu, r.y, i), __shfl_sync(0xffffffffu, r.z, i), __shfl_sync(0xffffffffu, r.w, i));
}

// The part of the second column that a row of d gives; out of the column's range: an error, as for any head value.
__device__ __forceinline__ uint32_t group_row_part(const GroupRule& P, uint32_t p, uint32_t a, uint32_t& e) {
  const int64_t v = P.c0 + P.mulp * p + P.k0 * a;
  if (v < 0 || v >= (int64_t)P.slots) { e |= kErrHeadRange; return 0; }
  return (uint32_t)v;
}
__device__ __forceinline__ uint32_t group_slot(const GroupRule& P, uint32_t b, uint32_t& e) {
  const uint64_t v = (uint64_t)P.k1 * b;
  if (v >= P.slots) { e |= kErrHeadRange; return 0; }
  return (uint32_t)v;
}

struct GroupSmem {
  uint32_t tab[64];                              // [32 + s]: tag that lands in slot s from row part 0; below 32: none
  float2 row[32];                                // rows of d: part (as an integer), tag
};

template <typename Op> struct GroupFold {
  typename Op::A acc = Op::identity();
  __device__ __forceinline__ void take(float t, bool there) { if (there) acc = Op::combine(acc, Op::lift(t)); }
  __device__ __forceinline__ float lower() { return Op::lower(acc); }
};
template <> struct GroupFold<OpLse> {            // one exponential a value
  float m = -3.402823466e38f, s = 0.f;
  __device__ __forceinline__ void take(float t, bool there) {
    t = there ? t : -INFINITY;
    const float d = t - m, x = expf(-fabsf(d));
    s = d > 0.f ? fmaf(s, x, 1.f) : s + x;
    m = fmaxf(m, t);
  }
  __device__ __forceinline__ float lower() { return s == 0.f ? -INFINITY : m + logf(s); }
};

template <typename KO, typename Op, bool TIMES>
__global__ void __launch_bounds__(kGroupBlock) k_group_rule(const __grid_constant__ GroupRule P, const KO* __restrict__ key0) {
  __shared__ GroupSmem s_warp[kGroupBlock / 32];
  __shared__ unsigned long long s_rows, s_cand;
  GroupSmem& sm = s_warp[warp_id()];
  const unsigned lane = lane_id();
  if (threadIdx.x == 0) { s_rows = 0; s_cand = 0; }
  sm.tab[lane] = kGroupEmpty;
  __syncthreads();
  unsigned long long cand = 0;
  uint32_t rows = 0, e = 0;
  const uint64_t w = (uint64_t)blockIdx.x * (kGroupBlock / 32) + warp_id();
  const uint32_t end = (uint32_t)min((uint64_t)P.n_groups, (w + 1) * P.per_warp);
  for (uint32_t p0 = (uint32_t)min((uint64_t)P.n_groups, w * P.per_warp); p0 < end; p0 += 32) {
    const uint4 runs = group_runs(P, p0 + lane, end);
    const int64_t top = P.top_c0 + P.top_mul * (p0 + lane);
    if (runs.x < runs.y && (top < 0 || top > (int64_t)P.top_mask)) e |= kErrHeadRange;
    uint32_t my_mask = 0;
    for (uint32_t todo = __ballot_sync(0xffffffffu, runs.x < runs.y); todo; todo &= todo - 1) {
      const int g = __ffs(todo) - 1;
      const uint32_t p = p0 + g;
      const uint4 r = group_runs_of(runs, g);
      uint32_t ka = 0;
      float ta = 0.f;
      if (r.x + lane < r.y) { ka = (uint32_t)key0[r.x + lane] & P.mask0; ta = P.tag0[r.x + lane]; }
      cand += (unsigned long long)(r.y - r.x) * (r.w - r.z);
      sm.tab[32 + lane] = kGroupEmpty;
      __syncwarp();
      uint32_t at_b = 0;
      if (r.z + lane < r.w) {
        const uint32_t z = group_slot(P, (uint32_t)P.col1[r.z + lane], e);
        sm.tab[32 + z] = __float_as_uint(P.tag1[r.z + lane]);
        at_b = 1u << z;
      }
      at_b = __reduce_or_sync(0xffffffffu, at_b);
      GroupFold<Op> f;
      uint32_t mask = 0;
      const uint32_t nr = min(32u, r.y - r.x);
      if (lane < nr) {
        const uint32_t off = group_row_part(P, p, ka, e);
        sm.row[lane] = make_float2(__uint_as_float(off), ta);
        mask = at_b << off;
        if (off + (31 - __clz(at_b)) >= P.slots) e |= kErrHeadRange;
      }
      __syncwarp();
      for (uint32_t i = 0; i < nr; ++i) {
        const float2 row = sm.row[i];
        const uint32_t bt = sm.tab[32 + lane - __float_as_uint(row.x)];
        f.take(TIMES ? row.y * __uint_as_float(bt) : row.y + __uint_as_float(bt), bt != kGroupEmpty);
      }
      __syncwarp();
      mask = __reduce_or_sync(0xffffffffu, mask);
      if ((mask >> lane) & 1u && lane < P.slots) P.agg[(size_t)p * P.slots + lane] = f.lower();
      if ((int)lane == g) my_mask = mask;
    }
    if (p0 + lane < end) P.mask[p0 + lane] = my_mask;
    rows += __popc(my_mask);
  }
  rows = __reduce_add_sync(0xffffffffu, rows);
  if (lane == 0 && cand) { atomicAdd(&s_cand, cand); atomicAdd(&s_rows, (unsigned long long)rows); }
  if (e) atomicOr(P.err, e);
  __syncthreads();
  if (threadIdx.x == 0) P.sums[blockIdx.x] = make_ulonglong2(s_rows, s_cand);
}

// totals: rows, candidates
template <typename K>
__global__ void __launch_bounds__(kGroupBlock) k_group_emit(const __grid_constant__ GroupRule P, K* __restrict__ keys, float* __restrict__ tags, unsigned long long* __restrict__ totals) {
  __shared__ uint32_t s_mask[kGroupBlock], s_off[kGroupBlock], sh[kGroupBlock / 32 + 1];
  __shared__ unsigned long long s_base[kGroupBlock / 32], s_cand;
  const unsigned lane = lane_id();
  if (threadIdx.x == 0) s_cand = 0;
  const bool last = blockIdx.x + 1 == gridDim.x;
  unsigned long long before = 0, cand = 0;
#pragma unroll 4
  for (uint32_t i = threadIdx.x; i < blockIdx.x + (last ? 1u : 0u); i += kGroupBlock) {
    const ulonglong2 s = P.sums[i];
    if (i < blockIdx.x) before += s.x;
    cand += s.y;
  }
#pragma unroll
  for (int d = 16; d; d >>= 1) before += __shfl_xor_sync(0xffffffffu, before, d);
  if (lane == 0) s_base[warp_id()] = before;
  __syncthreads();
  if (last && cand) atomicAdd(&s_cand, cand);
  unsigned long long base = 0;
  for (int i = 0; i < kGroupBlock / 32; ++i) base += s_base[i];
  const uint64_t per_block = (uint64_t)P.per_warp * (kGroupBlock / 32);
  const uint32_t first = (uint32_t)(blockIdx.x * per_block), end = (uint32_t)min((uint64_t)P.n_groups, first + per_block);
  for (uint32_t p0 = first; p0 < end; p0 += kGroupBlock) {
    const uint32_t n = min((uint32_t)kGroupBlock, end - p0), mk = threadIdx.x < n ? P.mask[p0 + threadIdx.x] : 0u;
    uint32_t total;
    s_off[threadIdx.x] = block_scan_excl<kGroupBlock, uint32_t>((uint32_t)__popc(mk), sh, total);
    s_mask[threadIdx.x] = mk;
    __syncthreads();
#pragma unroll 4
    for (uint32_t i = warp_id(); i < n; i += kGroupBlock / 32) {
      const uint32_t mask = s_mask[i], p = p0 + i;
      if ((mask >> lane) & 1u) {
        const size_t row = base + s_off[i] + __popc(mask & lanemask_lt());
        keys[row] = ((K)(uint32_t)(P.top_c0 + P.top_mul * p) << P.shift) | (K)lane;
        tags[row] = P.agg[(size_t)p * P.slots + lane];
      }
    }
    base += total;
    __syncthreads();
  }
  if (last && threadIdx.x == 0) { totals[0] = base; totals[1] = s_cand; }
}

// Half a warp per row of d while e's run has at most 16 rows.
template <typename KO, typename KH, bool LSE>
__global__ void __launch_bounds__(kGroupBlock) k_group_backward(const __grid_constant__ GroupRule P, const KO* __restrict__ key0, const __grid_constant__ BwdArgs bw) {
  struct Smem { float2 head[32], row[32]; float row_sum[32]; };
  __shared__ Smem s_warp[kGroupBlock / 32];
  Smem& sm = s_warp[warp_id()];
  const unsigned lane = lane_id();
  const KH* __restrict__ hk = reinterpret_cast<const KH*>(bw.head_keys);
  const uint64_t w = (uint64_t)blockIdx.x * (kGroupBlock / 32) + warp_id();
  const uint32_t end = (uint32_t)min((uint64_t)P.n_groups, (w + 1) * P.per_warp);
  uint32_t e = 0, h = 0;                         // rows before h are of earlier groups
  bool placed = false;
  for (uint32_t p0 = (uint32_t)min((uint64_t)P.n_groups, w * P.per_warp); p0 < end; p0 += 32) {
    const uint4 runs = group_runs(P, p0 + lane, end);
    for (uint32_t todo = __ballot_sync(0xffffffffu, runs.x < runs.y); todo; todo &= todo - 1) {
      const int gi = __ffs(todo) - 1;
      const uint32_t p = p0 + gi;
      const uint4 r = group_runs_of(runs, gi);
      const uint32_t nb = min(32u, r.w - r.z), wide = nb > 16 ? 32u : 16u, sub = lane & (wide - 1);
      uint32_t ka = 0, zb = 0;
      float ta = 0.f, tb = 0.f;
      if (r.x + lane < r.y) { ka = (uint32_t)key0[r.x + lane] & P.mask0; ta = P.tag0[r.x + lane]; }
      if (sub < nb) { zb = (uint32_t)P.col1[r.z + sub]; tb = P.tag1[r.z + sub]; }
      // the group's head rows, a lane per row, then a place per slot
      const KH top = (KH)(P.top_c0 + P.top_mul * p), want = top << P.shift;
      KH k = 0;
      bool at = h + lane < bw.n_head;
      if (at) k = hk[h + lane];
      if (!placed || __shfl_sync(0xffffffffu, (int)(at && k < want), 0)) {
        uint32_t lo = h, hi = bw.n_head;         // the first row >= want lies in [lo, hi]; 32 probes a step
        while (hi - lo > 32) {
          const uint32_t step = (hi - lo) / 32;
          const int n = __popc(__ballot_sync(0xffffffffu, hk[lo + (lane + 1) * step - 1] < want));
          if (n < 32) hi = lo + (n + 1) * step - 1;
          lo += n * step;
        }
        h = lo + __popc(__ballot_sync(0xffffffffu, lo + lane < hi && hk[lo + lane] < want));
        placed = true;
        at = h + lane < bw.n_head;
        if (at) k = hk[h + lane];
      }
      at = at && (k >> P.shift) == top;
      const uint32_t mine = (uint32_t)k & ((1u << P.shift) - 1u);
      if (at) sm.head[mine] = make_float2(bw.grad_head[h + lane], bw.head_tags[h + lane]);
      h += __popc(__ballot_sync(0xffffffffu, at));
      const uint32_t present = __reduce_or_sync(0xffffffffu, at ? 1u << mine : 0u);

      const uint32_t nr = min(32u, r.y - r.x);
      if (lane < nr) sm.row[lane] = make_float2(__uint_as_float(group_row_part(P, p, ka, e)), ta);
      sm.row_sum[lane] = 0.f;
      const uint32_t z = sub < nb ? group_slot(P, zb, e) : 0u;
      float inner = 0.f;
      __syncwarp();
      for (uint32_t i = lane / wide; i < nr + lane / wide; i += 32 / wide) {       // the same number of turns for every lane
        float to_a = 0.f;
        if (i < nr && sub < nb) {
          const float2 row = sm.row[i];
          const uint32_t slot = __float_as_uint(row.x) + z;
          if (slot > 31 || !((present >> slot) & 1u)) e |= kErrInternal;
          else {
            const float2 head = sm.head[slot];
            if (LSE) { to_a = head.x * expf(row.y + tb - head.y); inner += to_a; }
            else { to_a = head.x * tb; inner += head.x * row.y; }
          }
        }
#pragma unroll
        for (int d = 8; d; d >>= 1) to_a += __shfl_xor_sync(0xffffffffu, to_a, d);
        if (wide == 32) to_a += __shfl_xor_sync(0xffffffffu, to_a, 16);
        if (sub == 0 && i < nr) sm.row_sum[i] = to_a;
      }
      if (wide == 16) inner += __shfl_xor_sync(0xffffffffu, inner, 16);
      if (bw.grad_inner && lane < nb) atomicAdd(bw.grad_inner + r.z + lane, inner);
      __syncwarp();
      if (lane < nr) atomicAdd(bw.grad_outer + r.x + lane, sm.row_sum[lane]);
      __syncwarp();
    }
  }
  if (e) atomicOr(P.err, e);
}

}  // namespace xlog
