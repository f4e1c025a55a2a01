// Closing a cycle over dense lists: the materialised triangle and four-cycle joins when the lists to be intersected are dense in a
// small domain of the last variable w.
//
// A path (a row of r(x,y), or a two-path (x,y,z)) is closed by every w in both the list of its last column and the list of its
// first.  As bitmaps the two lists are met word by word, one AND where the list kernels (triangle.cuh, cycle4.cuh) read, test
// and rank entry by entry - a list of 64 entries over 1,024 values is 32 words.  Four lanes take a path, each a run of
// neighbouring words read 16 bytes at a time, so that a warp instruction serves eight paths.  Beside every word stands the
// place in the list of its first entry, so that a hit's place (for its tag) is that plus popcounts.  The bitmaps are made
// from a join index when first wanted and kept with it.
//
// Bound by instruction issue.  Four-cycle join, 4.2 M two-paths over 1,024 values, 16.8 M rows: count 0.55 -> 0.07 ms, write
// 1.55 -> 0.37 ms; a lane per word and the hits of a path written as they fell: 0.23 and 0.75.  Triangle join, 65,536 rows over
// 406 values, 4.2 M rows: 62 -> 9 us and 84 -> 61 us.
//
//   k_bits_lists   list entries -> bits, and running counts per word
//   k_bits_count   matches per path
//   k_bits_emit    the rows: hits are queued per warp with their place in the output and worked off 32 at a time, so that
//                  the two tag reads and the writes use every lane though a path has few hits
#pragma once
#include "common.cuh"

namespace xlog {

constexpr uint32_t kBitsMaxWords = 512;          // w below 2^14
constexpr int kBitsLanes = 4;                    // lanes per path
// words of a list: a lane takes 4 (short lists) or 8 words of every stretch of 16 or 32
inline uint32_t bits_padded(uint32_t words) { return words <= 16 ? 16u : (words + 31) / 32 * 32; }
constexpr uint32_t kBitsQueue = 256;             // hits a warp holds before it works them off

// A warp per list: its entries' bits are set in shared memory, then every word is written with the number of entries before it.
static __global__ void __launch_bounds__(256) k_bits_lists(const uint32_t* __restrict__ off, int64_t domain, const int32_t* __restrict__ col, uint32_t words, uint32_t* __restrict__ bits,
                                                           uint16_t* __restrict__ rank) {
  __shared__ uint32_t s_bits[8][kBitsMaxWords];
  uint32_t* const row = s_bits[warp_id()];
  const unsigned lane = lane_id();
  const int64_t nwarps = ((int64_t)gridDim.x * blockDim.x) >> 5;
  for (int64_t v = ((int64_t)blockIdx.x * blockDim.x + threadIdx.x) >> 5; v < domain; v += nwarps) {
    for (uint32_t k = lane; k < words; k += 32) row[k] = 0u;
    __syncwarp();
    for (uint32_t i = off[v] + lane; i < off[v + 1]; i += 32) { const uint32_t w = (uint32_t)col[i]; atomicOr(row + (w >> 5), 1u << (w & 31)); }
    __syncwarp();
    uint32_t run = 0;
    for (uint32_t k = 0; k < words; k += 32) {
      const bool in = k + lane < words;
      const uint32_t b = in ? row[k + lane] : 0u, n = (uint32_t)__popc(b), incl = warp_scan_incl(n);
      if (in) { bits[(size_t)v * words + k + lane] = b; rank[(size_t)v * words + k + lane] = (uint16_t)(run + incl - n); }
      run += __shfl_sync(0xffffffffu, incl, 31);
    }
    __syncwarp();
  }
}

struct BitsLists {
  const uint32_t* bits;            // [domain][words]
  const uint16_t* rank;
  const uint32_t* off;             // the index's offsets: list of v starts at off[v]
  const float* tag;                // its tags
  uint32_t domain;
};

struct BitsJoin {
  KeyLayout path;                  // the paths' key layout; A is looked up with the last column, B with the first
  KeyLayout head;                  // the path's columns, then w
  BitsLists A, B;
  uint32_t words;
  int times;
};

template <typename K2>
__device__ __forceinline__ bool bits_path(const BitsJoin& P, K2 key, uint32_t& a, uint32_t& b) {
  a = (uint32_t)key_col<K2>(P.path, key, P.path.arity - 1);
  b = (uint32_t)key_col<K2>(P.path, key, 0);
  const bool ok = a < P.A.domain && b < P.B.domain;
  if (!ok) a = b = 0u;
  return ok;
}

// A lane's words of one stretch of a list.
template <int WB>
__device__ __forceinline__ void bits_words_of(const uint32_t* __restrict__ row, bool live, uint32_t (&w)[WB]) {
#pragma unroll
  for (int q = 0; q < WB / 4; ++q) {
    const uint4 x = live ? reinterpret_cast<const uint4*>(row)[q] : make_uint4(0u, 0u, 0u, 0u);
    w[4 * q] = x.x; w[4 * q + 1] = x.y; w[4 * q + 2] = x.z; w[4 * q + 3] = x.w;
  }
}

// A warp takes 32 paths, eight per step.
template <typename K2, int WB>
__global__ void __launch_bounds__(256) k_bits_count(const __grid_constant__ BitsJoin P, const K2* __restrict__ keys, uint64_t n, uint32_t* __restrict__ cnt) {
  const uint64_t nwarps = ((uint64_t)gridDim.x * blockDim.x) >> 5;
  const unsigned lane = lane_id(), sub = lane % kBitsLanes;
  for (uint64_t base = (((uint64_t)blockIdx.x * blockDim.x + threadIdx.x) >> 5) * 32; base < n; base += nwarps * 32) {
    uint32_t a = 0, b = 0, mine = 0;
    const bool ok = base + lane < n && bits_path<K2>(P, keys[base + lane], a, b);
#pragma unroll
    for (int j = 0; j < kBitsLanes; ++j) {
      const int p = j * 8 + lane / kBitsLanes;
      const uint32_t* ra = P.A.bits + (size_t)(__shfl_sync(0xffffffffu, a, p) * P.words) + sub * WB;
      const uint32_t* rb = P.B.bits + (size_t)(__shfl_sync(0xffffffffu, b, p) * P.words) + sub * WB;
      uint32_t s = 0;
      for (uint32_t k = 0; k < P.words; k += WB * kBitsLanes) {
        uint32_t wa[WB], wb[WB];
        bits_words_of<WB>(ra + k, true, wa);
        bits_words_of<WB>(rb + k, true, wb);
#pragma unroll
        for (int q = 0; q < WB; ++q) s += __popc(wa[q] & wb[q]);
      }
#pragma unroll
      for (int d = kBitsLanes / 2; d; d >>= 1) s += __shfl_xor_sync(0xffffffffu, s, d);
      const uint32_t got = __shfl_sync(0xffffffffu, s, (lane % 8) * kBitsLanes);
      if ((int)lane / 8 == j) mine = got;
    }
    if (base + lane < n) cnt[base + lane] = ok ? mine : 0u;
  }
}

template <typename K2, typename K, int WB>
__global__ void __launch_bounds__(256) k_bits_emit(const __grid_constant__ BitsJoin P, const K2* __restrict__ keys, const float* __restrict__ tags, uint64_t n,
                                                   const uint64_t* __restrict__ off, K* __restrict__ out_keys, float* __restrict__ out_tags) {
  __shared__ uint4 s_queue[8][kBitsQueue];         // {output row, w | path << 14, place in A's list, in B's}
  uint4* queue = s_queue[warp_id()];
  const uint64_t nwarps = ((uint64_t)gridDim.x * blockDim.x) >> 5;
  const unsigned lane = lane_id(), sub = lane % kBitsLanes, first = lane - sub;
  for (uint64_t base = (((uint64_t)blockIdx.x * blockDim.x + threadIdx.x) >> 5) * 32; base < n; base += nwarps * 32) {
    uint32_t a = 0, b = 0, to = 0, ok = 0;
    K prefix = 0;
    float tag = 0.f;
    if (base + lane < n) {
      const K2 k2 = keys[base + lane];
      ok = bits_path<K2>(P, k2, a, b) ? 1u : 0u;
      to = (uint32_t)off[base + lane];
      tag = tags[base + lane];
#pragma unroll
      for (int c = 0; c < kMaxArity; ++c) if (c < P.path.arity) prefix |= (K)(uint32_t)key_col<K2>(P.path, k2, c) << P.head.shift[c];
    }
    auto write = [&](const uint4 h, const K pre, const float tg) {
      const float ta = P.A.tag[h.z], tb = P.B.tag[h.w];
      out_keys[h.x] = pre | ((K)(h.y & 0x3fffu) << P.head.shift[P.path.arity]);
      out_tags[h.x] = P.times ? (tg * ta) * tb : (tg + ta) + tb;
    };
    uint32_t qn = 0;                               // queued hits (uniform)
    auto flush = [&]() {
      __syncwarp();
      for (uint32_t i = 0; i < qn; i += 32) {
        const uint4 h = i + lane < qn ? queue[i + lane] : make_uint4(0u, 0u, 0u, 0u);
        const int p = h.y >> 14;
        const K pre = (K)__shfl_sync(0xffffffffu, prefix, p);
        const float tg = __shfl_sync(0xffffffffu, tag, p);
        if (i + lane < qn) write(h, pre, tg);
      }
      qn = 0;
      __syncwarp();
    };
#pragma unroll 1
    for (int j = 0; j < kBitsLanes; ++j) {
      const uint32_t p = j * 8 + lane / kBitsLanes;
      const uint32_t pa = __shfl_sync(0xffffffffu, a, p), pb = __shfl_sync(0xffffffffu, b, p);
      const bool live = __shfl_sync(0xffffffffu, ok, p) != 0u;
      uint32_t at = __shfl_sync(0xffffffffu, to, p);
      for (uint32_t k0 = sub * WB; k0 < P.words; k0 += WB * kBitsLanes) {
        const uint32_t ra = pa * P.words + k0, rb = pb * P.words + k0;
        uint32_t wa[WB], wb[WB];
        bits_words_of<WB>(P.A.bits + ra, live, wa);
        bits_words_of<WB>(P.B.bits + rb, live, wb);
        uint32_t mine = 0;
#pragma unroll
        for (int q = 0; q < WB; ++q) mine += __popc(wa[q] & wb[q]);
        const uint32_t incl = warp_scan_incl(mine), total = __shfl_sync(0xffffffffu, incl, 31);
        if (total == 0u) continue;                 // uniform
        const uint32_t before = __shfl_sync(0xffffffffu, incl - mine, first);
        uint32_t row = at + incl - mine - before;  // output row of the lane's next hit
        at += __shfl_sync(0xffffffffu, incl, first + kBitsLanes - 1) - before;
        if (qn + total > kBitsQueue) flush();
        const bool queued = total <= kBitsQueue;   // else the lanes have many hits each and write them themselves
        uint32_t pos = qn + incl - mine, from_a = 0, from_b = 0;
        K pre = 0;
        float tg = 0.f;
        if (mine) { from_a = P.A.off[pa] + P.A.rank[ra]; from_b = P.B.off[pb] + P.B.rank[rb]; }
        if (!queued) { pre = (K)__shfl_sync(0xffffffffu, prefix, p); tg = __shfl_sync(0xffffffffu, tag, p); }
#pragma unroll
        for (int q = 0; q < WB; ++q) {
          for (uint32_t m = wa[q] & wb[q]; m; m &= m - 1) {
            const uint32_t bit = __ffs(m) - 1, below = (1u << bit) - 1u;
            const uint4 h = make_uint4(row++, ((k0 + q) << 5) | bit | p << 14, from_a + __popc(wa[q] & below), from_b + __popc(wb[q] & below));
            if (queued) queue[pos++] = h; else write(h, pre, tg);
          }
          from_a += __popc(wa[q]); from_b += __popc(wb[q]);
        }
        if (queued) qn += total;
        __syncwarp();
      }
    }
    flush();
  }
}

}  // namespace xlog
