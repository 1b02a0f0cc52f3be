// cta_sort.cuh -- one CTA sorts up to NT*ITEMS (key, position) pairs that its
// threads hold in registers (element e = r*NT + threadIdx.x sits in slot r).
//
// The result is the lexicographic (key, position) order, left in shared
// memory.  Size-dependent choice (the paper's per-input-size algorithm choice,
// Section 6, applied to one bucket):
//
//   m <= kRankMax       rank-by-counting: slot = #{pairs smaller than me}
//                       (the ranking of Appendix "Fast Work-Inefficient
//                       Ranking", all in one CTA)
//   otherwise           split the bucket's key range [min, max] into
//                       two equal-width bins per slot of the CTA (a counting
//                       sort in shared memory), then order each bin that holds
//                       several elements by insertion (an element alone in
//                       its bin is already in place); the bins of a bucket
//                       are tiny unless its keys cluster
//   a crowded bin       refine the bins once: a bin that holds c elements is
//   (> kBinLimit)       cut into 2 c equal parts, so that the bins follow the
//                       keys' density (float64 values, whose bit patterns
//                       crowd a few octaves of a range of thousands)
//   still crowded       bitonic sort of the whole bucket (Appendix "Bitonic
//                       Sort"), which needs no assumption on the keys
//
// (k_local_sort ranks a crowded bucket of at most a pair a thread instead.)
//
// A bucket whose keys are all equal and whose elements arrive in position
// order (every bucket produced by the stable scatter) is already sorted; if
// they arrive in another order, the bins are taken over the positions.
#pragma once

#include "rsort_internal.cuh"

namespace rsort {

constexpr int kBinLimit = 16;
static_assert(kRankMax <= kLocalThreads, "rank-by-counting holds one element per thread");

struct CtaSortSmem {
  uint64_t* k;     // [cap]      cap = NT * ITEMS
  uint32_t* i;     // [cap]
  uint32_t* hist;  // BinSort's counters, then its list of bins to order
};

// Layout of the bins of a CTA with IT slots a thread: 2 * NT * IT 16-bit
// counters, two to a word, every thread's run of IT words 4 words apart from the
// next, so that eight lanes' 16-byte accesses to their runs cover all banks;
// then the end of the last bin, and the list of bins that hold several pairs.
template <int NT, int IT>
struct BinSort {
  static constexpr int log2c(int x) { return x <= 1 ? 0 : 1 + log2c(x / 2); }
  static constexpr int kCap = NT * IT;
  static constexpr int kLogIt = log2c(IT);
  static_assert((1 << kLogIt) == IT && IT % 4 == 0, "4, 8 or 16 slots a thread");
  static constexpr int kRun = IT + 4;                       // words from run to run
  static constexpr int kLogBins = log2c(2 * kCap);
  static_assert((1 << kLogBins) == 2 * kCap, "two bins per slot");
  static constexpr int kMulti = NT * kRun + 4;              // word of the list
  // pairs, counters, the end of the last bin, the list
  static constexpr size_t kSmem =
      (size_t)kCap * 12 + (size_t)NT * kRun * 4 + 16 + (size_t)kCap;
  // halfword of bin b's counter
  static __device__ __forceinline__ uint32_t half_of(uint32_t b) {
    return b + ((b >> (kLogIt + 1)) << 3);
  }
  // halfword of the bin after the one at halfword h
  static __device__ __forceinline__ uint32_t next_half(uint32_t h) {
    return h % (2 * kRun) == 2 * IT - 1 ? h + 9 : h + 1;
  }
};

// Runs fn(r) for every slot r of a thread that some thread of the CTA fills
// (m pairs, slot r holding element r*NT + tid), four slots per uniform branch.
template <int NT, int IT, typename Fn>
__device__ __forceinline__ void for_slots(uint32_t m, Fn fn) {
#pragma unroll
  for (int q = 0; q < IT; q += 4) {
    if (q == 0 || m > (uint32_t)(q * NT)) {
#pragma unroll
      for (int r = q; r < q + 4; ++r)
        if (r * NT + threadIdx.x < m) fn(r);
    }
  }
}

// Minimum and maximum of a 64-bit value over a warp: the high words, then the
// low words of the lanes that hold the extreme high word (four redux instead of
// twenty shuffles).
__device__ __forceinline__ uint64_t warp_min_u64(uint64_t v) {
  const uint32_t h = __reduce_min_sync(0xffffffffu, (uint32_t)(v >> 32));
  const uint32_t l =
      __reduce_min_sync(0xffffffffu, (uint32_t)(v >> 32) == h ? (uint32_t)v : 0xffffffffu);
  return ((uint64_t)h << 32) | l;
}
__device__ __forceinline__ uint64_t warp_max_u64(uint64_t v) {
  const uint32_t h = __reduce_max_sync(0xffffffffu, (uint32_t)(v >> 32));
  const uint32_t l = __reduce_max_sync(0xffffffffu, (uint32_t)(v >> 32) == h ? (uint32_t)v : 0u);
  return ((uint64_t)h << 32) | l;
}

// Over the CTA, one barrier; red (2 * NT/32 words) may be written again after
// the next barrier.
template <int NT>
__device__ __forceinline__ void block_minmax_u64(uint64_t& mn, uint64_t& mx, uint64_t* red) {
  constexpr int NW = NT / 32;
  const int lane = threadIdx.x & 31, w = threadIdx.x >> 5;
  mn = warp_min_u64(mn);
  mx = warp_max_u64(mx);
  if (lane == 0) {
    red[2 * w] = mn;
    red[2 * w + 1] = mx;
  }
  __syncthreads();
  mn = warp_min_u64(lane < NW ? red[2 * lane] : ~0ULL);
  mx = warp_max_u64(lane < NW ? red[2 * lane + 1] : 0ULL);
}

// After a sort in which the positions stood in for keys that were all equal
// to key_all: writes that key back into the sorted slots.
template <int NT>
__device__ __forceinline__ void restore_common_key(const CtaSortSmem& s, uint32_t m, int by_pos,
                                                   uint64_t key_all) {
  if (!by_pos) return;
  for (uint32_t t = threadIdx.x; t < m; t += NT) s.k[t] = key_all;
  __syncthreads();
}

// Adds the m elements of a bucket to the counter of the algorithm that sorted
// it (algo: kNumAlgos counters, or nullptr when nobody counts).
__device__ __forceinline__ void count_algo(uint64_t* algo, int which, uint32_t m) {
  if (algo && threadIdx.x == 0) atomicAdd((unsigned long long*)&algo[which], (unsigned long long)m);
}

// One compare-exchange of a bitonic network between two registers: the
// smaller pair ends in (ka, ia) when up, in (kb, ib) otherwise.
__device__ __forceinline__ void bitonic_swap(uint64_t& ka, uint32_t& ia, uint64_t& kb, uint32_t& ib,
                                             bool up) {
  if (pair_less(kb, ib, ka, ia) == up) {
    const uint64_t tk = ka;
    const uint32_t ti = ia;
    ka = kb;
    ia = ib;
    kb = tk;
    ib = ti;
  }
}

// Bitonic sort of the m pairs in s.k / s.i, padded to NT*ITEMS, in registers:
// thread t holds positions [t*ITEMS, (t+1)*ITEMS), strides below ITEMS are
// exchanges between a thread's own registers, strides below 32*ITEMS shuffles inside a warp, and
// only longer ones pass through shared memory (6 of the 78 steps of 4096
// pairs), where a thread's pairs sit NT apart so that no bank conflicts.  The
// sorted pairs end in s.k / s.i.
//   Bound by the shuffles (three words per pair and step); the network over
//   shared memory alone pays two barriers and four random accesses per pair
//   and step.
template <int NT, int ITEMS>
__device__ __noinline__ void cta_bitonic_regs(uint32_t m, CtaSortSmem s) {
  const uint32_t tid = threadIdx.x;
  uint64_t key[ITEMS];
  uint32_t idx[ITEMS];
  // (any thread may hold any pair at first)
#pragma unroll
  for (int r = 0; r < ITEMS; ++r) {
    const uint32_t e = r * NT + tid;
    key[r] = e < m ? s.k[e] : ~0ULL;
    idx[r] = e < m ? s.i[e] : ~0u;
  }
  for (uint32_t size = 2; size <= (uint32_t)(NT * ITEMS); size <<= 1) {
    // strides across warps: every pair meets the same register of thread tid ^ d
    for (uint32_t d = size / (2 * ITEMS); d >= 32; d >>= 1) {
      __syncthreads();
#pragma unroll
      for (int r = 0; r < ITEMS; ++r) {
        s.k[r * NT + tid] = key[r];
        s.i[r * NT + tid] = idx[r];
      }
      __syncthreads();
      const bool keep_min = ((tid & d) == 0) == (((tid * ITEMS) & size) == 0);
#pragma unroll
      for (int r = 0; r < ITEMS; ++r) {
        const uint64_t ko = s.k[r * NT + (tid ^ d)];
        const uint32_t io = s.i[r * NT + (tid ^ d)];
        if (pair_less(ko, io, key[r], idx[r]) == keep_min) {
          key[r] = ko;
          idx[r] = io;
        }
      }
    }
    // strides inside a warp
    for (uint32_t d = min(size / (2 * ITEMS), 16u); d >= 1; d >>= 1) {
      const bool keep_min = ((tid & d) == 0) == (((tid * ITEMS) & size) == 0);
#pragma unroll
      for (int r = 0; r < ITEMS; ++r) {
        const uint64_t ko = __shfl_xor_sync(0xffffffffu, key[r], (int)d);
        const uint32_t io = __shfl_xor_sync(0xffffffffu, idx[r], (int)d);
        if (pair_less(ko, io, key[r], idx[r]) == keep_min) {
          key[r] = ko;
          idx[r] = io;
        }
      }
    }
    // strides inside a thread
#pragma unroll
    for (int st = ITEMS / 2; st > 0; st >>= 1) {
      if ((uint32_t)st < size) {
#pragma unroll
        for (int r = 0; r < ITEMS; ++r)
          if ((r & st) == 0)
            bitonic_swap(key[r], idx[r], key[r + st], idx[r + st],
                         ((tid * ITEMS + r) & size) == 0);
      }
    }
  }
  // a thread's consecutive positions go out rotated by its number (32 lanes
  // then hit different banks) and are read back in output order
  __syncthreads();
#pragma unroll
  for (int r = 0; r < ITEMS; ++r) {
    const uint32_t q = tid * ITEMS + ((r + tid) & (ITEMS - 1));
    s.k[q] = key[r];
    s.i[q] = idx[r];
  }
  __syncthreads();
#pragma unroll
  for (int r = 0; r < ITEMS; ++r) {
    const uint32_t e = r * NT + tid, t = e / ITEMS;
    const uint32_t q = t * ITEMS + ((e + t) & (ITEMS - 1));
    key[r] = s.k[q];
    idx[r] = s.i[q];
  }
  __syncthreads();
#pragma unroll
  for (int r = 0; r < ITEMS; ++r) {
    s.k[r * NT + tid] = key[r];
    s.i[r * NT + tid] = idx[r];
  }
  __syncthreads();
}

// Bitonic sort of the m pairs in s.k / s.i (Appendix "Bitonic Sort"), ordered
// by (key, position).  The register network sorts NT*ITEMS pairs; a bucket of at
// most an eighth of that is padded to its own power of two with (UINT64_MAX,
// UINT32_MAX) and sorted in shared memory.
// SIZED: a half or a quarter of NT*ITEMS pairs where they hold the bucket (40,000
// segments of 500 keys, half of them one value: 1485 us with 1024 pairs, 880 with
// 512).  The kernels that rarely come here do without the code of three networks:
// it cost a sort of 2^20 keys 1 us of 75.
template <int NT, int ITEMS, bool SIZED>
__device__ __forceinline__ void cta_bitonic_pairs(uint32_t m, const CtaSortSmem& s) {
  constexpr uint32_t kCap = NT * ITEMS;
  if (m > kCap / 8) {
    if constexpr (SIZED) {
      if (m <= kCap / 4) return cta_bitonic_regs<NT, ITEMS / 4>(m, s);
      if (m <= kCap / 2) return cta_bitonic_regs<NT, ITEMS / 2>(m, s);
    }
    return cta_bitonic_regs<NT, ITEMS>(m, s);
  }
  const uint32_t P = next_pow2_u32(m);
  for (uint32_t e = m + threadIdx.x; e < P; e += NT) { s.k[e] = ~0ULL; s.i[e] = ~0u; }
  block_bitonic_sort<NT>(s.k, s.i, (int)P);
}

template <int NT, int IT>
__device__ __forceinline__ void clear_bins(uint32_t* hist) {
  uint4* run = (uint4*)(hist + threadIdx.x * BinSort<NT, IT>::kRun);
#pragma unroll
  for (int q = 0; q < IT / 4; ++q) run[q] = make_uint4(0, 0, 0, 0);
}

// Counts one pair of the bin whose counter is halfword h; returns h << 16 | its
// rank inside the bin.
__device__ __forceinline__ uint32_t count_bin(uint32_t h, uint32_t* hist) {
  const uint32_t sh = (h & 1) << 4;
  const uint32_t old = atomicAdd(&hist[h >> 1], 1u << sh);
  return (h << 16) | ((old >> sh) & 0xffffu);
}

// Exclusive scan of the counters in place (m pairs; each thread its run of
// words, a word's two counts added by one dp2a), one barrier inside; s_sum holds
// NT/32 words.  Returns whether a bin holds kBinLimit pairs or more (the same in
// every thread): one of the high bits of the OR of all counters.  The caller
// synchronises before it reads the starts.
template <int NT, int IT>
__device__ __forceinline__ bool scan_bins(uint32_t* hist, uint32_t m, uint32_t* s_sum) {
  using BS = BinSort<NT, IT>;
  constexpr int NW = NT / 32;
  const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
  uint4* run = (uint4*)(hist + threadIdx.x * BS::kRun);
  uint32_t sum = 0, any = 0;
#pragma unroll
  for (int q = 0; q < IT / 4; ++q) {
    const uint4 v = run[q];
    sum = __dp2a_lo(v.x, 0x0101u, sum);
    sum = __dp2a_lo(v.y, 0x0101u, sum);
    sum = __dp2a_lo(v.z, 0x0101u, sum);
    sum = __dp2a_lo(v.w, 0x0101u, sum);
    any |= v.x | v.y | v.z | v.w;
  }
  uint32_t inc = sum;
#pragma unroll
  for (int o = 1; o < 32; o <<= 1) {
    const uint32_t y = __shfl_up_sync(0xffffffffu, inc, o);
    if (lane >= o) inc += y;
  }
  static_assert((kBinLimit & (kBinLimit - 1)) == 0, "the crowd test reads high bits");
  constexpr uint32_t kHigh = 0xffffu & ~(uint32_t)(kBinLimit - 1);
  const bool crowd = __any_sync(0xffffffffu, (any & (kHigh | (kHigh << 16))) != 0);
  if (lane == 31) s_sum[warp] = inc | (crowd ? 0x80000000u : 0u);
  __syncthreads();
  uint32_t pre = 0, all = 0;
#pragma unroll
  for (int w = 0; w < NW; ++w) {
    const uint32_t v = s_sum[w];
    pre += w < warp ? v : 0u;
    all |= v;
  }
  uint32_t at = (pre & 0xffffu) + inc - sum;  // (the sums' crowd flags fall away)
#pragma unroll
  for (int q = 0; q < IT / 4; ++q) {
    uint4 v = run[q];
    auto step = [&](uint32_t& w) {
      const uint32_t c = w;
      w = at * 0x10001u + (c << 16);
      at = __dp2a_lo(c, 0x0101u, at);
    };
    step(v.x);
    step(v.y);
    step(v.z);
    step(v.w);
    run[q] = v;
  }
  if (threadIdx.x == NT - 1) ((uint16_t*)hist)[NT * BS::kRun * 2] = (uint16_t)m;
  return (all >> 31) != 0;
}

// Counting-sort scatter of the pairs into their bins; the second one to land in
// a bin puts the bin on the list of bins that still need ordering.
template <int NT, int IT>
__device__ __forceinline__ void place_in_bins(const uint64_t (&key)[IT], const uint32_t (&idx)[IT],
                                              const uint32_t (&hr)[IT], uint32_t m,
                                              const CtaSortSmem& s, uint32_t* nmulti) {
  const uint16_t* half = (const uint16_t*)s.hist;
  uint16_t* multi = (uint16_t*)(s.hist + BinSort<NT, IT>::kMulti);
  for_slots<NT, IT>(m, [&](int r) {
    const uint32_t h = hr[r] >> 16, o = hr[r] & 0xffffu;
    const uint32_t p = half[h] + o;
    s.k[p] = key[r];
    s.i[p] = idx[r];
    if (o == 1) multi[atomicAdd(nmulti, 1u)] = (uint16_t)h;
  });
}

// Orders every listed bin in place by insertion (fewer than kBinLimit pairs; one
// alone in its bin is already in its final slot).
template <int NT, int IT>
__device__ __forceinline__ void order_bins(const CtaSortSmem& s, uint32_t nmulti) {
  const uint16_t* half = (const uint16_t*)s.hist;
  const uint16_t* multi = (const uint16_t*)(s.hist + BinSort<NT, IT>::kMulti);
  for (uint32_t j = threadIdx.x; j < nmulti; j += NT) {
    const uint32_t h = multi[j];
    const uint32_t lo = half[h], cnt = half[BinSort<NT, IT>::next_half(h)] - lo;
    uint64_t* bk = s.k + lo;
    uint32_t* bi = s.i + lo;
    for (uint32_t a = 1; a < cnt; ++a) {
      const uint64_t ka = bk[a];
      const uint32_t ia = bi[a];
      uint32_t q = a;
      while (q > 0 && pair_less(ka, ia, bk[q - 1], bi[q - 1])) {
        bk[q] = bk[q - 1];
        bi[q] = bi[q - 1];
        --q;
      }
      bk[q] = ka;
      bi[q] = ia;
    }
  }
}

// Sorts the m pairs in s.k / s.i when their equal-width bins over [mn, mx]
// (bin = (key - mn) >> shift; s.hist holds the scanned counters) are crowded.
// The bins are refined once: bin b, whose c elements start at slot lo, is cut
// into 2c equal parts numbered from 2 lo, so the 2m parts of all bins fit the
// counters, are in key order, and follow the keys' density.  A key's part is
// its offset in the bin times 2c over the bin's width 2^shift; where the bins
// are one key wide (shift 0: copies of a few neighbouring keys) it is the
// offset of its position in the range of all positions.  A part that is
// crowded still (copies of keys far apart, or keys in a cluster far narrower
// than a bin) sends the bucket to the bitonic sort.  Returns the algorithm that
// finished.  Not inlined: it would cost the common path registers.
//   One rsort_sort of 3001 normal float64 keys, by the bitonic network over
//   shared memory and six launches: 90 us; with refined bins and one launch
//   (k_direct_sort): 9.6 us.
template <int NT, int ITEMS, bool SIZED>
__device__ __noinline__ int cta_sort_crowded(uint32_t m, uint64_t mn, int shift, CtaSortSmem s,
                                             uint32_t* s_sum, uint64_t* red) {
  using BS = BinSort<NT, ITEMS>;
  const uint32_t tid = threadIdx.x;
  {
    __shared__ uint32_t s_nmulti;
    const uint16_t* half = (const uint16_t*)s.hist;
    uint64_t key[ITEMS];
    uint32_t idx[ITEMS], hr[ITEMS];
    uint64_t imn = ~0ULL, imx = 0;
    for_slots<NT, ITEMS>(m, [&](int r) {
      const uint32_t e = r * NT + tid;
      key[r] = s.k[e];
      idx[r] = s.i[e];
      imn = idx[r] < imn ? idx[r] : imn;
      imx = idx[r] > imx ? idx[r] : imx;
    });
    int pshift = 0;  // positions' range in bits, when they order the parts
    if (shift == 0) {
      block_minmax_u64<NT>(imn, imx, red);
      pshift = imx > imn ? 64 - __clzll((long long)(imx - imn)) : 1;
    }
    for_slots<NT, ITEMS>(m, [&](int r) {
      const uint32_t h = BS::half_of((uint32_t)((key[r] - mn) >> shift));
      const uint32_t lo = half[h], c = half[BS::next_half(h)] - lo;
      const uint64_t off = shift ? (key[r] - mn) << (64 - shift)
                                 : ((uint64_t)idx[r] - imn) << (64 - pshift);
      hr[r] = BS::half_of(2 * lo + (uint32_t)__umul64hi(off, (uint64_t)(2 * c)));
    });
    if (tid == 0) s_nmulti = 0;
    __syncthreads();
    clear_bins<NT, ITEMS>(s.hist);
    __syncthreads();
    for_slots<NT, ITEMS>(m, [&](int r) { hr[r] = count_bin(hr[r], s.hist); });
    __syncthreads();
    const bool crowd = scan_bins<NT, ITEMS>(s.hist, m, s_sum);
    __syncthreads();
    if (!crowd) {
      place_in_bins<NT, ITEMS>(key, idx, hr, m, s, &s_nmulti);
      __syncthreads();
      order_bins<NT, ITEMS>(s, s_nmulti);
      __syncthreads();
      return kAlgoBins;
    }
  }
  cta_bitonic_pairs<NT, ITEMS, SIZED>(m, s);
  return kAlgoBitonic;
}

// Sorts the m pairs; on return s.k[0..m) / s.i[0..m) hold them in order.
// in_position_order() says whether the elements arrive with increasing
// positions; it is asked only when all keys are equal.  algo (nullable) gets
// m added to the counter of the branch taken (kAlgoRank, kAlgoInOrder,
// kAlgoBitonic or kAlgoBins).  rank_max bounds rank-by-counting (at most NT
// elements: one per thread); force_bitonic sorts every larger bucket by
// bitonic sort instead of the bins; SIZED: see cta_bitonic_pairs.
template <int NT, int ITEMS, bool SIZED = false, typename InOrderFn>
__device__ void cta_sort_pairs(uint64_t (&key)[ITEMS], uint32_t (&idx)[ITEMS], uint32_t m,
                               InOrderFn in_position_order, const CtaSortSmem& s, uint64_t* red,
                               uint64_t* scan_sm, uint64_t* algo, uint32_t rank_max = kRankMax,
                               bool force_bitonic = false) {
  const uint32_t tid = threadIdx.x;
  if (m <= rank_max && m <= (uint32_t)NT) {
    count_algo(algo, kAlgoRank, m);
#pragma unroll
    for (int r = 0; r < ITEMS; ++r) {
      const uint32_t e = r * NT + tid;
      if (e < m) { s.k[e] = key[r]; s.i[e] = idx[r]; }
    }
    __syncthreads();
    uint32_t rank = 0;
    if (tid < m) {
      for (uint32_t q = 0; q < m; ++q) rank += pair_less(s.k[q], s.i[q], key[0], idx[0]) ? 1u : 0u;
    }
    __syncthreads();
    if (tid < m) { s.k[rank] = key[0]; s.i[rank] = idx[0]; }
    __syncthreads();
    return;
  }
  if (force_bitonic) {
    count_algo(algo, kAlgoBitonic, m);
#pragma unroll
    for (int r = 0; r < ITEMS; ++r) {
      const uint32_t e = r * NT + tid;
      if (e < m) { s.k[e] = key[r]; s.i[e] = idx[r]; }
    }
    __syncthreads();
    cta_bitonic_pairs<NT, ITEMS, SIZED>(m, s);
#pragma unroll
    for (int r = 0; r < ITEMS; ++r) {
      key[r] = 0;
      idx[r] = 0;
    }
    return;
  }
  uint64_t mn = ~0ULL, mx = 0;
  for_slots<NT, ITEMS>(m, [&](int r) {
    mn = key[r] < mn ? key[r] : mn;
    mx = key[r] > mx ? key[r] : mx;
  });
  block_minmax_u64<NT>(mn, mx, red);
  if (mn == mx && in_position_order()) {
    count_algo(algo, kAlgoInOrder, m);
#pragma unroll
    for (int r = 0; r < ITEMS; ++r) {
      const uint32_t e = r * NT + tid;
      if (e < m) { s.k[e] = key[r]; s.i[e] = idx[r]; }
    }
    __syncthreads();
    return;
  }
  // all keys equal, in no particular order: (key, position) order is the
  // order of the positions, so the positions (distinct) stand in for the
  // keys below and the common key is put back at the end
  __shared__ uint64_t s_key_all;
  __shared__ int s_by_pos;
  if (tid == 0) {
    s_by_pos = mn == mx;
    s_key_all = mn;
  }
  if (mn == mx) {
    __syncthreads();  // (red is written again)
    mn = ~0ULL;
    mx = 0;
    for_slots<NT, ITEMS>(m, [&](int r) {
      key[r] = idx[r];
      mn = key[r] < mn ? key[r] : mn;
      mx = key[r] > mx ? key[r] : mx;
    });
    block_minmax_u64<NT>(mn, mx, red);
  }
  // equal-width bins over [mn, mx]
  using BS = BinSort<NT, ITEMS>;
  uint32_t* s_sum = (uint32_t*)scan_sm;
  const uint64_t range = mx - mn;
  const int bits = range ? 64 - __clzll((long long)range) : 0;
  const int shift = bits > BS::kLogBins ? bits - BS::kLogBins : 0;
  __shared__ uint32_t s_nmulti;
  clear_bins<NT, ITEMS>(s.hist);
  if (tid == 0) s_nmulti = 0;
  __syncthreads();
  uint32_t hr[ITEMS];
  for_slots<NT, ITEMS>(m, [&](int r) {
    hr[r] = count_bin(BS::half_of((uint32_t)((key[r] - mn) >> shift)), s.hist);
  });
  __syncthreads();
  const bool crowd = scan_bins<NT, ITEMS>(s.hist, m, s_sum);
  if (crowd) {
#pragma unroll
    for (int r = 0; r < ITEMS; ++r) {
      const uint32_t e = r * NT + tid;
      if (e < m) { s.k[e] = key[r]; s.i[e] = idx[r]; }
    }
  }
  __syncthreads();
  if (crowd) {
    const int how = cta_sort_crowded<NT, ITEMS, SIZED>(m, mn, shift, s, s_sum, red);
    // (so that no register of the pairs is kept across the call: a caller's loop
    // would keep those of slots it does not load, 32 bytes spilled or 124)
#pragma unroll
    for (int r = 0; r < ITEMS; ++r) {
      key[r] = 0;
      idx[r] = 0;
    }
    count_algo(algo, how, m);
    restore_common_key<NT>(s, m, s_by_pos, s_key_all);
    return;
  }
  count_algo(algo, kAlgoBins, m);
  place_in_bins<NT, ITEMS>(key, idx, hr, m, s, &s_nmulti);
  __syncthreads();
  order_bins<NT, ITEMS>(s, s_nmulti);
  __syncthreads();
  restore_common_key<NT>(s, m, s_by_pos, s_key_all);
}

}  // namespace rsort
