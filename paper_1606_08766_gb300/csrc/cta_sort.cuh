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
//                       2 * next_pow2(m) equal-width bins (a counting sort in
//                       shared memory), then order each bin that holds
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
  uint32_t* hist;  // [cap + cap/4 + cap/2]  up to 2*cap 16-bit bin counters
                   //   packed in pairs (one pad word after every thread's run
                   //   of counter words), then the list of bins holding
                   //   several elements
};

// Shared memory per element of capacity that a CtaSortSmem needs.
constexpr int kCtaSortBytesPerElem = 8 + 4 + 4 + 1 + 2;

// Counter word w of a scan in which every thread owns 2^lp consecutive words
// sits at w + (w >> lp): each thread's run starts one bank further on, so the
// lanes of a warp walking their runs in step hit distinct banks.
__device__ __forceinline__ uint32_t padded_word(uint32_t w, int lp) { return w + (w >> lp); }

template <int NT>
__device__ __forceinline__ void block_minmax_u64(uint64_t& mn, uint64_t& mx, uint64_t* red) {
  const int lane = threadIdx.x & 31, w = threadIdx.x >> 5;
#pragma unroll
  for (int o = 16; o > 0; o >>= 1) {
    const uint64_t a = __shfl_xor_sync(0xffffffffu, mn, o);
    const uint64_t b = __shfl_xor_sync(0xffffffffu, mx, o);
    mn = a < mn ? a : mn;
    mx = b > mx ? b : mx;
  }
  if (lane == 0) {
    red[2 * w] = mn;
    red[2 * w + 1] = mx;
  }
  __syncthreads();
  mn = red[0];
  mx = red[1];
#pragma unroll
  for (int q = 1; q < NT / 32; ++q) {
    mn = red[2 * q] < mn ? red[2 * q] : mn;
    mx = red[2 * q + 1] > mx ? red[2 * q + 1] : mx;
  }
  __syncthreads();
}

__device__ __forceinline__ uint32_t bin_start(const uint32_t* hist, uint32_t b, int lp) {
  return (hist[padded_word(b >> 1, lp)] >> ((b & 1) << 4)) & 0xffffu;
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
// by (key, position).  The register network always sorts NT*ITEMS pairs; a
// bucket of at most an eighth of that is padded to its own power of two with
// (UINT64_MAX, UINT32_MAX) and sorted in shared memory.
template <int NT, int ITEMS>
__device__ __forceinline__ void cta_bitonic_pairs(uint32_t m, const CtaSortSmem& s) {
  if (m > (uint32_t)(NT * ITEMS / 8)) {
    cta_bitonic_regs<NT, ITEMS>(m, s);
    return;
  }
  const uint32_t P = next_pow2_u32(m);
  for (uint32_t e = m + threadIdx.x; e < P; e += NT) { s.k[e] = ~0ULL; s.i[e] = ~0u; }
  block_bitonic_sort<NT>(s.k, s.i, (int)P);
}

// Layout of a bucket's bin counters: nb 16-bit counters packed in words, each
// thread scanning a run of 2^lp of them.
struct BinShape {
  uint32_t nb, words, per;
  int lp;
};

template <int NT>
__device__ __forceinline__ BinShape bin_shape(uint32_t m) {
  BinShape g;
  g.nb = 2 * next_pow2_u32(m);
  g.words = g.nb / 2;
  g.per = (g.words + NT - 1) / NT;  // a power of two
  g.lp = log2_u32(g.per);
  return g;
}

template <int NT>
__device__ __forceinline__ void clear_bins(const BinShape& g, uint32_t* hist) {
  for (uint32_t w = threadIdx.x; w < g.words + (g.words >> g.lp); w += NT) hist[w] = 0;
}

// Counts one element of bin b; returns bin << 16 | rank inside the bin.
__device__ __forceinline__ uint32_t count_bin(uint32_t b, const BinShape& g, uint32_t* hist) {
  const uint32_t sh = (b & 1) << 4;
  const uint32_t old = atomicAdd(&hist[padded_word(b >> 1, g.lp)], 1u << sh);
  return (b << 16) | ((old >> sh) & 0xffffu);
}

// Exclusive scan of the counters in place (each thread a run of words), which
// also finds out whether any bin is crowded (the same answer in every thread).
template <int NT>
__device__ __forceinline__ bool scan_bins(const BinShape& g, uint32_t* hist, uint64_t* scan_sm) {
  const uint32_t w0 = threadIdx.x * g.per;
  bool crowd = false;
  uint32_t loc = 0;
  for (uint32_t w = w0; w < w0 + g.per && w < g.words; ++w) {
    const uint32_t v = hist[padded_word(w, g.lp)];
    const uint32_t a = v & 0xffffu, b = v >> 16;
    loc += a + b;
    crowd |= a > (uint32_t)kBinLimit || b > (uint32_t)kBinLimit;
  }
  uint64_t tot;
  uint32_t run = (uint32_t)block_excl_scan_u64<NT>(loc, &tot, scan_sm);
  for (uint32_t w = w0; w < w0 + g.per && w < g.words; ++w) {
    const uint32_t pw = padded_word(w, g.lp);
    const uint32_t v = hist[pw];
    const uint32_t lo = run, hi = run + (v & 0xffffu);
    hist[pw] = lo | (hi << 16);
    run = hi + (v >> 16);
  }
  return __syncthreads_or(crowd);
}

// Counting-sort scatter of the pairs into their bins; the second element to
// land in a bin puts the bin on the list of bins that still need ordering.
template <int NT, int ITEMS>
__device__ __forceinline__ void place_in_bins(const uint64_t (&key)[ITEMS],
                                              const uint32_t (&idx)[ITEMS],
                                              const uint32_t (&bs)[ITEMS], uint32_t m,
                                              const BinShape& g, const CtaSortSmem& s,
                                              uint32_t* nmulti) {
  constexpr uint32_t kCap = NT * ITEMS;
  uint32_t* multi = s.hist + kCap + kCap / 4;
#pragma unroll
  for (int r = 0; r < ITEMS; ++r) {
    if (r * NT + threadIdx.x < m) {
      const uint32_t b = bs[r] >> 16, o = bs[r] & 0xffffu;
      const uint32_t p = bin_start(s.hist, b, g.lp) + o;
      s.k[p] = key[r];
      s.i[p] = idx[r];
      if (o == 1) multi[atomicAdd(nmulti, 1u)] = b;
    }
  }
}

// Orders every listed bin in place by insertion (at most kBinLimit elements;
// an element alone in its bin is already in its final slot).
template <int NT, int ITEMS>
__device__ __forceinline__ void order_bins(uint32_t m, const BinShape& g, const CtaSortSmem& s,
                                           uint32_t nmulti) {
  constexpr uint32_t kCap = NT * ITEMS;
  const uint32_t* multi = s.hist + kCap + kCap / 4;
  for (uint32_t j = threadIdx.x; j < nmulti; j += NT) {
    const uint32_t b = multi[j];
    const uint32_t lo = bin_start(s.hist, b, g.lp);
    const uint32_t hi = b + 1 < g.nb ? bin_start(s.hist, b + 1, g.lp) : m;
    uint64_t* bk = s.k + lo;
    uint32_t* bi = s.i + lo;
    for (uint32_t a = 1; a < hi - lo; ++a) {
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
//   (k_direct_sort): 15 us.
template <int NT, int ITEMS>
__device__ __noinline__ int cta_sort_crowded(uint32_t m, uint64_t mn, int shift, CtaSortSmem s,
                                             uint64_t* scan_sm, uint64_t* red) {
  const uint32_t tid = threadIdx.x;
  {
    const BinShape g = bin_shape<NT>(m);
    __shared__ uint32_t s_nmulti;
    uint64_t key[ITEMS];
    uint32_t idx[ITEMS], bs[ITEMS];
    uint64_t imn = ~0ULL, imx = 0;
#pragma unroll
    for (int r = 0; r < ITEMS; ++r) {
      const uint32_t e = r * NT + tid;
      if (e < m) {
        key[r] = s.k[e];
        idx[r] = s.i[e];
        imn = idx[r] < imn ? idx[r] : imn;
        imx = idx[r] > imx ? idx[r] : imx;
      }
    }
    int pshift = 0;  // positions' range in bits, when they order the parts
    if (shift == 0) {
      block_minmax_u64<NT>(imn, imx, red);
      pshift = imx > imn ? 64 - __clzll((long long)(imx - imn)) : 1;
    }
#pragma unroll
    for (int r = 0; r < ITEMS; ++r) {
      if (r * NT + tid < m) {
        const uint32_t b = (uint32_t)((key[r] - mn) >> shift);
        const uint32_t lo = bin_start(s.hist, b, g.lp);
        const uint32_t hi = b + 1 < g.nb ? bin_start(s.hist, b + 1, g.lp) : m;
        const uint64_t off = shift ? (key[r] - mn) << (64 - shift)
                                   : ((uint64_t)idx[r] - imn) << (64 - pshift);
        bs[r] = 2 * lo + (uint32_t)__umul64hi(off, (uint64_t)(2 * (hi - lo)));
      }
    }
    if (tid == 0) s_nmulti = 0;
    __syncthreads();
    clear_bins<NT>(g, s.hist);
    __syncthreads();
#pragma unroll
    for (int r = 0; r < ITEMS; ++r)
      if (r * NT + tid < m) bs[r] = count_bin(bs[r], g, s.hist);
    __syncthreads();
    if (!scan_bins<NT>(g, s.hist, scan_sm)) {
      place_in_bins<NT, ITEMS>(key, idx, bs, m, g, s, &s_nmulti);
      __syncthreads();
      order_bins<NT, ITEMS>(m, g, s, s_nmulti);
      __syncthreads();
      return kAlgoBins;
    }
  }
  cta_bitonic_pairs<NT, ITEMS>(m, s);
  return kAlgoBitonic;
}

// No-op for cta_sort_pairs' released callback.
struct NoRelease {
  __device__ void operator()() const {}
};

// Sorts the m pairs; on return s.k[0..m) / s.i[0..m) hold them in order.
// in_position_order() says whether the elements arrive with increasing
// positions; it is asked only when all keys are equal.  algo (nullable) gets
// m added to the counter of the branch taken (kAlgoRank, kAlgoInOrder,
// kAlgoBitonic or kAlgoBins).  rank_max bounds rank-by-counting (at most NT
// elements: one per thread); force_bitonic sorts every larger bucket by
// bitonic sort instead of the bins.  released() is called once by every
// thread of the CTA, together, as soon as key[] and idx[] are no longer read
// (the pairs are in shared memory): the caller may then load the next
// bucket into them while this one is finished.
template <int NT, int ITEMS, typename InOrderFn, typename ReleaseFn = NoRelease>
__device__ void cta_sort_pairs(uint64_t (&key)[ITEMS], uint32_t (&idx)[ITEMS], uint32_t m,
                               InOrderFn in_position_order, const CtaSortSmem& s, uint64_t* red,
                               uint64_t* scan_sm, uint64_t* algo, uint32_t rank_max = kRankMax,
                               bool force_bitonic = false, ReleaseFn released = ReleaseFn()) {
  static_assert(ITEMS >= 4, "the padded counters need cap/4 >= NT words of slack");
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
    released();
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
    cta_bitonic_pairs<NT, ITEMS>(m, s);
#pragma unroll
    for (int r = 0; r < ITEMS; ++r) {
      key[r] = 0;
      idx[r] = 0;
    }
    released();
    return;
  }
  uint64_t mn = ~0ULL, mx = 0;
#pragma unroll
  for (int r = 0; r < ITEMS; ++r) {
    if (r * NT + tid < m) {
      mn = key[r] < mn ? key[r] : mn;
      mx = key[r] > mx ? key[r] : mx;
    }
  }
  block_minmax_u64<NT>(mn, mx, red);
  if (mn == mx && in_position_order()) {
    count_algo(algo, kAlgoInOrder, m);
#pragma unroll
    for (int r = 0; r < ITEMS; ++r) {
      const uint32_t e = r * NT + tid;
      if (e < m) { s.k[e] = key[r]; s.i[e] = idx[r]; }
    }
    __syncthreads();
    released();
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
    mn = ~0ULL;
    mx = 0;
#pragma unroll
    for (int r = 0; r < ITEMS; ++r) {
      if (r * NT + tid < m) {
        key[r] = idx[r];
        mn = key[r] < mn ? key[r] : mn;
        mx = key[r] > mx ? key[r] : mx;
      }
    }
    block_minmax_u64<NT>(mn, mx, red);
  }
  // equal-width bins over [mn, mx]
  const BinShape g = bin_shape<NT>(m);  // g.nb <= 2 * kCap
  const int lognb = log2_u32(g.nb);
  const uint64_t range = mx - mn;
  const int bits = range ? 64 - __clzll((long long)range) : 0;
  const int shift = bits > lognb ? bits - lognb : 0;
  clear_bins<NT>(g, s.hist);
  __shared__ uint32_t s_nmulti;
  if (tid == 0) s_nmulti = 0;
  __syncthreads();
  uint32_t bs[ITEMS];
#pragma unroll
  for (int r = 0; r < ITEMS; ++r)
    if (r * NT + tid < m) bs[r] = count_bin((uint32_t)((key[r] - mn) >> shift), g, s.hist);
  __syncthreads();
  if (scan_bins<NT>(g, s.hist, scan_sm)) {
#pragma unroll
    for (int r = 0; r < ITEMS; ++r) {
      const uint32_t e = r * NT + tid;
      if (e < m) { s.k[e] = key[r]; s.i[e] = idx[r]; }
    }
    __syncthreads();
    const int how = cta_sort_crowded<NT, ITEMS>(m, mn, shift, s, scan_sm, red);
    // (no register of the pairs is kept across the call)
#pragma unroll
    for (int r = 0; r < ITEMS; ++r) {
      key[r] = 0;
      idx[r] = 0;
    }
    count_algo(algo, how, m);
    restore_common_key<NT>(s, m, s_by_pos, s_key_all);
    released();
    return;
  }
  count_algo(algo, kAlgoBins, m);
  place_in_bins<NT, ITEMS>(key, idx, bs, m, g, s, &s_nmulti);
  __syncthreads();
  released();
  order_bins<NT, ITEMS>(m, g, s, s_nmulti);
  __syncthreads();
  restore_common_key<NT>(s, m, s_by_pos, s_key_all);
}

}  // namespace rsort
