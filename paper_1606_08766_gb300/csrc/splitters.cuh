// splitters.cuh -- the splitters of a partition step in shared memory and
// the two classifiers that search them (Appendix "Robust Multi-Level Sample
// Sort" of Axtmann & Sanders: the Super Scalar Sample Sort classifier, with
// the search repeated on a key tie using positions as tie-breakers).
//
// Shared by the classify / scatter kernels of every level.
#pragma once

#include "rsort_internal.cuh"

namespace rsort {

// Index of the last segment whose field is <= x (segments sorted by field).
template <typename F>
__device__ __forceinline__ uint32_t find_seg(const LevelSeg* segs, uint32_t G, uint64_t x,
                                             F field) {
  uint32_t lo = 0, hi = G;
  while (lo < hi) {
    const uint32_t mid = (lo + hi) >> 1;
    if (field(segs[mid]) <= x) lo = mid + 1; else hi = mid;
  }
  return lo - 1;
}

// Segment of chunk c: the map that the plan wrote (chunk_seg), one dependent
// load where a binary search over the segments' first chunks took log2 G of
// them, ~0.6 us each and exposed once per chunk (33,000 segments of one chunk:
// level-1 scatter 2.77 -> 2.27 ms).
__device__ __forceinline__ uint32_t seg_of_chunk(const uint32_t* chunk_seg, uint32_t G,
                                                 uint64_t c) {
  return G == 1 ? 0u : __ldg(chunk_seg + c);
}

__device__ __forceinline__ uint32_t ceil_log2_dev(uint32_t k) {
  uint32_t l = 0;
  while ((1u << l) < k) ++l;
  return l;
}

// An ordinary load: the sample's is in a call's first launch (k_sample_sort), which
// may be set up while the launch before it still writes these keys (the last call's
// output, sorted again), and a load through the read-only path is allowed only where
// the data does not change while the kernel is resident.  The kernels that read keys
// through that path start two launches later or more, when the keys are complete.
__device__ __forceinline__ uint64_t load_key(const Src& s, uint64_t pos) {
  const uint64_t k = s.key[pos];
  return s.map_f64 ? f64_to_ordered(k) : k;
}

// ---------------------------------------------------------------------------
// Splitter structures in shared memory
//
// The k-1 splitters of a segment are the sorted sample's elements
// floor(j*S/k), j = 1..k-1 (Appendix "Generalizing Quicksort": every S/k-th
// sample), kept as sorted (key, position) pairs.  Two classifiers search them,
// both returning the same bucket:
//   tree   the branchless implicit search tree of Super Scalar Sample Sort that
//          the appendix names: the keys in Eytzinger order, padded with
//          UINT64_MAX to Kp - 1 = next_pow2(k) - 1 nodes;
//   table  a lookup table of 4 to 8 bins per splitter over the leading bits of
//          (key - smallest splitter key) giving every bin's first splitter; a
//          key steps from there to the first splitter that is not smaller, one
//          or two reads, as long as no bin holds more than kLinearMax; else it
//          searches its bin's splitters by halving.  float64 keys, whose bit
//          patterns crowd a few octaves of a range of thousands, get bins of
//          equal width in value instead where that keeps them small (2*10^7
//          normal keys, 512 buckets: 194 us with 150 splitters in a bin, 81).
// A key equal to splitter keys is then placed among the run of those
// splitters by its position (tie_break).
// ---------------------------------------------------------------------------
constexpr int kTableBitsMax = 13;
constexpr uint32_t kLinearMax = 6;

struct Splitters {
  uint64_t* tree;   // [Kp]   node i at tree[i], i = 1..Kp-1          (tree mode)
  uint16_t* tbl;    // [2^tbits] first splitter of a bin (table mode)
  uint64_t* key;    // [k]    sorted splitter keys, then UINT64_MAX
  uint32_t* idx;    // [k-1]  their positions (tie-breakers)
  uint16_t* rend;   // [k-1]  end of the run of splitters whose key equals key[j]
  uint64_t lo, hi;  // smallest / largest splitter key
  int logK;         // log2(Kp)
  int tbits;        // table bits
  uint32_t tmax;    // last table entry (2^tbits - 1)
  int shift;        // key bits dropped before the table index
  int linear;       // 1: no bin holds more than kLinearMax splitters
  int by_value;     // 1: bins of equal width in float64 value
  float flo, fscale;  // value of the smallest splitter, bins per unit
  int mode;         // 0 tree, 1 table
  int ntb;          // 1: no tie-breaking, classify by key only (ablation)
  uint32_t nspl;    // k - 1
};

__host__ __device__ inline int table_bits_for(uint32_t kp) {
  const int b = log2_u32(kp) + 2;
  return b < kTableBitsMax ? b : kTableBitsMax;
}
__host__ __device__ inline size_t table_bytes(uint32_t kp) {
  return (size_t)2 << table_bits_for(kp);
}

// Bin of a key in the table.  Monotone in the key either way: the conversion to
// float, the subtraction and the product round monotonically, and the keys
// beyond the largest splitter (infinities and NaNs among them) take the last
// bin.
__device__ __forceinline__ uint32_t bin_by_bits(uint64_t x, const Splitters& sp) {
  const uint64_t t = (x > sp.lo ? x - sp.lo : 0ull) >> sp.shift;
  return t < sp.tmax ? (uint32_t)t : sp.tmax;
}
__device__ __forceinline__ uint32_t bin_by_value(uint64_t x, const Splitters& sp) {
  const float v = (float)__longlong_as_double((long long)ordered_to_f64(x));
  const uint32_t t = __float2uint_rz(__fmul_rn(__fsub_rn(v, sp.flo), sp.fscale));
  return x > sp.hi || t > sp.tmax ? sp.tmax : t;
}

// Fills the table by a histogram of the splitters' bins and its exclusive scan;
// returns the largest bin's splitters (the same in every thread).
template <int NT, typename BinFn>
__device__ __forceinline__ uint32_t build_table(const Splitters& sp, BinFn bin_of) {
  __shared__ uint32_t s_scan[NT / 32];
  __shared__ uint32_t s_max;
  const uint32_t words = (sp.tmax + 1) / 2;
  uint32_t* w = reinterpret_cast<uint32_t*>(sp.tbl);
  const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
  for (uint32_t q = threadIdx.x; q < words; q += NT) w[q] = 0;
  if (threadIdx.x == 0) s_max = 0;
  __syncthreads();
  for (uint32_t j = threadIdx.x; j < sp.nspl; j += NT) {
    const uint32_t t = bin_of(sp.key[j]);
    atomicAdd(&w[t >> 1], 1u << ((t & 1) << 4));
  }
  __syncthreads();
  const uint32_t per = (words + NT - 1) / NT;
  const uint32_t q0 = min(threadIdx.x * per, words), q1 = min(q0 + per, words);
  uint32_t sum = 0, most = 0;
  for (uint32_t q = q0; q < q1; ++q) {
    const uint32_t a = w[q] & 0xffffu, b = w[q] >> 16;
    sum += a + b;
    most = max(most, max(a, b));
  }
  uint32_t inc = sum;
#pragma unroll
  for (int o = 1; o < 32; o <<= 1) {
    const uint32_t y = __shfl_up_sync(0xffffffffu, inc, o);
    if (lane >= o) inc += y;
  }
  most = __reduce_max_sync(0xffffffffu, most);
  if (lane == 31) s_scan[warp] = inc;
  if (lane == 0) atomicMax(&s_max, most);
  __syncthreads();
  uint32_t at = inc - sum;
  for (int q = 0; q < warp; ++q) at += s_scan[q];
  for (uint32_t q = q0; q < q1; ++q) {
    const uint32_t a = w[q] & 0xffffu, b = w[q] >> 16;
    w[q] = at | ((at + a) << 16);
    at += a + b;
  }
  most = s_max;
  __syncthreads();
  return most;
}

// F64: the keys are mapped float64 patterns (bins by value are tried).
template <int NT, bool F64 = false>
__device__ void load_splitters(const LevelSeg& sg, const uint64_t* ssk, const uint32_t* ssi,
                               Splitters& sp) {
  const uint32_t k = sg.k;
  const uint32_t Kp = next_pow2_u32(k);
  sp.nspl = k - 1;
  sp.logK = log2_u32(Kp);
  // (j + 1) S < 2^32: at most kMaxFine splitters of 16 * 11 * kMaxK samples
  static_assert((uint64_t)kMaxFine * 16 * 11 * kMaxK < (1ull << 32), "32-bit sample ranks");
  for (uint32_t j = threadIdx.x; j < sp.nspl; j += NT) {
    const uint32_t r = (j + 1) * sg.S / k;
    sp.key[j] = ssk[sg.samp_off + r];
    sp.idx[j] = ssi[sg.samp_off + r];
  }
  if (threadIdx.x == 0) sp.key[sp.nspl] = ~0ULL;
  __syncthreads();
  // end of every run of equal splitter keys (keys are sorted, so the run of
  // key[j] is contiguous); tie-breaks search positions inside the run only
  for (uint32_t j = threadIdx.x; j < sp.nspl; j += NT) {
    const uint64_t kj = sp.key[j];
    uint32_t lo = j + 1, hi = sp.nspl;
    if (lo < hi && sp.key[lo] != kj) hi = lo;
    while (lo < hi) {
      const uint32_t mid = (lo + hi) >> 1;
      if (sp.key[mid] == kj) lo = mid + 1; else hi = mid;
    }
    sp.rend[j] = (uint16_t)lo;
  }
  sp.by_value = 0;
  if (sp.mode == 0) {
    for (uint32_t i = threadIdx.x + 1; i < Kp; i += NT) {
      const int d = 31 - __clz(i);
      const uint32_t r = i - (1u << d);
      const uint32_t in = ((2 * r + 1) << (sp.logK - 1 - d)) - 1;
      sp.tree[i] = in < sp.nspl ? sp.key[in] : ~0ULL;
    }
  } else if (sp.nspl > 0) {
    sp.lo = sp.key[0];
    sp.hi = sp.key[sp.nspl - 1];
    const uint64_t range = sp.hi - sp.lo;
    const int bits = range ? 64 - __clzll((long long)range) : 0;
    sp.tbits = table_bits_for(Kp);
    sp.shift = bits > sp.tbits ? bits - sp.tbits : 0;
    sp.tmax = (1u << sp.tbits) - 1;
    uint32_t most = build_table<NT>(sp, [&](uint64_t x) { return bin_by_bits(x, sp); });
    if (F64 && most > kLinearMax) {
      const double vlo = __longlong_as_double((long long)ordered_to_f64(sp.lo));
      const double vhi = __longlong_as_double((long long)ordered_to_f64(sp.hi));
      const float flo = (float)vlo, fscale = (float)(sp.tmax + 1) / ((float)vhi - flo);
      // (finite values, and a finite scale; NaNs fail every comparison)
      if (vlo > -1e37 && vhi < 1e37 && fscale > 0.0f && fscale < 1e37f) {
        sp.flo = flo;
        sp.fscale = fscale;
        const uint32_t mv = build_table<NT>(sp, [&](uint64_t x) { return bin_by_value(x, sp); });
        if (mv <= kLinearMax || 2 * mv < most) {
          sp.by_value = 1;
          most = mv;
        } else {
          build_table<NT>(sp, [&](uint64_t x) { return bin_by_bits(x, sp); });
        }
      }
    }
    sp.linear = most <= kLinearMax;
  } else {
    // no splitters: one bin, empty, so every key lands in bucket 0
    sp.lo = 0;
    sp.hi = 0;
    sp.tbits = 0;
    sp.tmax = 0;
    sp.shift = 0;
    sp.linear = 0;
    if (threadIdx.x == 0) sp.tbl[0] = 0;
  }
  __syncthreads();
}

// Bucket of element (x, i): the number of splitters lexicographically smaller
// than (x, i).  R elements descend the tree level by level together (R
// independent shared-memory loads in flight per level).  The descent counts
// the splitters whose key is smaller than x and remembers the key of the last
// node where it turned left, which is the bounding splitter's key; only if x
// equals it is the search repeated on the run of equal splitter keys with
// positions as tie-breakers (pos_of(r) is evaluated only then).
//
// The splitters whose key is x are [bb, rend[bb]), in increasing position;
// the bucket is bb plus the number of them placed before position i.  A long
// run (many copies of one key) holds positions of a stratified sample, close
// to evenly spaced: the search starts at an interpolated guess and gallops
// to a bracket around the answer, a few steps instead of log2 of the run.
__device__ __forceinline__ uint32_t tie_break(uint32_t lo, uint32_t hi, uint32_t i,
                                              const Splitters& sp) {
  if (hi - lo > 8) {
    const uint32_t p0 = sp.idx[lo], p1 = sp.idx[hi - 1];
    if (i <= p0) return lo;
    if (i > p1) return hi;
    // now idx[lo] < i <= idx[hi - 1]: the answer is in (lo, hi - 1]
    const float f = __fdividef((float)(i - p0) * (float)(hi - 1 - lo), (float)(p1 - p0));
    uint32_t g = lo + (uint32_t)f;
    g = g < lo + 1 ? lo + 1 : (g > hi - 1 ? hi - 1 : g);
    uint32_t a, b;  // idx[a] < i <= idx[b]
    if (sp.idx[g] < i) {
      a = g;
      uint32_t d = 1;
      while (a + d < hi - 1 && sp.idx[a + d] < i) {
        a += d;
        d <<= 1;
      }
      b = a + d < hi - 1 ? a + d : hi - 1;
    } else {
      b = g;
      uint32_t d = 1;
      while (b - lo > d && sp.idx[b - d] >= i) {
        b -= d;
        d <<= 1;
      }
      a = b - lo > d ? b - d : lo;
    }
    lo = a + 1;
    hi = b;
  }
  while (lo < hi) {
    const uint32_t mid = (lo + hi) >> 1;
    if (sp.idx[mid] < i) lo = mid + 1; else hi = mid;
  }
  return lo;
}

// The band of every run of splitters for a chunk of positions [p0, p1] (level 1,
// whose positions rise with the element): band[j], j the run's first splitter,
// holds the buckets of the two positions when their key ties with the run, first |
// last << 16.  A sample puts a run's splitters far apart, so nearly always the two
// are the same and a tie needs no search.  The caller's barrier makes the bands
// visible.
template <int NT>
__device__ __forceinline__ void load_bands(uint32_t p0, uint32_t p1, uint32_t* band,
                                           const Splitters& sp) {
  for (uint32_t j = threadIdx.x; j < sp.nspl; j += NT)
    if (j == 0 || sp.key[j] != sp.key[j - 1])
      band[j] = tie_break(j, sp.rend[j], p0, sp) | (tie_break(j, sp.rend[j], p1, sp) << 16);
}

template <int R, typename PosFn>
__device__ __forceinline__ void classify_batch_tree(const uint64_t (&x)[R], uint32_t (&b)[R],
                                                    PosFn pos_of, const Splitters& sp) {
  uint32_t j[R];
  uint64_t ub[R];
#pragma unroll
  for (int r = 0; r < R; ++r) {
    j[r] = 1;
    ub[r] = ~0ULL;
  }
  for (int l = 0; l < sp.logK; ++l) {
#pragma unroll
    for (int r = 0; r < R; ++r) {
      const uint64_t t = sp.tree[j[r]];
      const bool right = x[r] > t;
      j[r] = 2 * j[r] + (right ? 1u : 0u);
      ub[r] = right ? ub[r] : t;
    }
  }
#pragma unroll
  for (int r = 0; r < R; ++r) {
    uint32_t bb = j[r] - (1u << sp.logK);
    if (!sp.ntb && bb < sp.nspl && ub[r] == x[r]) bb = tie_break(bb, sp.rend[bb], pos_of(r), sp);
    b[r] = bb;
  }
}

// Same result through the table: one table read per element, then the first
// splitter of its bin that is not smaller, step by step where the bins are
// small (usually the first one read) and by halving otherwise.
// PAIRS: elements 2j and 2j+1 sit at consecutive positions whenever
// valid(2j) and valid(2j+1); when both tie with the same run of splitter keys,
// the second element's bucket is the first's or the next: one comparison instead
// of a search.  (Only one splitter position can lie between the two elements,
// but with fewer samples than buckets several splitters share it.)
template <int R, bool PAIRS = false, bool F64 = false, typename PosFn, typename ValidFn>
__device__ __forceinline__ void classify_batch_table(const uint64_t (&x)[R], uint32_t (&b)[R],
                                                     PosFn pos_of, ValidFn valid,
                                                     const Splitters& sp) {
  // A key below the smallest splitter reads bin 0 and one above the largest
  // the last bin: each then finds no splitter on its far side, so no case
  // needs its own branch.
  uint64_t ub[R];  // key of the first splitter that is not smaller
  if (sp.linear) {
    if (F64 && sp.by_value) {
#pragma unroll
      for (int r = 0; r < R; ++r) b[r] = sp.tbl[bin_by_value(x[r], sp)];
    } else {
#pragma unroll
      for (int r = 0; r < R; ++r) b[r] = sp.tbl[bin_by_bits(x[r], sp)];
    }
#pragma unroll
    for (int r = 0; r < R; ++r) ub[r] = sp.key[b[r]];
#pragma unroll
    for (int r = 0; r < R; ++r) {
      // (the key after the last splitter is the largest there is)
      while (ub[r] < x[r]) ub[r] = sp.key[++b[r]];
    }
  } else {
#pragma unroll
    for (int r = 0; r < R; ++r) {
      const uint32_t t = F64 && sp.by_value ? bin_by_value(x[r], sp) : bin_by_bits(x[r], sp);
      uint32_t lo = sp.tbl[t], hi = t < sp.tmax ? (uint32_t)sp.tbl[t + 1] : sp.nspl;
      uint64_t u = sp.key[hi];
      // the bin's first splitter may already bound x (always so when a run of
      // copies of x fills the bin): then no search is needed
      if (lo < hi) {
        const uint64_t k0 = sp.key[lo];
        if (k0 >= x[r]) {
          hi = lo;
          u = k0;
        } else {
          ++lo;
        }
      }
      while (lo < hi) {
        const uint32_t mid = (lo + hi) >> 1;
        const uint64_t km = sp.key[mid];
        if (km < x[r]) {
          lo = mid + 1;
        } else {
          hi = mid;
          u = km;
        }
      }
      b[r] = lo;
      ub[r] = u;
    }
  }
  if (sp.ntb) return;
  bool tie = false;
#pragma unroll
  for (int r = 0; r < R; ++r) tie |= ub[r] == x[r];
  if (!tie) return;
  bool prev_tied = false;
#pragma unroll
  for (int r = 0; r < R; ++r) {
    const bool tied = ub[r] == x[r] && b[r] < sp.nspl;
    if (tied) {
      if (PAIRS && (r & 1) && prev_tied && x[r] == x[r - 1] && valid(r - 1) && valid(r)) {
        const uint32_t re = sp.rend[b[r]], pos = pos_of(r);
        uint32_t pb = b[r - 1];
        while (pb < re && sp.idx[pb] < pos) ++pb;
        b[r] = pb;
      } else {
        b[r] = tie_break(b[r], sp.rend[b[r]], pos_of(r), sp);
      }
    }
    prev_tied = tied;
  }
}

template <int R, typename PosFn>
__device__ __forceinline__ void classify_batch(const uint64_t (&x)[R], uint32_t (&b)[R],
                                               PosFn pos_of, const Splitters& sp) {
  if (sp.mode == 0) classify_batch_tree<R>(x, b, pos_of, sp);
  else classify_batch_table<R>(x, b, pos_of, [](int) { return false; }, sp);
}

// The same for elements in consecutive-position pairs (see
// classify_batch_table); valid(e) says whether element e is a real element.
template <int R, bool F64, typename PosFn, typename ValidFn>
__device__ __forceinline__ void classify_batch_pairs(const uint64_t (&x)[R], uint32_t (&b)[R],
                                                     PosFn pos_of, ValidFn valid,
                                                     const Splitters& sp) {
  if (sp.mode == 0) classify_batch_tree<R>(x, b, pos_of, sp);
  else classify_batch_table<R, true, F64>(x, b, pos_of, valid, sp);
}

// The same for a table whose splitters hold runs, with the bands of the chunk:
// runs fill bins, so the bin's first splitter nearly always bounds the key, and
// the others search the bin.
template <int R, bool F64, typename PosFn>
__device__ __forceinline__ void classify_batch_bands(const uint64_t (&x)[R], uint32_t (&b)[R],
                                                     PosFn pos_of, const uint32_t* band,
                                                     const Splitters& sp) {
  uint64_t ub[R];
#pragma unroll
  for (int r = 0; r < R; ++r)
    b[r] = F64 && sp.by_value ? bin_by_value(x[r], sp) : bin_by_bits(x[r], sp);
#pragma unroll
  for (int r = 0; r < R; ++r) {
    const uint32_t t = b[r];
    b[r] = sp.tbl[t];
    ub[r] = sp.key[b[r]];
    if (ub[r] < x[r]) {
      uint32_t lo = b[r] + 1, hi = t < sp.tmax ? (uint32_t)sp.tbl[t + 1] : sp.nspl;
      while (lo < hi) {
        const uint32_t mid = (lo + hi) >> 1;
        if (sp.key[mid] < x[r]) lo = mid + 1; else hi = mid;
      }
      b[r] = lo;
      ub[r] = sp.key[lo];
    }
  }
#pragma unroll
  for (int r = 0; r < R; ++r) {
    if (ub[r] == x[r] && b[r] < sp.nspl) {
      const uint32_t w = band[b[r]], lo = w & 0xffffu, hi = w >> 16;
      b[r] = lo == hi ? lo : tie_break(lo, hi, pos_of(r), sp);
    }
  }
}

}  // namespace rsort
