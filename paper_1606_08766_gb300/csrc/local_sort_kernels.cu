// local_sort_kernels.cu -- the in-SM sort of every final bucket, chosen by
// bucket size as the paper chooses its algorithm by input size (Section 6,
// "four algorithms cover the entire range"; Appendix "Parameter Tuning"):
//
//   size 1 or equality bucket  copy through (a stable scatter already left
//   of a stable level          the elements in position order)
//   size <= kBucketCap         rank-by-counting for tiny buckets, equal-width
//                              bins for the rest; where keys cluster, refined
//                              bins, then the bitonic network (cta_sort.cuh)
//   larger (only after the     merge sort through global memory by one CTA:
//   last partition level)      bitonic-sorted runs, then pairwise merges
//
// Kernels:
//   k_direct_sort  a whole sort of at most kBucketCap keys, in one launch
//   k_local_sort   one instantiation per size class with a CTA shape that fits
//                  it: <= 1024 keys (128 threads, 8 CTAs per SM), <= 2048 keys
//                  (128 threads, 5 per SM), <= 4096 keys (256 threads, 2 per
//                  SM)
//   k_local_crowded  a class's crowded buckets, of a large batch
//   k_local_rest   what the classes leave (other crowded, copied and oversize
//                  buckets), or every bucket of a call that has few
// Buckets are taken from device work lists with atomic cursors by persistent
// grids.  The final store restores float64 bit patterns.
#include "cta_quicksort.cuh"
#include "cta_sort.cuh"
#include "rsort_internal.cuh"

namespace rsort {

namespace {

struct Scope {
  const LaunchEnv& e;
  Scope(const LaunchEnv& env, const char* name) : e(env) {
    if (e.timer) e.timer->begin(name, e.stream);
  }
  ~Scope() {
    if (e.timer) e.timer->end(e.stream);
    if (e.launches) ++*e.launches;
  }
};

struct Bufs {
  const uint64_t* in_key;
  Dst out;
  Dst tmp;
  int f64;
};

__device__ __forceinline__ void load_elem(const Bufs& B, const FinalItem& f, uint64_t j,
                                          uint64_t& k, uint32_t& i) {
  const uint64_t pos = f.start + j;
  if (f.where == kWhereInput) {
    const uint64_t raw = B.in_key[pos];
    k = B.f64 ? f64_to_ordered(raw) : raw;
    i = (uint32_t)(pos - f.aux);
  } else {
    const Dst& s = f.where == kWhereOut ? B.out : B.tmp;
    k = s.key[pos];
    i = s.idx[pos];
  }
}

__device__ __forceinline__ void store_out(const Bufs& B, uint64_t pos, uint64_t k, uint32_t i) {
  B.out.key[pos] = B.f64 ? ordered_to_f64(k) : k;
  B.out.idx[pos] = i;
}

// Merge-path split: number of elements of A among the first d outputs of
// merge(A, B); (key, idx) pairs are distinct.
__device__ __forceinline__ uint64_t merge_split(const uint64_t* ak, const uint32_t* ai, uint64_t na,
                                                const uint64_t* bk, const uint32_t* bi, uint64_t nb,
                                                uint64_t d) {
  uint64_t lo = d > nb ? d - nb : 0;
  uint64_t hi = d < na ? d : na;
  while (lo < hi) {
    const uint64_t mid = (lo + hi) >> 1;
    if (pair_less(ak[mid], ai[mid], bk[d - 1 - mid], bi[d - 1 - mid])) lo = mid + 1;
    else hi = mid;
  }
  return lo;
}

// Oversize bucket (more than kBucketCap elements after the last partition
// level; the sampling makes this vanishingly rare).  One CTA sorts runs of
// kBucketCap in shared memory, then merges runs pairwise through the two
// global buffers.  The bucket's range in the other buffer is free: other
// levels only write ranges of segments that are still being partitioned.
// Threads of k_local_rest: its buckets are few or its tail is one bucket long,
// so latency counts (10^5 keys: 256 threads 17.5 us, 512 15.2, 1024 16.7).
constexpr int kRestThreads = 512;
__device__ void sort_big(const Bufs& B, const FinalItem& f, uint64_t* sk, uint32_t* si) {
  constexpr int NT = kRestThreads;
  const uint64_t m = f.size;
  Dst A = f.where == kWhereOut ? B.out : B.tmp;
  Dst C = f.where == kWhereOut ? B.tmp : B.out;
  // runs
  for (uint64_t r0 = 0; r0 < m; r0 += kBucketCap) {
    const int len = (int)umin64(kBucketCap, m - r0);
    for (int t = threadIdx.x; t < kBucketCap; t += NT) {
      if (t < len) {
        sk[t] = A.key[f.start + r0 + t];
        si[t] = A.idx[f.start + r0 + t];
      } else {
        sk[t] = ~0ULL;
        si[t] = ~0u;
      }
    }
    block_bitonic_sort<NT>(sk, si, kBucketCap);
    for (int t = threadIdx.x; t < len; t += NT) {
      C.key[f.start + r0 + t] = sk[t];
      C.idx[f.start + r0 + t] = si[t];
    }
    __syncthreads();
  }
  Dst cur = C, nxt = A;
  constexpr int E = 8;
  for (uint64_t w = kBucketCap; w < m; w *= 2) {
    for (uint64_t p0 = 0; p0 < m; p0 += 2 * w) {
      const uint64_t na = umin64(w, m - p0);
      const uint64_t nb = p0 + w < m ? umin64(w, m - p0 - w) : 0;
      const uint64_t* ak = cur.key + f.start + p0;
      const uint32_t* ai = cur.idx + f.start + p0;
      const uint64_t* bk = ak + na;
      const uint32_t* bi = ai + na;
      for (uint64_t d0 = (uint64_t)threadIdx.x * E; d0 < na + nb; d0 += (uint64_t)NT * E) {
        uint64_t i = merge_split(ak, ai, na, bk, bi, nb, d0);
        uint64_t j = d0 - i;
        for (int e = 0; e < E && d0 + e < na + nb; ++e) {
          bool take_a;
          if (i >= na) take_a = false;
          else if (j >= nb) take_a = true;
          else take_a = pair_less(ak[i], ai[i], bk[j], bi[j]);
          const uint64_t o = f.start + p0 + d0 + e;
          if (take_a) { nxt.key[o] = ak[i]; nxt.idx[o] = ai[i]; ++i; }
          else { nxt.key[o] = bk[j]; nxt.idx[o] = bi[j]; ++j; }
        }
      }
    }
    __syncthreads();
    Dst t = cur; cur = nxt; nxt = t;
  }
  // result lives in cur; move it to the output with the final key map
  for (uint64_t t = threadIdx.x; t < m; t += NT) {
    const uint64_t pos = f.start + t;
    store_out(B, pos, cur.key[pos], cur.idx[pos]);
  }
  __syncthreads();
}

template <int NT, int IT>
__device__ __forceinline__ void load_bucket(const Bufs& B, const FinalItem& f,
                                            uint64_t (&key)[IT], uint32_t (&idx)[IT]) {
#pragma unroll
  for (int r = 0; r < IT; ++r) {
    const uint32_t e = r * NT + threadIdx.x;
    if (e < f.size) load_elem(B, f, e, key[r], idx[r]);
  }
}

// Next item of size class cls for this CTA (atomic work counter), or -1.
__device__ __forceinline__ int64_t next_item(DevState* st, int cls, uint64_t cap,
                                             uint32_t* s_item) {
  if (threadIdx.x == 0) *s_item = atomicAdd(&st->cursor_c[cls], 1u);
  __syncthreads();
  const uint32_t it = *s_item;
  __syncthreads();
  return it < umin64(st->nfinal_c[cls], cap) ? (int64_t)it : -1;
}

// ---------------------------------------------------------------------------
// The common in-SM sort of a size class: equal-width bins, one CTA per bucket.
//
// A bucket of a partition level brings the range of its keys along (its two
// splitters); an input bucket's is reduced here.  Its pairs sit in registers,
// IT a thread; every pair takes its rank inside its bin from one shared-memory
// atomic on the bin's 16-bit counter, the counters are scanned, the pairs go
// to their slots, and the few bins that hold several are ordered by insertion.
// A bucket with a crowded bin of more pairs than threads is handed on instead (a
// list of its own), so that no register of this kernel serves that case: with the
// refined bins and the bitonic network in this kernel the compiler spilled, and
// the 1025..2048-key class of a 2^28-key sort took 2.63 to 3.40 ms.  Up to a pair a
// thread it is ranked by counting here, and a bucket of one key alone needs no
// other kernel either: it is in order, or its bins are taken over the positions.
//   200,000 uint64 segments of 100 keys, all of a segment equal: 1980 us when such
//   buckets were handed on, 386 here; half of them equal: 6550, 1313.  7*10^7 keys
//   of 10,000 values, most of whose buckets hold one: 5055, 4436.
//   2^28 uniform keys, before / after: 1025..2048 keys 2.12 / 1.50 ms (3.5
//   TB/s of keys and positions read and written), 2049..4096 0.53 / 0.33,
//   up to 1024 0.12 / 0.087.
//
// The kernel is bound by its instructions and by the latency between its
// barriers, not by memory, hence
//   - the counters of a thread's run (IT words, two bins each) are cleared,
//     summed and replaced by 16-byte accesses, runs 4 words apart so that
//     eight lanes' accesses cover all banks; a word is added to the running
//     sum by one dp2a; whether a bin is crowded falls out of the OR of the
//     words;
//   - slots beyond the bucket's size are skipped four at a time by uniform
//     branches (a bucket of 1536 keys uses 12 of 16 slots);
//   - six block barriers per bucket; the claim of the next bucket and its item
//     travel while this one is sorted, and its loads go out as soon as this
//     one's pairs have left the registers.
// ---------------------------------------------------------------------------
// REFINE: crowded bins are refined once (as in cta_sort_crowded) before the
// bucket is given up; the instantiations for a batch's float64 buckets that
// span many octaves (a separate kernel for the same reason of registers).
//   100,000 normal float64 segments of 1 to 2^15 keys, all in-SM kernels:
//   9.0 ms with the bitonic network for such buckets, 3.3 ms with these.
template <int NT, int IT, int CLS, int MINB, bool REFINE>
__global__ void __launch_bounds__(NT, MINB)
k_local_sort(DevState* st, FinalItem* items, uint64_t cap, Bufs B, int crowd_list) {
  pdl_entry();
  using BS = BinSort<NT, IT>;
  constexpr int NW = NT / 32;
  extern __shared__ __align__(16) unsigned char smem_raw[];
  uint64_t* sk = (uint64_t*)smem_raw;                  // [kCap]
  uint32_t* si = (uint32_t*)(sk + BS::kCap);           // [kCap]
  uint32_t* hist = si + BS::kCap;                      // [NT * kRun + 4]
  uint16_t* half = (uint16_t*)hist;
  uint16_t* multi = (uint16_t*)(hist + NT * BS::kRun + 4);  // [kCap / 2]
  __shared__ __align__(16) uint32_t s_sum[NW];
  __shared__ uint64_t s_red[2 * NW];
  __shared__ FinalItem s_f;
  __shared__ uint32_t s_nmulti;
  constexpr int kList = REFINE ? kListRefine + (CLS - kClassSmall) : CLS;
  const uint32_t nitems = (uint32_t)umin64(st->nfinal_c[kList], cap);
  const uint32_t rank_max = min(st->local.rank_max, (uint32_t)NT);
  const uint32_t tid = threadIdx.x;
  const int lane = tid & 31, warp = tid >> 5;
  uint64_t key[IT];
  uint32_t idx[IT];
  auto load = [&](const FinalItem& f) {
    if (f.where == kWhereInput) {
      const uint64_t* kp = B.in_key + f.start + tid;
      const uint32_t i0 = (uint32_t)(f.start - f.aux) + tid;
      for_slots<NT, IT>(f.size, [&](int r) {
        const uint64_t raw = kp[r * NT];
        key[r] = B.f64 ? f64_to_ordered(raw) : raw;
        idx[r] = i0 + r * NT;
      });
    } else {
      const Dst& d = f.where == kWhereOut ? B.out : B.tmp;
      const uint64_t* kp = d.key + f.start + tid;
      const uint32_t* ip = d.idx + f.start + tid;
      for_slots<NT, IT>(f.size, [&](int r) {
        key[r] = kp[r * NT];
        idx[r] = ip[r * NT];
      });
    }
  };
  // the CTA's first bucket by its number, the others by the work counter
  // (which starts at the grid's size)
  FinalItem f{};
  if (blockIdx.x < nitems) {
    f = items[item_slot(kList, blockIdx.x, cap)];
    load(f);
  }
  while (f.size) {
    const uint32_t m = f.size;
    // the next bucket: thread 0 claims it now, reads its item below and
    // publishes it before the registers free
    uint32_t claim = 0;
    if (tid == 0) claim = gridDim.x + atomicAdd(&st->cursor_c[kList], 1u);
    FinalItem fn{};
    // all keys equal and in position order: sorted as they come
    bool in_order = false;
    bool sorted = m > rank_max;
    if (m > rank_max) {
      // smallest key and width of the key range in bits
      uint64_t mn;
      int bits;
      if (f.where == kWhereInput || f.bits == kBitsUnknown) {
        uint64_t mx = 0;
        mn = ~0ULL;
        for_slots<NT, IT>(m, [&](int r) {
          mn = key[r] < mn ? key[r] : mn;
          mx = key[r] > mx ? key[r] : mx;
        });
        block_minmax_u64<NT>(mn, mx, s_red);
        bits = mx != mn ? 64 - __clzll((long long)(mx - mn)) : 0;
      } else {
        mn = f.aux;
        bits = f.bits;
      }
      in_order = bits == 0 && f.kind == kKindSort;
      if (!in_order) {
        const int shift = bits > BS::kLogBins ? bits - BS::kLogBins : 0;
        uint32_t hr[IT];  // counter halfword, then that << 16 | rank inside the bin
        if (bits == 0) {
          // all keys equal, in no particular order: bins of their positions
          uint64_t a = ~0ULL, b = 0;
          for_slots<NT, IT>(m, [&](int r) {
            a = idx[r] < a ? idx[r] : a;
            b = idx[r] > b ? idx[r] : b;
          });
          __syncthreads();  // (s_red is written again)
          block_minmax_u64<NT>(a, b, s_red);
          const int pb = b != a ? 64 - __clzll((long long)(b - a)) : 0;
          const int ps = pb > BS::kLogBins ? pb - BS::kLogBins : 0;
          for_slots<NT, IT>(m, [&](int r) { hr[r] = BS::half_of((uint32_t)((idx[r] - a) >> ps)); });
        } else {
          for_slots<NT, IT>(m, [&](int r) {
            hr[r] = BS::half_of((uint32_t)((key[r] - mn) >> shift));
          });
        }
        if (tid == 0) s_nmulti = 0;
#pragma unroll 1
        for (int pass = 0;; ++pass) {
          clear_bins<NT, IT>(hist);
          uint4* run = (uint4*)(hist + tid * BS::kRun);
          __syncthreads();  // (1) counters clear; the previous bucket written out
          for_slots<NT, IT>(m, [&](int r) {
            const uint32_t h = hr[r];
            const uint32_t sh = (h & 1) << 4;
            const uint32_t old = atomicAdd(&hist[h >> 1], 1u << sh);
            hr[r] = (h << 16) | ((old >> sh) & 0xffffu);
          });
          if (tid == 0 && pass == 0 && claim < nitems) fn = items[item_slot(kList, claim, cap)];
          __syncthreads();  // (2) counts complete
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
          // a bin of kBinLimit or more pairs sets one of the high bits
          static_assert((kBinLimit & (kBinLimit - 1)) == 0, "the crowd test reads high bits");
          constexpr uint32_t kHigh = 0xffffu & ~(uint32_t)(kBinLimit - 1);
          const bool crowd = __any_sync(0xffffffffu, (any & (kHigh | (kHigh << 16))) != 0);
          if (lane == 31) s_sum[warp] = inc | (crowd ? 0x80000000u : 0u);
          __syncthreads();  // (3) warp sums
          uint32_t pre = 0, all = 0;
#pragma unroll
          for (int w = 0; w < NW; ++w) {
            const uint32_t v = s_sum[w];
            pre += w < warp ? v : 0u;
            all |= v;
          }
          sorted = (all >> 31) == 0;
          const bool again = REFINE && pass == 0 && !sorted && shift > 0;
          if (sorted || again) {
            // (the crowd flags of the sums before, if any, shift out of at)
            uint32_t at = (pre & 0xffffu) + inc - sum;
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
            if (tid == NT - 1) half[NT * BS::kRun * 2] = (uint16_t)m;
          }
          if (!again) break;
          __syncthreads();
          // bin b, whose c pairs start at slot lo, becomes 2c parts from 2 lo
          for_slots<NT, IT>(m, [&](int r) {
            const uint32_t h = hr[r] >> 16;
            const uint32_t lo = half[h], c = half[BS::next_half(h)] - lo;
            const uint64_t off = (key[r] - mn) << (64 - shift);
            hr[r] = BS::half_of(2 * lo + (uint32_t)__umul64hi(off, (uint64_t)(2 * c)));
          });
          __syncthreads();
        }
        if (tid == 0) s_f = fn;
        if (!sorted && m > (uint32_t)NT) {
          // crowded: the bucket goes to the call's list of such buckets
          if (tid == 0) {
            const uint32_t slot = atomicAdd(&st->nfinal_c[crowd_list], 1u);
            const int a = crowd_array(crowd_list);
            const int end = a == kClassCopy ? kClassBig : kListRefine + a - kClassSmall;
            if ((uint64_t)slot + st->nfinal_c[a] + st->nfinal_c[end] < cap)
              items[crowd_slot(st, crowd_list, slot, cap)] = f;
            else
              atomicOr(&st->error, kErrFinalCap);
          }
          __syncthreads();
          f = s_f;
          load(f);
          continue;
        }
        if (sorted) {
          __syncthreads();  // (4) bin starts in place
          for_slots<NT, IT>(m, [&](int r) {
            const uint32_t h = hr[r] >> 16, o = hr[r] & 0xffffu;
            const uint32_t p = half[h] + o;
            sk[p] = key[r];
            si[p] = idx[r];
            if (o == 1) multi[atomicAdd(&s_nmulti, 1u)] = (uint16_t)h;
          });
          if (tid == 0) count_algo(st->algo_elems, kAlgoBins, m);
          __syncthreads();  // (5) pairs in place, the registers are free
          fn = s_f;
          load(fn);
          // order every listed bin by insertion (an element alone in its bin is
          // already in its final slot)
          const uint32_t nmulti = s_nmulti;
          for (uint32_t j = tid; j < nmulti; j += NT) {
            const uint32_t h = multi[j];
            const uint32_t lo = half[h], cnt = half[BS::next_half(h)] - lo;
            uint64_t* bk = sk + lo;
            uint32_t* bi = si + lo;
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
      }
    }
    if (!sorted || in_order) {
      // in order already, or (tiny buckets, and crowded ones that have a thread a
      // pair) rank-by-counting (Appendix "Fast Work-Inefficient Ranking")
      __syncthreads();  // the previous bucket has been written out
      if (in_order) {
        for_slots<NT, IT>(m, [&](int r) {
          sk[r * NT + tid] = key[r];
          si[r * NT + tid] = idx[r];
        });
      } else if (tid < m) {
        sk[tid] = key[0];
        si[tid] = idx[0];
      }
      if (tid == 0) {
        if (claim < nitems) fn = items[item_slot(kList, claim, cap)];
        s_f = fn;
        count_algo(st->algo_elems, in_order ? kAlgoInOrder : kAlgoRank, m);
      }
      __syncthreads();
      if (!in_order) {
        uint32_t rank = 0;
        if (tid < m)
          for (uint32_t q = 0; q < m; ++q)
            rank += pair_less(sk[q], si[q], key[0], idx[0]) ? 1u : 0u;
        __syncthreads();
        if (tid < m) {
          sk[rank] = key[0];
          si[rank] = idx[0];
        }
      }
      fn = s_f;
      load(fn);
    }
    __syncthreads();  // (6) sorted
    {
      uint64_t* ko = B.out.key + f.start;
      uint32_t* io = B.out.idx + f.start;
      if (B.f64) {
        for (uint32_t t = tid; t < m; t += NT) {
          ko[t] = ordered_to_f64(sk[t]);
          io[t] = si[t];
        }
      } else {
#pragma unroll 4
        for (uint32_t t = tid; t < m; t += NT) {
          ko[t] = sk[t];
          io[t] = si[t];
        }
      }
    }
    f = fn;
  }
}

// The medium class sorted by quicksort instead (tunable "medium_sort" = 1):
// pivots from the binary-tree median approximation of a sample of every
// segment (cta_quicksort.cuh).  The result is the same; the bins of
// cta_sort_pairs measured faster, so this is an alternative, not the default.
template <int NT, int CAP, int CLS>
__global__ void __launch_bounds__(NT, 1)
k_local_quicksort(DevState* st, const FinalItem* items, uint64_t cap, Bufs B, uint64_t seed) {
  pdl_entry();
  extern __shared__ __align__(16) unsigned char smem_raw[];
  const QsSmem q = qs_carve(smem_raw, CAP);
  __shared__ uint64_t scan_sm[NT / 32];
  __shared__ uint64_t red[2 * NT / 32];
  __shared__ uint32_t s_item;
  const FinalItem* list = items + (uint64_t)CLS * cap;
  for (;;) {
    const int64_t it = next_item(st, CLS, cap, &s_item);
    if (it < 0) break;
    const FinalItem f = list[it];
    count_algo(st->algo_elems, kAlgoQuick, f.size);
    for (uint32_t t = threadIdx.x; t < f.size; t += NT) {
      uint64_t k;
      uint32_t i;
      load_elem(B, f, t, k, i);
      q.ak[t] = k;
      q.ai[t] = i;
    }
    __syncthreads();
    cta_quicksort_pairs<NT>(q, f.size, splitmix64_at(seed, (uint64_t)it), scan_sm, red);
    for (uint32_t t = threadIdx.x; t < f.size; t += NT) store_out(B, f.start + t, q.ak[t], q.ai[t]);
    __syncthreads();
  }
}

// The crowded buckets of a class (cta_sort_pairs: refined bins, the bitonic
// network), by CTAs of their size; with `own` the class's whole list, every bucket
// by bitonic sort (tunables sort_small, sort_mid).
//   k_local_rest takes them in sorts and small batches, which have few; in a large
//   batch they can be all there is, and two CTAs of 512 threads an SM are too few
//   for small ones: 20,000 segments of 1000 keys, half of them one value, 4058 us
//   there, 846 here.  sort_mid on a sort of 8*10^6 keys: 1181 there, 672 here.
template <int NT, int IT, int CLS, int MINB>
__global__ void __launch_bounds__(NT, MINB)
k_local_crowded(DevState* st, const FinalItem* items, uint64_t cap, Bufs B, bool own) {
  pdl_entry();
  using BS = BinSort<NT, IT>;
  extern __shared__ __align__(16) unsigned char smem_raw[];
  CtaSortSmem s;
  s.k = (uint64_t*)smem_raw;
  s.i = (uint32_t*)(s.k + BS::kCap);
  s.hist = s.i + BS::kCap;
  __shared__ uint64_t red[2 * NT / 32];
  __shared__ uint64_t scan_sm[NT / 32];
  __shared__ uint32_t s_next;
  constexpr int kCrowd = CLS == kClassSmall ? kListCrowdSmall : kListCrowdMid;
  const int list = own ? CLS : kCrowd;
  const uint32_t total = (uint32_t)umin64(st->nfinal_c[list], cap);
  const uint32_t rank_max = own ? st->local.rank_max : 0u;  // (small crowded ones are done)
  for (uint32_t at = blockIdx.x; at < total;) {
    const FinalItem f = items[own ? item_slot(CLS, at, cap) : crowd_slot(st, kCrowd, at, cap)];
    if (threadIdx.x == 0) s_next = gridDim.x + atomicAdd(&st->cursor_c[list], 1u);
    uint64_t key[IT];
    uint32_t idx[IT];
    load_bucket<NT, IT>(B, f, key, idx);
    cta_sort_pairs<NT, IT, true>(key, idx, f.size, [&] { return f.kind == kKindSort; }, s, red,
                                 scan_sm, st->algo_elems, rank_max, own);
    for (uint32_t t = threadIdx.x; t < f.size; t += NT)
      store_out(B, f.start + t, s.k[t], s.i[t]);
    __syncthreads();
    at = s_next;
    __syncthreads();
  }
}

// Everything the class kernels leave, by 512-thread CTAs of 8 slots: the
// copy-through buckets (size 1, or equality buckets already in position order:
// a coalesced copy that restores float64 bit patterns), the buckets with
// crowded bins (cta_sort_pairs: refined bins, the bitonic network), and the
// oversize ones (after the last partition level; rare).  lists: bit l takes list
// l; with the size classes' own lists a call of few buckets finishes in this one
// launch, whose slowest bucket bounds it, instead of one launch per class, each as
// long as its slowest bucket.  bitonic: bit c sorts class c's buckets by bitonic
// sort.  BATCH: networks fitted to a bucket (SIZED); 1000 segments of 1000 keys
// spread over 63 octaves 243 us without, 99 with.
template <bool BATCH>
__global__ void __launch_bounds__(kRestThreads, 2)
k_local_rest(DevState* st, const FinalItem* items, uint64_t cap, Bufs B, uint32_t lists,
             uint32_t bitonic) {
  pdl_entry();
  constexpr int NT = kRestThreads, IT = kBucketCap / kRestThreads;
  extern __shared__ __align__(16) unsigned char smem_raw[];
  CtaSortSmem s;
  s.k = (uint64_t*)smem_raw;
  s.i = (uint32_t*)(s.k + NT * IT);
  s.hist = s.i + NT * IT;
  __shared__ uint64_t red[2 * NT / 32];
  __shared__ uint64_t scan_sm[NT / 32];
  __shared__ uint32_t s_next;
  const uint32_t rank_max = st->local.rank_max;
  // lists in turn, the longest work first (an oversize bucket's merges run
  // longest)
  constexpr int kLists = kListCrowd + 1;
  auto list_of = [](int q) {
    constexpr int order[kLists] = {kClassBig,       kListCrowd,      kListRefine + 2,
                                   kClassMedium,    kListRefine + 1, kClassMid,
                                   kListRefine + 0, kClassSmall,     kClassCopy};
    return order[q];
  };
  uint32_t end[kLists], total = 0;
#pragma unroll
  for (int q = 0; q < kLists; ++q) {
    const int l = list_of(q);
    total += (lists >> l) & 1u ? (uint32_t)umin64(st->nfinal_c[l], cap) : 0u;
    end[q] = total;
  }
  uint32_t at = blockIdx.x;
  while (at < total) {
    int l = list_of(0);
    uint32_t from = 0;
#pragma unroll
    for (int q = 0; q + 1 < kLists; ++q) {
      if (at >= end[q]) {
        l = list_of(q + 1);
        from = end[q];
      }
    }
    const FinalItem f = items[l == kListCrowd ? crowd_slot(st, l, at - from, cap)
                                              : item_slot(l, at - from, cap)];
    if (threadIdx.x == 0) s_next = gridDim.x + atomicAdd(&st->cursor_rest, 1u);
    if (l == kClassCopy) {
      if (f.where != kWhereOut || B.f64) {  // else already in place
        for (uint32_t t = threadIdx.x; t < f.size; t += NT) {
          uint64_t k;
          uint32_t i;
          load_elem(B, f, t, k, i);
          store_out(B, f.start + t, k, i);
        }
      }
    } else if (l == kClassBig) {
      count_algo(st->algo_elems, kAlgoMerge, f.size);
      sort_big(B, f, s.k, s.i);
    } else {
      uint64_t key[IT];
      uint32_t idx[IT];
      load_bucket<NT, IT>(B, f, key, idx);
      cta_sort_pairs<NT, IT, BATCH>(key, idx, f.size, [&] { return f.kind == kKindSort; }, s, red,
                                    scan_sm, st->algo_elems, rank_max, (bitonic >> l) & 1u);
      for (uint32_t t = threadIdx.x; t < f.size; t += NT)
        store_out(B, f.start + t, s.k[t], s.i[t]);
    }
    __syncthreads();
    at = s_next;
    __syncthreads();
  }
}

// A whole sort of n <= kBucketCap keys by one CTA, which also resets the
// control block (statistics and the error word are read from it): one launch
// instead of six.  One bucket alone is bound by the latency of its steps, so
// it takes 512 threads, eight slots each (1024 of four measured 1 to 2 us slower).
constexpr int kDirectThreads = 512;
__global__ void __launch_bounds__(kDirectThreads, 1)
k_direct_sort(DevState* st, Bufs B, uint32_t n, LocalPlan local) {
  pdl_entry();
  constexpr int NT = kDirectThreads, IT = kBucketCap / kDirectThreads;
  extern __shared__ __align__(16) unsigned char smem_raw[];
  CtaSortSmem s;
  s.k = (uint64_t*)smem_raw;
  s.i = (uint32_t*)(s.k + NT * IT);
  s.hist = s.i + NT * IT;
  __shared__ uint64_t red[2 * NT / 32];
  __shared__ uint64_t scan_sm[NT / 32];
  FinalItem f;
  f.start = f.aux = 0;
  f.size = n;
  f.where = kWhereInput;
  f.kind = kKindSort;
  f.bits = kBitsUnknown;
  uint64_t key[IT];
  uint32_t idx[IT];
  load_bucket<NT, IT>(B, f, key, idx);
  static_assert(sizeof(DevState) % 4 == 0 && sizeof(DevState) / 4 <= NT, "one word a thread");
  if (threadIdx.x < sizeof(DevState) / 4) reinterpret_cast<uint32_t*>(st)[threadIdx.x] = 0;
  __syncthreads();
  const int c = n == 1 ? kClassCopy
                       : (n <= local.small_cap ? kClassSmall
                                               : (n <= local.mid_cap ? kClassMid : kClassMedium));
  if (threadIdx.x == 0) {
    st->local = local;
    st->nfinal_c[c] = 1;
    st->class_elems[c] = n;
  }
  if (n > 1)
    cta_sort_pairs<NT, IT>(key, idx, n, [&] { return true; }, s, red, scan_sm, st->algo_elems,
                           local.rank_max, local.algo[c - kClassSmall] == kLocalBitonic);
  if (n == 1) {
    if (threadIdx.x == 0) store_out(B, 0, key[0], idx[0]);
  } else {
    for (uint32_t t = threadIdx.x; t < n; t += NT) store_out(B, t, s.k[t], s.i[t]);
  }
}

// Resident CTAs per SM of the small class: the sort is latency-bound per
// bucket, so more buckets in flight per SM pay more than registers.
constexpr int kSmallPerSm = 8;
constexpr int kSmallRefinePerSm = 6;
constexpr int kSmallThreads = 128;
constexpr int kSmallItems = kSmallCap / kSmallThreads;  // 8
static_assert(kSmallThreads * kSmallItems == (int)kSmallCap, "small class fits one CTA");
// The mid class (1025..2048 keys): 128 threads of 16 slots, 5 CTAs per SM
// (256 threads of 8 slots measured 3 % slower: every bucket's fixed work --
// scans, reductions -- is spread over fewer keys per thread).
constexpr int kMidThreads = 128;
constexpr int kMidItems = (int)kMidCap / kMidThreads;  // 16
constexpr int kMidPerSm = 5;
constexpr int kMidRefinePerSm = 4;
static_assert(kMidThreads * kMidItems == (int)kMidCap, "mid class fits one CTA");
// Their crowded buckets: the network's registers (three words a pair) set the
// shape.
constexpr int kSmallCrowdPerSm = 8;
constexpr int kMidCrowdThreads = 256;
constexpr int kMidCrowdItems = (int)kMidCap / kMidCrowdThreads;  // 8
constexpr int kMidCrowdPerSm = 4;
// The medium class (2049..4096 keys): 256 threads of 16 slots, two CTAs per
// SM (with the next bucket claimed and loaded early, this measured 2 %
// faster than 512 threads of 8 slots, which had spread every bucket's fixed
// work over half the keys per thread).
constexpr int kMediumThreads = 256;
constexpr int kMediumPerSm = 2;
constexpr int kMediumItems = kBucketCap / kMediumThreads;  // 16
static_assert(kMediumThreads * kMediumItems == kBucketCap, "medium class fits one CTA");


constexpr size_t kDirectSmem = BinSort<kDirectThreads, kBucketCap / kDirectThreads>::kSmem;
constexpr size_t kRestSmem = BinSort<kRestThreads, kBucketCap / kRestThreads>::kSmem;

// Calls whose buckets cannot outnumber this many per SM finish in one launch
// of k_local_rest: 66 buckets (10^5 keys) 54 -> 15 us, 714 buckets (2^20 keys)
// 43 -> 29 us against a launch per class; the class kernels sort a bucket in
// less SM time and win above.
constexpr uint64_t kOneLaunchPerSm = 8;
// Batches that may have more buckets than this per SM launch k_local_crowded for
// the small and the mid class: the two launches cost 3 us, against 38 of 1000
// uniform segments of 1000 keys and 147 of 10,000 of 1100.
constexpr uint64_t kCrowdLaunchPerSm = 54;

template <int NT, int IT, int CLS, int MINB, bool REFINE>
void launch_class(const LaunchEnv& e, DevState* st, FinalItem* items, uint64_t cap, const Bufs& B,
                  int crowd_list, const char* name) {
  Scope sc(e, name);
  launch_kernel(e, k_local_sort<NT, IT, CLS, MINB, REFINE>, e.num_sms * MINB, NT,
                BinSort<NT, IT>::kSmem, st, items, cap, B, crowd_list);
}

template <int NT, int IT, int CLS, int MINB>
void launch_crowded(const LaunchEnv& e, DevState* st, const FinalItem* items, uint64_t cap,
                    const Bufs& B, bool own, const char* name) {
  static_assert(BinSort<NT, IT>::kSmem <= 44 * 1024, "within the default limit (with statics)");
  Scope sc(e, name);
  launch_kernel(e, k_local_crowded<NT, IT, CLS, MINB>, e.num_sms * MINB, NT,
                BinSort<NT, IT>::kSmem, st, items, cap, B, own);
}

template <int NT, int IT, int CLS, int MINB, int MINBR>
void set_class_attributes() {
  cudaFuncSetAttribute(k_local_sort<NT, IT, CLS, MINB, false>,
                       cudaFuncAttributeMaxDynamicSharedMemorySize, (int)BinSort<NT, IT>::kSmem);
  cudaFuncSetAttribute(k_local_sort<NT, IT, CLS, MINBR, true>,
                       cudaFuncAttributeMaxDynamicSharedMemorySize, (int)BinSort<NT, IT>::kSmem);
}

}  // namespace

void set_local_kernel_attributes() {
  set_class_attributes<kSmallThreads, kSmallItems, kClassSmall, kSmallPerSm, kSmallRefinePerSm>();
  set_class_attributes<kMidThreads, kMidItems, kClassMid, kMidPerSm, kMidRefinePerSm>();
  set_class_attributes<kMediumThreads, kMediumItems, kClassMedium, kMediumPerSm,
                       kMediumPerSm>();
  cudaFuncSetAttribute(k_direct_sort, cudaFuncAttributeMaxDynamicSharedMemorySize,
                       (int)kDirectSmem);
  cudaFuncSetAttribute(k_local_quicksort<kLocalThreads, (int)kMidCap, kClassMid>,
                       cudaFuncAttributeMaxDynamicSharedMemorySize, (int)qs_smem_bytes(kMidCap));
  cudaFuncSetAttribute(k_local_quicksort<kLocalThreads, kBucketCap, kClassMedium>,
                       cudaFuncAttributeMaxDynamicSharedMemorySize, (int)qs_smem_bytes(kBucketCap));
  cudaFuncSetAttribute(k_local_rest<false>, cudaFuncAttributeMaxDynamicSharedMemorySize,
                       (int)kRestSmem);
  // (k_local_crowded needs no attribute, k_local_rest<true> gets it where it is
  // launched: the kernels of batches alone are not loaded before the first one.
  // Loaded with the others they move the others' code, and a sort of 5000 keys or
  // a partition of 4096 took 1 us of 30 longer.)
}

bool direct_sort_takes(const LocalPlan& local, uint64_t n) {
  const int c = n <= local.small_cap ? 0 : (n <= local.mid_cap ? 1 : 2);
  return n <= (uint64_t)kBucketCap && local.algo[c] != kLocalQuick;
}

void launch_direct_sort(const LaunchEnv& e, DevState* st, const uint64_t* in_key, Dst out,
                        uint32_t n, int f64) {
  Bufs B;
  B.in_key = in_key;
  B.out = out;
  B.tmp = out;
  B.f64 = f64;
  Scope sc(e, "direct_sort");
  launch_kernel(e, k_direct_sort, 1, kDirectThreads, kDirectSmem, st, B, n, e.local);
}

void launch_local_sort(const LaunchEnv& e, DevState* st, FinalItem* items, uint64_t item_cap,
                       uint64_t max_items, const uint64_t* in_key, Dst out, Dst tmp, int f64,
                       bool segmented) {
  Bufs B;
  B.in_key = in_key;
  B.out = out;
  B.tmp = tmp;
  B.f64 = f64;
  // k_local_rest takes every class of a call with few buckets, the medium class
  // when its algorithm is bitonic, and what the class kernels note as crowded
  const uint8_t* algo = e.local.algo;
  const bool one = max_items <= kOneLaunchPerSm * (uint64_t)e.num_sms;
  const bool refine = segmented && f64;
  uint32_t lists = (1u << kClassCopy) | (1u << kClassBig) | (1u << kListCrowd), bitonic = 0;
  for (int c = kClassSmall; c <= kClassMedium; ++c) {
    const uint8_t a = algo[c - kClassSmall];
    if (a == kLocalBitonic) bitonic |= 1u << c;
    if ((a == kLocalBitonic && (one || c == kClassMedium)) || (one && a == kLocalBins))
      lists |= 1u << c;
    if (one && a == kLocalBins) lists |= 1u << (kListRefine + c - kClassSmall);
  }
  auto own = [&](int c) { return algo[c - kClassSmall] == kLocalBins && !((lists >> c) & 1u); };
  // the small and the mid class's crowded buckets in kernels of their shape
  const bool split = segmented && max_items > kCrowdLaunchPerSm * (uint64_t)e.num_sms;
  const int crowd_small = split ? kListCrowdSmall : kListCrowd;
  const int crowd_mid = split ? kListCrowdMid : kListCrowd;
  auto crowded = [&](int c) {
    return own(c) ? split : algo[c - kClassSmall] == kLocalBitonic && !one;
  };
  if (own(kClassSmall)) {
    launch_class<kSmallThreads, kSmallItems, kClassSmall, kSmallPerSm, false>(
        e, st, items, item_cap, B, crowd_small, "local_sort");
    if (refine)
      launch_class<kSmallThreads, kSmallItems, kClassSmall, kSmallRefinePerSm, true>(
          e, st, items, item_cap, B, crowd_small, "local_sort_refine");
  }
  if (algo[kClassMid - kClassSmall] == kLocalQuick) {
    Scope sc(e, "local_sort_mid");
    launch_kernel(e, k_local_quicksort<kLocalThreads, (int)kMidCap, kClassMid>, e.num_sms * 2,
                  kLocalThreads, qs_smem_bytes(kMidCap), st, items, item_cap, B,
                  0x243f6a8885a308d3ULL);
  } else if (own(kClassMid)) {
    launch_class<kMidThreads, kMidItems, kClassMid, kMidPerSm, false>(
        e, st, items, item_cap, B, crowd_mid, "local_sort_mid");
    if (refine)
      launch_class<kMidThreads, kMidItems, kClassMid, kMidRefinePerSm, true>(
          e, st, items, item_cap, B, crowd_mid, "local_sort_mid_refine");
  }
  if (algo[kClassMedium - kClassSmall] == kLocalQuick) {
    Scope sc(e, "local_sort_medium");
    launch_kernel(e, k_local_quicksort<kLocalThreads, kBucketCap, kClassMedium>, e.num_sms * 2,
                  kLocalThreads, qs_smem_bytes(kBucketCap), st, items, item_cap, B,
                  0x9e3779b97f4a7c15ULL);
  } else if (own(kClassMedium)) {
    launch_class<kMediumThreads, kMediumItems, kClassMedium, kMediumPerSm, false>(
        e, st, items, item_cap, B, kListCrowd, "local_sort_medium");
    if (refine)
      launch_class<kMediumThreads, kMediumItems, kClassMedium, kMediumPerSm, true>(
          e, st, items, item_cap, B, kListCrowd, "local_sort_medium_refine");
  }
  if (crowded(kClassSmall))
    launch_crowded<kSmallThreads, kSmallItems, kClassSmall, kSmallCrowdPerSm>(
        e, st, items, item_cap, B, !own(kClassSmall), "local_sort_crowded");
  if (crowded(kClassMid))
    launch_crowded<kMidCrowdThreads, kMidCrowdItems, kClassMid, kMidCrowdPerSm>(
        e, st, items, item_cap, B, !own(kClassMid), "local_sort_mid_crowded");
  {
    Scope sc(e, "local_rest");
    const uint64_t grid = umin64(umax64(max_items, 1), (uint64_t)e.num_sms * 2);
    if (segmented) {
      cudaFuncSetAttribute(k_local_rest<true>, cudaFuncAttributeMaxDynamicSharedMemorySize,
                           (int)kRestSmem);
      launch_kernel(e, k_local_rest<true>, (int)grid, kRestThreads, kRestSmem, st, items, item_cap,
                    B, lists, bitonic);
    } else {
      launch_kernel(e, k_local_rest<false>, (int)grid, kRestThreads, kRestSmem, st, items, item_cap,
                    B, lists, bitonic);
    }
  }
}

}  // namespace rsort
