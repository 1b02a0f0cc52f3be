// unit_scatter.cu -- the classify and scatter passes of a stable partition
// level (the data exchange of Appendix "Robust Multi-Level Sample Sort",
// MPI_Alltoallv in the paper, a stable scatter through HBM here) with the
// bucket of every element computed once and its output written in whole
// sectors.
//
// k_classify_ids   classifies every element of a chunk once (splitters in
//                  shared memory, the same classifiers as every other level)
//                  and stores its bucket id (16 bits) beside the per-chunk
//                  bucket histogram.  Keys stream through 16-byte loads (two
//                  keys each) straight into registers.
//
// k_scatter_units  reads keys and stored bucket ids of a sub-tile into
//                  registers, ranks every element among the elements of its
//                  bucket (stable: warp order, then lane order), and writes
//                  every bucket's run in whole UNITS of 8 elements -- 64 bytes
//                  of keys and 32 bytes of positions, aligned in the output --
//                  each stored by 8 consecutive lanes of one warp instruction,
//                  so every output sector is written whole and once.  Elements
//                  that fill units go through a bucket-sorted sub-tile in
//                  shared memory; a bucket's others (at most 7) wait in its
//                  carry slots and go out with its next elements.  Only the
//                  first and last unit of a bucket in a chunk, shared with the
//                  neighbouring chunks' ranges, are written in part.
//
// The carry area holds 7 (key, position) slots per bucket, so the scatter
// serves levels with at most kUnitMaxK buckets.
#include "async_copy.cuh"
#include "bulk_copy.cuh"
#include "rsort_internal.cuh"
#include "splitters.cuh"

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

constexpr int kUnit = 8;    // elements per output unit
constexpr int kCarry = 7;   // carry slots per bucket (kUnit - 1)

// Streaming loads of data read once: no L1 allocation, L2 evict-first.
__device__ __forceinline__ void ld_stream_v2(uint64_t& a, uint64_t& b, const uint64_t* p,
                                             uint64_t pol) {
  asm("ld.global.nc.L1::no_allocate.L2::cache_hint.v2.u64 {%0, %1}, [%2], %3;"
      : "=l"(a), "=l"(b)
      : "l"(p), "l"(pol));
}
__device__ __forceinline__ uint64_t ld_stream_u64(const uint64_t* p, uint64_t pol) {
  uint64_t v;
  asm("ld.global.nc.L1::no_allocate.L2::cache_hint.u64 %0, [%1], %2;" : "=l"(v) : "l"(p), "l"(pol));
  return v;
}
__device__ __forceinline__ uint32_t ld_stream_u32(const uint32_t* p, uint64_t pol) {
  uint32_t v;
  asm("ld.global.nc.L1::no_allocate.L2::cache_hint.u32 %0, [%1], %2;" : "=r"(v) : "l"(p), "l"(pol));
  return v;
}
__device__ __forceinline__ uint32_t ld_stream_u16(const uint16_t* p, uint64_t pol) {
  unsigned short v;
  asm("ld.global.nc.L1::no_allocate.L2::cache_hint.u16 %0, [%1], %2;" : "=h"(v) : "l"(p), "l"(pol));
  return v;
}

// Key bits as the level stores them: conv 1 maps float64 patterns to the
// order map, 2 maps them back, 0 leaves them.
__device__ __forceinline__ uint64_t conv_key(uint64_t k, int conv) {
  return conv == 1 ? f64_to_ordered(k) : (conv == 2 ? ordered_to_f64(k) : k);
}

// ---------------------------------------------------------------------------
// Classify with stored bucket ids
// ---------------------------------------------------------------------------
// Level 1 with its order left to the device (LevelParams::stable ==
// kOrderAuto): the classify counts the level's equality buckets, those whose
// two bounding splitters hold one key (every element of such a bucket has that
// key, so in position order it is final and skips the levels below), one
// segment's by the CTA of its first chunk.  The scatter and the collect keep
// input order when they are at least 1/kAutoOrderShare of the buckets
// (duplicate-heavy inputs) and rank by atomics otherwise.
template <int NT>
__device__ __forceinline__ void count_equality_buckets(DevState* st, const Splitters& sp) {
  uint32_t cnt = 0;
  for (uint32_t j = threadIdx.x; j + 1 < sp.nspl; j += NT) cnt += sp.key[j] == sp.key[j + 1];
#pragma unroll
  for (int o = 16; o > 0; o >>= 1) cnt += __shfl_down_sync(0xffffffffu, cnt, o);
  if ((threadIdx.x & 31) == 0 && cnt) atomicAdd(&st->l1_eq, cnt);
}

constexpr int kCiPairs = 4;  // 16-byte loads (two keys) per thread per step
// steps ahead of the current one whose keys are asked into L2 (0 or 1: none;
// the next step's keys are already in registers)
constexpr int kCiPrefetch = 2;

// Bound by shared-memory wavefronts (79 % of the SM's rate: table, splitter and
// counter accesses at random banks).  What got it there, 2^28 uniform keys, level
// 1 / level 2: a table step to the first splitter that is not smaller instead of
// a search (0.92 -> 0.82 ms at level 1), steps that lie inside the chunk without
// checks or 64-bit index arithmetic (0.82 -> 0.60), this kernel instead of one
// staged by cp.async at the deeper levels (0.96 -> 0.87, then 0.66).  Four CTAs
// per SM (64 registers) 0.81 / 0.72, four keys a thread 0.92 / 0.86.
// VEC: the key array is 16-byte aligned (pairs are read by 16-byte loads);
// MAP: the keys are float64 bit patterns, mapped to the order map on load.
// BANDS: one segment and long chunks (kBandMinW); if some splitters are equal, ties
// are placed by bands (load_bands) instead of a search each: duplicate-heavy 2^26
// keys 434 -> 251 us.  Distinct keys pay 2 % of the pass for looking (2^26 keys 168 ->
// 172 us), so the other levels take the form without; a loop of its own for either
// case cost them 20 % (spilled registers).
// FINE: the segment is cut by the over * k - 1 splitters of its fine partitions
// instead; their sizes over the whole level are added to hist[over * k].
template <int NT, bool VEC, bool MAP, bool FINE, bool BANDS>
__global__ void __launch_bounds__(NT, 3)
k_classify_ids(DevState* st, const LevelSeg* segs, Src src, const uint64_t* ssk,
               const uint32_t* ssi, uint32_t* hist, uint32_t kmax, int mode, bool count_eq,
               uint32_t over) {
  pdl_entry();
  constexpr int R = 2 * kCiPairs;  // keys per thread per step
  extern __shared__ __align__(16) unsigned char smem_raw[];
  Splitters sp;
  uint32_t* cnt;
  {
    unsigned char* p = smem_raw;
    const size_t Kp = next_pow2_u32(kmax);
    sp.mode = mode & 1;
    sp.ntb = (mode >> 1) & 1;
    sp.tree = nullptr;
    sp.tbl = nullptr;
    if (sp.mode == 0) {
      sp.tree = (uint64_t*)p;
      p += Kp * 8;
    } else {
      sp.tbl = (uint16_t*)p;
      p += table_bytes((uint32_t)Kp);
    }
    sp.key = (uint64_t*)p; p += (size_t)kmax * 8;
    sp.idx = (uint32_t*)p; p += (size_t)kmax * 4;
    cnt = (uint32_t*)p; p += (size_t)kmax * 4;
    if (BANDS) p += (size_t)kmax * 4;  // (the bands, after the counters)
    sp.rend = (uint16_t*)p;
  }
  const uint64_t pol = l2_evict_first_policy();
  const uint64_t total = st->total_chunks;
  const uint32_t G = st->cur_nseg;
  const int lane = threadIdx.x & 31;
  uint32_t cur_g = 0xffffffffu;
  int runs = 0;  // BANDS: some splitter keys are equal
  for (uint64_t c = blockIdx.x; c < total; c += gridDim.x) {
    const uint32_t g = seg_of_chunk(src.chunk_seg, G, c);
    LevelSeg sg = segs[g];
    // (no sample, no fine splitters: every element is in fine partition 0)
    if (FINE) sg.k = sg.S > 0 ? sg.k * over : 1;
    __syncthreads();
    if (!FINE || g != cur_g)
      for (uint32_t b = threadIdx.x; b < sg.k; b += NT) cnt[b] = 0;
    if (g != cur_g) {
      load_splitters<NT, MAP>(sg, ssk, ssi, sp);
      cur_g = g;
      if (BANDS) {
        int eq = 0;
        for (uint32_t j = threadIdx.x; j + 1 < sp.nspl; j += NT) eq |= sp.key[j] == sp.key[j + 1];
        runs = __syncthreads_or(eq);
      }
    }
    const uint64_t cl = c - sg.chunk_off;
    const uint64_t cs = sg.start + cl * sg.W;
    const uint64_t ce = umin64(cs + sg.W, sg.start + sg.m);
    if (BANDS && runs)
      load_bands<NT>((uint32_t)(cs - sg.start), (uint32_t)(ce - 1 - sg.start), cnt + kmax, sp);
    __syncthreads();
    if (count_eq && cl == 0) count_equality_buckets<NT>(st, sp);
    // pairs start at the even position at or below cs (16-byte aligned when
    // the key array is).  VEC: every pair wholly before ce is read by one
    // 16-byte load, from a position clamped into that range (pairs past it
    // read a valid pair and discard it), so the loop has no load branch; an
    // odd chunk end's last key is handled after the loop.  Otherwise every
    // key is read by its own checked load.
    const uint64_t ps = cs & ~1ull;
    const uint64_t npairs = VEC ? (ce - ps) >> 1 : (ce - ps + 1) >> 1;
    auto load = [&](uint64_t p0, uint64_t (&x)[R]) {
#pragma unroll
      for (int r = 0; r < kCiPairs; ++r) {
        const uint64_t j = p0 + (uint64_t)r * NT + threadIdx.x;
        if constexpr (VEC) {
          uint64_t a, b;
          ld_stream_v2(a, b, src.key + ps + 2 * (j < npairs ? j : npairs - 1), pol);
          x[2 * r] = j < npairs ? a : 0;
          x[2 * r + 1] = j < npairs ? b : 0;
        } else {
          const uint64_t pos = ps + 2 * j;
          x[2 * r] = x[2 * r + 1] = 0;
          if (j < npairs) {
            x[2 * r] = ld_stream_u64(src.key + pos, pol);
            if (pos + 1 < ce) x[2 * r + 1] = ld_stream_u64(src.key + pos + 1, pol);
          }
        }
      }
    };
    // one thread asks L2 for the keys of the step starting at pair p0
    auto prefetch = [&](uint64_t p0) {
      if (kCiPrefetch < 2 || threadIdx.x != 0 || p0 >= npairs) return;
      const uint64_t a = umax64(ps + 2 * p0, cs);
      const uint64_t e = umin64(ps + 2 * (p0 + (uint64_t)NT * kCiPairs), ce);
      prefetch_l2_range(src.key + a, src.key + e);
    };
    for (int d = 2; d < kCiPrefetch; ++d) prefetch((uint64_t)d * NT * kCiPairs);
    constexpr uint64_t kStep = (uint64_t)NT * kCiPairs;  // pairs per step
    // steps [w0, w1) hold only pairs inside the chunk: they are read, stored and
    // counted without a check (the first step may start one key before the
    // chunk, the last may be short)
    const uint64_t w0 = VEC ? (ps == cs ? 0 : kStep) : ~0ull;
    const uint64_t w1 = VEC ? npairs / kStep * kStep : 0;
    auto load_step = [&](uint64_t p0, uint64_t (&x)[R]) {
      if (VEC && p0 < w1) {  // (whole pairs, also where the first key is not the chunk's)
        const uint64_t* kp = src.key + ps + 2 * (p0 + threadIdx.x);
#pragma unroll
        for (int r = 0; r < kCiPairs; ++r)
          ld_stream_v2(x[2 * r], x[2 * r + 1], kp + 2 * r * NT, pol);
      } else {
        load(p0, x);
      }
    };
    uint64_t x[R], xn[R];
    if (npairs > 0) load_step(0, x);
    for (uint64_t p0 = 0; p0 < npairs; p0 += kStep) {
      prefetch(p0 + (uint64_t)kCiPrefetch * kStep);
      load_step(p0 + kStep, xn);
      uint64_t key[R];
#pragma unroll
      for (int e = 0; e < R; ++e) key[e] = MAP ? f64_to_ordered(x[e]) : x[e];
      uint32_t bk[R];
      // positions are read only on a key tie, and only inside the chunk (a
      // padding slot's result is discarded)
      // (each thread's elements come in pairs of consecutive positions)
      auto pos_at = [&](int e) {
        return ps + 2 * (p0 + (uint64_t)(e >> 1) * NT + threadIdx.x) + (e & 1);
      };
      auto valid = [&](int e) {
        const uint64_t pos = pos_at(e);
        return (p0 + (uint64_t)(e >> 1) * NT + threadIdx.x) < npairs && pos >= cs && pos < ce;
      };
      if (BANDS && runs) {
        classify_batch_bands<R, MAP>(key, bk, [&](int e) {
          return valid(e) ? (uint32_t)(pos_at(e) - sg.start) : 0u;
        }, cnt + kmax, sp);
      } else {
        classify_batch_pairs<R, MAP>(key, bk, [&](int e) {
          if (!valid(e)) return 0u;
          const uint64_t pos = pos_at(e);
          return src.idx ? src.idx[pos] : (uint32_t)(pos - sg.start);
        }, [&](int e) { return valid(e) && src.idx == nullptr; }, sp);
      }
      // runs of one bucket across the warp (duplicate-heavy inputs) take one
      // atomic per warp and slot; otherwise one atomic per key
      const uint32_t b0 = __shfl_sync(0xffffffffu, bk[0], 0);
      const bool skewed = __popc(__ballot_sync(0xffffffffu, bk[0] == b0)) > 8;
      if (p0 >= w0 && p0 < w1) {
        uint16_t* bp = src.bid + ps + 2 * (p0 + threadIdx.x);
#pragma unroll
        for (int r = 0; r < kCiPairs; ++r)
          *reinterpret_cast<uint32_t*>(bp + 2 * r * NT) = bk[2 * r] | (bk[2 * r + 1] << 16);
        if (!skewed) {
#pragma unroll
          for (int e = 0; e < R; ++e) atomicAdd(&cnt[bk[e]], 1u);
        } else {
#pragma unroll
          for (int e = 0; e < R; ++e) {
            const uint32_t bl = __shfl_sync(0xffffffffu, bk[e], 0);
            if (__all_sync(0xffffffffu, bk[e] == bl)) {
              if (lane == 0) atomicAdd(&cnt[bl], 32u);
            } else {
              atomicAdd(&cnt[bk[e]], 1u);
            }
          }
        }
      } else {
#pragma unroll
        for (int r = 0; r < kCiPairs; ++r) {
          const uint64_t j = p0 + (uint64_t)r * NT + threadIdx.x;
          const uint64_t pos = ps + 2 * j;
          const bool v0 = j < npairs && pos >= cs && pos < ce;
          const bool v1 = j < npairs && pos + 1 < ce;
          if (v0) {
            src.bid[pos] = (uint16_t)bk[2 * r];
            atomicAdd(&cnt[bk[2 * r]], 1u);
          }
          if (v1) {
            src.bid[pos + 1] = (uint16_t)bk[2 * r + 1];
            atomicAdd(&cnt[bk[2 * r + 1]], 1u);
          }
        }
      }
#pragma unroll
      for (int e = 0; e < R; ++e) x[e] = xn[e];
    }
    // VEC: an odd chunk end's last key (the pair it starts would read one key
    // past the chunk)
    if (VEC && threadIdx.x == 0 && ((ce - ps) & 1) && ce - 1 >= cs) {
      const uint64_t pos = ce - 1;
      const uint64_t raw = ld_stream_u64(src.key + pos, pol);
      uint64_t k1[1] = {MAP ? f64_to_ordered(raw) : raw};
      uint32_t b1[1];
      classify_batch_pairs<1, MAP>(k1, b1, [&](int) {
        return src.idx ? src.idx[pos] : (uint32_t)(pos - sg.start);
      }, [](int) { return false; }, sp);
      src.bid[pos] = (uint16_t)b1[0];
      atomicAdd(&cnt[b1[0]], 1u);
    }
    __syncthreads();
    if (!FINE)
      for (uint32_t b = threadIdx.x; b < sg.k; b += NT)
        hist[sg.hist_off + (uint64_t)b * sg.nunits + cl] = cnt[b];
  }
  if (FINE && cur_g != 0xffffffffu)
    for (uint32_t b = threadIdx.x; b <= sp.nspl; b += NT)
      if (cnt[b]) atomicAdd(&hist[b], cnt[b]);
}

// The second half of an overpartitioned step's classify: the stored fine ids
// become bucket ids (map[f]: the bucket of fine partition f) and are counted
// per chunk.  A bucket's splitters are fine splitters, so this is the bucket a
// second classification would find; it reads 2 bytes an element instead of 8
// and searches nothing (2^24 keys, 256 buckets of 2560 fine partitions: the
// step 390 -> 350 us).
constexpr int kMapThreads = 256;
constexpr int kMapVecs = 4;  // 16-byte loads per thread per step

__host__ __device__ inline size_t map_ids_smem_bytes(uint32_t K, uint32_t kmax) {
  return (size_t)kmax * 4 + (((size_t)K * 2 + 15) & ~(size_t)15);
}

__global__ void __launch_bounds__(kMapThreads)
k_map_ids(const DevState* st, const LevelSeg* segs, Src src, const uint32_t* map, uint32_t over,
          uint32_t* hist, uint32_t kmax) {
  pdl_entry();
  constexpr int NT = kMapThreads;
  extern __shared__ __align__(16) unsigned char smem_raw[];
  uint32_t* cnt = (uint32_t*)smem_raw;        // [kmax]
  uint16_t* to = (uint16_t*)(cnt + kmax);     // [k over]
  const uint64_t total = st->total_chunks;
  if (blockIdx.x >= total) return;
  const LevelSeg sg = segs[0];  // (the step has one segment)
  for (uint32_t f = threadIdx.x; f < sg.k * over; f += NT) to[f] = (uint16_t)map[f];
  const int lane = threadIdx.x & 31;
  for (uint64_t c = blockIdx.x; c < total; c += gridDim.x) {
    __syncthreads();
    for (uint32_t b = threadIdx.x; b < sg.k; b += NT) cnt[b] = 0;
    __syncthreads();
    const uint64_t cs = sg.start + c * sg.W;
    const uint64_t ce = umin64(cs + sg.W, sg.start + sg.m);
    // [cs, a0) and [a1, ce) singly, the 16-byte aligned part between in vectors
    const uint64_t head = ((16 - ((uintptr_t)(src.bid + cs) & 15)) & 15) / 2;
    const uint64_t a0 = umin64(cs + head, ce);
    const uint64_t nv = (ce - a0) / 8;
    const uint64_t a1 = a0 + nv * 8;
    const uint32_t singles = (uint32_t)((a0 - cs) + (ce - a1));
    if (threadIdx.x < singles) {
      const uint64_t pos = threadIdx.x < a0 - cs ? cs + threadIdx.x
                                                 : a1 + (threadIdx.x - (a0 - cs));
      const uint32_t b = to[src.bid[pos]];
      src.bid[pos] = (uint16_t)b;
      atomicAdd(&cnt[b], 1u);
    }
    uint4* vec = reinterpret_cast<uint4*>(src.bid + a0);
    for (uint64_t v0 = 0; v0 < nv; v0 += (uint64_t)NT * kMapVecs) {
      uint4 x[kMapVecs];
#pragma unroll
      for (int r = 0; r < kMapVecs; ++r) {
        const uint64_t v = v0 + (uint64_t)r * NT + threadIdx.x;
        x[r] = v < nv ? vec[v] : make_uint4(0, 0, 0, 0);
      }
#pragma unroll
      for (int r = 0; r < kMapVecs; ++r) {
        const uint64_t v = v0 + (uint64_t)r * NT + threadIdx.x;
        const bool in = v < nv;
        uint32_t b[8];
        const uint32_t w[4] = {x[r].x, x[r].y, x[r].z, x[r].w};
#pragma unroll
        for (int e = 0; e < 4; ++e) {
          b[2 * e] = to[w[e] & 0xffffu];
          b[2 * e + 1] = to[w[e] >> 16];
        }
        if (in)
          vec[v] = make_uint4(b[0] | (b[1] << 16), b[2] | (b[3] << 16), b[4] | (b[5] << 16),
                              b[6] | (b[7] << 16));
        // a warp whose elements all lie in one bucket (runs of copies of a key)
        // takes one atomic, one where many do takes one a slot that agrees
        const uint32_t b0 = __shfl_sync(0xffffffffu, b[0], 0);
        bool same = in;
#pragma unroll
        for (int e = 0; e < 8; ++e) same = same && b[e] == b0;
        if (__all_sync(0xffffffffu, same)) {
          if (lane == 0) atomicAdd(&cnt[b0], 256u);
        } else if (__popc(__ballot_sync(0xffffffffu, in && b[0] == b0)) > 8) {
#pragma unroll
          for (int e = 0; e < 8; ++e) {
            const uint32_t bl = __shfl_sync(0xffffffffu, b[e], 0);
            if (__all_sync(0xffffffffu, in && b[e] == bl)) {
              if (lane == 0) atomicAdd(&cnt[bl], 32u);
            } else if (in) {
              atomicAdd(&cnt[b[e]], 1u);
            }
          }
        } else if (in) {
#pragma unroll
          for (int e = 0; e < 8; ++e) atomicAdd(&cnt[b[e]], 1u);
        }
      }
    }
    __syncthreads();
    for (uint32_t b = threadIdx.x; b < sg.k; b += NT)
      hist[sg.hist_off + (uint64_t)b * sg.nunits + c] = cnt[b];
  }
}

// ---------------------------------------------------------------------------
// The same classify pass with its keys staged by bulk copies: one thread
// keeps a ring of kCbStages shared-memory stages of kCbStageKeys keys filled
// through the tensor memory accelerator (cp.async.bulk, completed on one
// mbarrier per stage), running ahead across the CTA's chunks, so every SM
// has up to 2 x 4 x 16 KB of loads in flight without holding registers for
// them.  A stage starts at an even position (16-byte aligned when the key
// array is) and ends at an even one; a chunk's odd last key is read directly.
// ---------------------------------------------------------------------------
constexpr int kCbStageKeys = 2048;
constexpr int kCbStages = 4;

__host__ __device__ inline size_t classify_bulk_smem_bytes(size_t common) {
  return ((common + 127) & ~(size_t)127) + (size_t)kCbStages * kCbStageKeys * 8 +
         (size_t)kCbStages * 16;
}

// Warp-specialised: NC consumer threads classify, one producer warp (the
// last) streams the stages.  Per stage a "full" barrier (one arrival with the
// expected bytes) and an "empty" barrier (one arrival per consumer warp);
// there is no block barrier inside a chunk.  Every wait is bounded: a wait
// that gives up raises kErrWait, the CTA drains its copies and returns.
template <int NC>
__global__ void __launch_bounds__(NC + 32, 2)
k_classify_bulk(DevState* st, const LevelSeg* segs, Src src, const uint64_t* ssk,
                const uint32_t* ssi, uint32_t* hist, uint32_t kmax, int mode, size_t common,
                bool count_eq) {
  pdl_entry();
  constexpr int NT = NC + 32;
  constexpr int NCW = NC / 32;         // consumer warps
  constexpr int SK = kCbStageKeys;
  constexpr int NST = kCbStages;
  constexpr int PER = SK / (2 * NC);   // key pairs per consumer thread per stage
  constexpr int R = 2 * PER;
  static_assert(PER * 2 * NC == SK, "a stage is whole pairs per consumer thread");
  extern __shared__ __align__(128) unsigned char smem_raw[];
  Splitters sp;
  uint32_t* cnt;
  {
    unsigned char* p = smem_raw;
    const size_t Kp = next_pow2_u32(kmax);
    sp.mode = mode & 1;
    sp.ntb = (mode >> 1) & 1;
    sp.tree = nullptr;
    sp.tbl = nullptr;
    if (sp.mode == 0) {
      sp.tree = (uint64_t*)p;
      p += Kp * 8;
    } else {
      sp.tbl = (uint16_t*)p;
      p += table_bytes((uint32_t)Kp);
    }
    sp.key = (uint64_t*)p; p += (size_t)kmax * 8;
    sp.idx = (uint32_t*)p; p += (size_t)kmax * 4;
    cnt = (uint32_t*)p; p += (size_t)kmax * 4;
    sp.rend = (uint16_t*)p;
  }
  uint64_t* stage = (uint64_t*)(smem_raw + ((common + 127) & ~(size_t)127));
  uint64_t* full = stage + (size_t)NST * SK;
  uint64_t* empty = full + NST;
  __shared__ uint32_t s_abort;
  const uint64_t pol = l2_evict_first_policy();
  const uint64_t total = st->total_chunks;
  const uint32_t G = st->cur_nseg;
  const uint32_t tid = threadIdx.x;
  const int lane = tid & 31, warp = tid >> 5;
  const bool producer = warp == NCW;
  if (tid == 0) {
    for (int b = 0; b < NST; ++b) {
      mbar_init(&full[b], 1);
      mbar_init(&empty[b], NCW);
    }
    mbar_fence_init();
    s_abort = 0;
  }
  __syncthreads();
  uint32_t next = 0;   // stages issued (producer) / consumed (consumers) so far
  uint32_t cur_g = 0xffffffffu;
  for (uint64_t c = blockIdx.x; c < total; c += gridDim.x) {
    const uint32_t g = seg_of_chunk(src.chunk_seg, G, c);
    const LevelSeg sg = segs[g];
    if (__syncthreads_or(s_abort != 0)) break;
    if (g != cur_g) {
      load_splitters<NT>(sg, ssk, ssi, sp);
      cur_g = g;
    }
    for (uint32_t b = tid; b < sg.k; b += NT) cnt[b] = 0;
    __syncthreads();
    const uint64_t cl = c - sg.chunk_off;
    if (count_eq && cl == 0) count_equality_buckets<NT>(st, sp);
    const uint64_t cs = sg.start + cl * sg.W;
    const uint64_t ce = umin64(cs + sg.W, sg.start + sg.m);
    const uint64_t ps = cs & ~1ull, pe = ce & ~1ull;
    const uint32_t nstg = pe > ps ? (uint32_t)((pe - ps + SK - 1) / SK) : 0u;
    if (producer) {
      if (lane == 0) {
        for (uint32_t s = 0; s < nstg; ++s, ++next) {
          const uint32_t buf = next % NST, use = next / NST;
          if (use > 0 && !mbar_wait_bounded(&empty[buf], (use - 1) & 1u, kBulkWaitPolls)) {
            atomicOr(&s_abort, 1u);
            break;
          }
          const uint64_t a = ps + (uint64_t)s * SK;
          const uint64_t b = umin64(a + SK, pe);
          fence_proxy_async_smem();
          bulk_copy_g2s(stage + (size_t)buf * SK, src.key + a, (uint32_t)((b - a) * 8),
                        &full[buf], pol);
        }
      }
      next = __shfl_sync(0xffffffffu, next, 0);
    } else {
      auto count = [&](bool v, uint32_t b) {
        const uint32_t bl = __shfl_sync(0xffffffffu, b, 0);
        if (__all_sync(0xffffffffu, v && b == bl)) {
          if (lane == 0) atomicAdd(&cnt[bl], 32u);
        } else if (v) {
          atomicAdd(&cnt[b], 1u);
        }
      };
      for (uint32_t s = 0; s < nstg; ++s, ++next) {
        const uint32_t buf = next % NST, use = next / NST;
        const bool ok = mbar_wait_bounded(&full[buf], use & 1u, kBulkWaitPolls);
        if (!__all_sync(0xffffffffu, ok)) {
          if (lane == 0) atomicOr(&s_abort, 1u);
          break;
        }
        const uint64_t a = ps + (uint64_t)s * SK;
        const uint64_t b = umin64(a + SK, pe);
        const uint64_t* stg = stage + (size_t)buf * SK;
        uint64_t key[R];
#pragma unroll
        for (int r = 0; r < PER; ++r) {
          const uint32_t j = r * NC + tid;
          key[2 * r] = key[2 * r + 1] = 0;
          if (a + 2 * j < b) {
            const uint4 v = *reinterpret_cast<const uint4*>(stg + 2 * j);
            key[2 * r] = ((uint64_t)v.y << 32) | v.x;
            key[2 * r + 1] = ((uint64_t)v.w << 32) | v.z;
          }
        }
        __syncwarp();
        if (lane == 0) mbar_arrive(&empty[buf]);  // this warp is done with the stage
#pragma unroll
        for (int e = 0; e < R; ++e) key[e] = src.map_f64 ? f64_to_ordered(key[e]) : key[e];
        uint32_t bk[R];
        classify_batch<R>(key, bk, [&](int e) {
          const uint64_t pos = a + 2 * ((uint64_t)(e >> 1) * NC + tid) + (e & 1);
          if (pos < cs || pos >= ce) return 0u;
          return src.idx ? src.idx[pos] : (uint32_t)(pos - sg.start);
        }, sp);
#pragma unroll
        for (int r = 0; r < PER; ++r) {
          const uint64_t pos = a + 2 * ((uint64_t)r * NC + tid);
          const bool v0 = pos < b && pos >= cs;
          const bool v1 = pos + 1 < b;
          if (v0 && v1) {
            *reinterpret_cast<uint32_t*>(src.bid + pos) = bk[2 * r] | (bk[2 * r + 1] << 16);
          } else if (v1) {
            src.bid[pos + 1] = (uint16_t)bk[2 * r + 1];
          }
          count(v0, bk[2 * r]);
          count(v1, bk[2 * r + 1]);
        }
      }
      // the consumer warps agree on the stage count (an abort ends them early)
    }
    __syncthreads();
    if (s_abort) break;
    // an odd chunk end: its last key is read directly
    if ((ce & 1) && ce - 1 >= cs && tid == 0) {
      uint64_t x[1] = {load_key(src, ce - 1)};
      uint32_t bk[1];
      classify_batch<1>(x, bk, [&](int) {
        return src.idx ? src.idx[ce - 1] : (uint32_t)(ce - 1 - sg.start);
      }, sp);
      src.bid[ce - 1] = (uint16_t)bk[0];
      atomicAdd(&cnt[bk[0]], 1u);
    }
    __syncthreads();
    for (uint32_t b = tid; b < sg.k; b += NT)
      hist[sg.hist_off + (uint64_t)b * sg.nunits + cl] = cnt[b];
  }
  __syncthreads();
  if (s_abort) {
    if (tid == 0) atomicOr(&st->error, kErrWait);
    // copies still in flight must land before the CTA's shared memory goes:
    // the producer waits for the phases of the last stages it issued (a
    // landed one answers at once)
    if (producer && lane == 0) {
      const uint32_t from = next > (uint32_t)NST ? next - NST : 0u;
      for (uint32_t i = from; i < next; ++i)
        mbar_wait_bounded(&full[i % NST], (i / NST) & 1u, kBulkWaitPolls);
    }
  }
}

// ---------------------------------------------------------------------------
// Scatter in whole units
// ---------------------------------------------------------------------------
// The stable scatter keeps 16-bit counters per warp and bucket (its per-warp
// winner slots lie in the sorted slots, unused while it ranks), the unordered
// one a counter per bucket; with that 12 elements a thread fit either (stable
// with 8: partition of 2^26 keys, 1024 buckets 750 -> 709 us, duplicate-heavy
// 2^26 keys 566 -> 520).  Up to kUsSmallK buckets two CTAs of 256 threads
// share an SM, each other's barriers and latencies overlapping (2^28 keys, level
// 2: 1.70 -> 1.61 ms; 100,000 segments 2.20 -> 1.90); above, the carry area
// leaves room for one, of 512 threads (640, 768 and 1024 threads with fewer
// elements each measured 1.97, 2.00 and 2.05 ms against 1.91 at level 1).
constexpr int kUsThreads = 512;
constexpr int kUsThreadsSmall = 256;
constexpr int kUsItems = 12;       // elements per thread
constexpr uint32_t kUsSmallK = 512;
// sub-tiles ahead whose bytes are asked into L2 when a sub-tile starts (0:
// none): with 1, the next sub-tile's register loads find their bytes on the way
constexpr int kUsPrefetch = 1;
// a bucket with at most this many whole units in a sub-tile writes their
// records itself; those of the others (skewed inputs) are written by a warp
// each from a list
constexpr int kUsDirectUnits = 16;
// bits of the per-bucket sub-tile word (info)
constexpr int kInfoSlotBits = 13;      // first sorted slot
constexpr int kInfoUnitShift = 13;     // elements that leave in whole units (14 bits)
constexpr int kInfoCarryShift = 27;    // carry slot of the first one that does not (3 bits)
// bits of the second word of a per-unit record (the first is the output
// position of the unit's slot 0)
constexpr int kRecFirstShift = 14;     // sorted slot of slot 0 + 8 (14 bits) below
constexpr int kRecBucketShift = 20;    // carry count, phantoms (3 + 3 bits) below

__host__ __device__ inline uint32_t us_max_units(uint32_t kmax, uint32_t st) {
  return (st + kCarry * kmax) / kUnit + 1;
}

// Buckets of a sub-tile of st elements that can have more than kUsDirectUnits
// units.
__host__ __device__ constexpr uint32_t us_max_big(uint32_t st) {
  return st / (kUsDirectUnits * kUnit) + 1;
}

// Per-warp counter rows start on 16-byte boundaries (they are cleared by 16-byte
// stores).
__host__ __device__ inline uint32_t us_cnt_stride(uint32_t kmax) { return (kmax + 7) & ~7u; }

__host__ __device__ inline size_t us_smem_bytes(uint32_t kmax, uint32_t nt, uint32_t it,
                                                bool stable) {
  const uint32_t nw = nt / 32, st = nt * it;
  size_t b = 0;
  b += (size_t)(st + kmax * kCarry) * 8;         // sorted keys, carried keys
  b += (size_t)us_max_units(kmax, st) * 8;       // per-unit records
  b += (size_t)(st + kmax * kCarry) * 4;         // sorted positions, carried ones
  b += (size_t)kmax * 12;                        // per-bucket obase, meta, info
  b = (b + 15) & ~(size_t)15;
  b += stable ? (size_t)nw * us_cnt_stride(kmax) * 2 : (size_t)kmax * 4;  // counters
  return (b + 15) & ~(size_t)15;
}

// Ranks every valid element (bucket id != 0xffffffff) of a thread's IT among
// the elements of its bucket in the sub-tile, in no particular order, by
// shared-memory atomics on the bucket counters cnt.  Atomics on one word
// serialise, so runs of one bucket (duplicate-heavy inputs, where the copies
// of a key fill a bucket by position) are ranked per warp: a warp whose
// whole window lies in one bucket takes one atomic; a window where lane 0's
// bucket holds more than 8 lanes of the first round takes one atomic per
// distinct bucket and round; otherwise every element takes its own.
template <int IT>
__device__ __forceinline__ void rank_by_atomics(const uint32_t (&bid)[IT], uint32_t (&rank)[IT],
                                                uint32_t* cnt, int lane, uint32_t ltmask) {
  const uint32_t b0 = __shfl_sync(0xffffffffu, bid[0], 0);
  bool same = b0 != 0xffffffffu;
#pragma unroll
  for (int r = 0; r < IT; ++r) same = same && bid[r] == b0;
  if (__all_sync(0xffffffffu, same)) {
    uint32_t base = 0;
    if (lane == 0) base = atomicAdd(&cnt[b0], 32u * IT);
    base = __shfl_sync(0xffffffffu, base, 0);
#pragma unroll
    for (int r = 0; r < IT; ++r) rank[r] = base + r * 32 + lane;
  } else if (__popc(__ballot_sync(0xffffffffu, bid[0] == b0)) > 8) {
#pragma unroll
    for (int r = 0; r < IT; ++r) {
      const uint32_t b = bid[r];
      const uint32_t peers = __match_any_sync(0xffffffffu, b);
      const int leader = __ffs(peers) - 1;
      uint32_t base = 0;
      if (b != 0xffffffffu && lane == leader) base = atomicAdd(&cnt[b], __popc(peers));
      rank[r] = __shfl_sync(0xffffffffu, base, leader) + __popc(peers & ltmask);
    }
  } else {
#pragma unroll
    for (int r = 0; r < IT; ++r)
      if (bid[r] != 0xffffffffu) rank[r] = atomicAdd(&cnt[bid[r]], 1u);
  }
}

// HAS_IDX: the level reads stored positions (deeper levels); otherwise the
// position is implicit (level 1: offset in the segment).
// STABLE: elements of a bucket keep input order (ranks from per-warp counters
// and a prefix over the warps); otherwise (a full sort's level 1, whose
// buckets the in-SM sort orders by (key, position) anyway) every element takes
// its rank from one shared-memory atomic on its bucket's counter.
//
// The kernel is bound by shared-memory wavefronts and by the latency between
// its barriers (one CTA per SM), so every element goes through shared memory
// once: from the elements of its bucket before it and the bucket's carry it
// knows whether it leaves in a whole unit of this sub-tile (then it goes to its
// sorted slot) or stays (then it waits in its thread's registers until the old
// carry has been written out, and goes to its carry slot).  Copying the
// incomplete units from the sorted slots to the carry area instead took 0.44 of
// 1.39 shared-memory wavefronts per element.  2^28 uniform keys: level 1 2.03 ->
// 1.91 ms, level 2 1.79 -> 1.70.
template <int NT, int IT, bool HAS_IDX, bool STABLE>
__device__ __forceinline__ void scatter_units(const DevState* st, const LevelSeg* segs, Src src,
                                              const uint32_t* hist_scan, Dst dst, uint32_t kmax,
                                              int conv, uint32_t aoff) {
  constexpr int NW = NT / 32;
  constexpr int ST = NT * IT;
  static_assert(ST <= (1 << kInfoSlotBits), "sorted slots fit the info word");
  static_assert(ST + kUnit < (1 << kRecFirstShift) && kUnitMaxK <= (1 << (32 - kRecBucketShift)),
                "sorted slots and buckets fit the unit record");
  static_assert((ST + kCarry * kUnitMaxK) / kUnit < (1 << 17), "units fit the packed scan");
  extern __shared__ __align__(16) unsigned char smem_raw[];
  unsigned char* p = smem_raw;
  // sorted slots, then bucket b's carry slots from ST + 7 b on
  uint64_t* skey = (uint64_t*)p; p += (size_t)(ST + kmax * kCarry) * 8;
  const uint32_t umax = us_max_units(kmax, ST);
  // per whole unit of the sub-tile: its output position, and the sorted slot
  // of its slot 0 + 8 | (carry count | phantoms << 3) << 14 | bucket << 20
  // (carry count and phantoms only in a bucket's first unit)
  uint2* urec = (uint2*)p; p += (size_t)umax * 8;
  uint32_t* sidx = (uint32_t*)p; p += (size_t)(ST + kmax * kCarry) * 4;
  // per-bucket state:
  //   obase  output position of the bucket's current unit start (mod 2^32)
  //   meta   carry count | phantoms << 3
  //   info   of the sub-tile: first sorted slot | elements that leave in whole
  //          units << 13 | carry slot of the first one that stays << 27
  uint32_t* obase = (uint32_t*)p; p += (size_t)kmax * 4;
  uint32_t* meta = (uint32_t*)p; p += (size_t)kmax * 4;
  uint32_t* info = (uint32_t*)p; p += (size_t)kmax * 4;
  p = smem_raw + (((p - smem_raw) + 15) & ~(size_t)15);
  const uint32_t kst = us_cnt_stride(kmax);
  uint16_t* wcnt = (uint16_t*)p;
  // [NW][kmax] winner lanes, in the sorted slots (written out when ranking starts)
  uint8_t* wwin = (uint8_t*)skey;
  static_assert(!STABLE || (size_t)ST * 8 >= (size_t)NW * kUnitMaxK,
                "the winner slots fit the sorted keys");
  __shared__ __align__(16) uint32_t s_scan[NW];
  __shared__ uint4 s_bigs[us_max_big(ST)];  // buckets of many units: first record, units, record
  __shared__ uint32_t s_nbig;
  if (threadIdx.x == 0) s_nbig = 0;

  const uint64_t pol = l2_evict_first_policy();
  const uint64_t total = st->total_chunks;
  const uint32_t G = st->cur_nseg;
  const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
  const uint32_t tid = threadIdx.x;
  const uint32_t ltmask = lanemask_lt();
  uint16_t* my_cnt = wcnt + (size_t)warp * kst;
  uint8_t* my_win = wwin + (size_t)warp * kmax;
  uint32_t* ucnt = reinterpret_cast<uint32_t*>(wcnt);  // unordered: one counter per bucket
  if (!STABLE)
    for (uint32_t b = tid; b < kmax; b += NT) ucnt[b] = 0;

  for (uint64_t c = blockIdx.x; c < total; c += gridDim.x) {
    const uint32_t g = seg_of_chunk(src.chunk_seg, G, c);
    const LevelSeg sg = segs[g];
    const uint32_t k = sg.k;
    const int nbits = k > 32 ? 5 : (int)ceil_log2_dev(k);
    const uint64_t cl = c - sg.chunk_off;
    const uint64_t cs = sg.start + cl * sg.W;
    const uint64_t ce = umin64(cs + sg.W, sg.start + sg.m);
    const uint64_t nst = (ce - cs + ST - 1) / ST;
    // buckets handled by this thread in the per-bucket phases
    const uint32_t per = (k + NT - 1) / NT;
    const uint32_t bb0 = min(tid * per, k);
    const uint32_t bb1 = min(bb0 + per, k);
    const uint32_t q0 = (uint32_t)warp * (IT * 32) + lane;
    uint64_t key[IT];
    uint32_t idx[IT], bid[IT];
    // (a whole sub-tile is loaded without checks, at constant offsets from one
    // address per array)
    auto load_bid = [&](uint64_t s) {
      if (s >= nst) return;
      const uint64_t b0 = cs + s * ST;
      const uint16_t* bp = src.bid + b0 + q0;
      if (b0 + ST <= ce) {
#pragma unroll
        for (int r = 0; r < IT; ++r) bid[r] = ld_stream_u16(bp + r * 32, pol);
      } else {
        const uint32_t left = (uint32_t)(ce - b0);
#pragma unroll
        for (int r = 0; r < IT; ++r) {
          bid[r] = 0xffffffffu;
          if (q0 + r * 32 < left) bid[r] = ld_stream_u16(bp + r * 32, pol);
        }
      }
    };
    auto load_key = [&](uint64_t s) {
      if (s >= nst) return;
      const uint64_t b0 = cs + s * ST;
      const uint64_t* kp = src.key + b0 + q0;
      const uint32_t* ip = HAS_IDX ? src.idx + b0 + q0 : nullptr;
      if (b0 + ST <= ce) {
#pragma unroll
        for (int r = 0; r < IT; ++r) {
          key[r] = ld_stream_u64(kp + r * 32, pol);
          if (HAS_IDX) idx[r] = ld_stream_u32(ip + r * 32, pol);
        }
      } else {
        const uint32_t left = (uint32_t)(ce - b0);
#pragma unroll
        for (int r = 0; r < IT; ++r) {
          if (q0 + r * 32 < left) {
            key[r] = ld_stream_u64(kp + r * 32, pol);
            if (HAS_IDX) idx[r] = ld_stream_u32(ip + r * 32, pol);
          }
        }
      }
    };
    // one thread asks L2 for sub-tile s's keys, positions and bucket ids
    auto prefetch = [&](uint64_t s) {
      if (kUsPrefetch == 0 || tid != 0 || s >= nst) return;
      const uint64_t a = cs + s * ST, e = umin64(a + ST, ce);
      prefetch_l2_range(src.key + a, src.key + e);
      if (HAS_IDX) prefetch_l2_range(src.idx + a, src.idx + e);
      prefetch_l2_range(src.bid + a, src.bid + e);
    };
    load_bid(0);
    load_key(0);
    for (int d = 1; d < kUsPrefetch; ++d) prefetch(d);
    __syncthreads();  // the previous chunk is done with every shared array
    // output state of every bucket: the chunk's first position p0, the unit
    // start at or below it (units start at positions = aoff mod 8) and the
    // slots before p0 in that unit (phantoms: held, never written)
    for (uint32_t b = tid; b < k; b += NT) {
      const uint32_t p0 = (uint32_t)(hist_scan[sg.hist_off + (uint64_t)b * sg.nunits + cl] +
                                     sg.delta);
      const uint32_t a = (p0 - aoff) & (kUnit - 1);
      obase[b] = p0 - a;
      meta[b] = a | (a << 3);
    }
    for (uint64_t s = 0; s < nst; ++s) {
      prefetch(s + kUsPrefetch);
      // -- 1. rank every element among its bucket's elements of this warp
      //    (stable: earlier rounds, then lower lanes), or of the sub-tile
      //    (unordered: a shared-memory atomic)
      uint32_t lrank[IT];
      if constexpr (!STABLE) {
        rank_by_atomics<IT>(bid, lrank, ucnt, lane, ltmask);
      } else {
      for (uint32_t q = lane; q < (k + 7) / 8; q += 32)
        ((uint4*)my_cnt)[q] = make_uint4(0, 0, 0, 0);
      __syncwarp();
      // a warp whose whole window lies in one bucket (runs of copies of a
      // key) ranks its elements by their place in the window
      const uint32_t b0 = __shfl_sync(0xffffffffu, bid[0], 0);
      bool same = b0 != 0xffffffffu;
#pragma unroll
      for (int r = 0; r < IT; ++r) same = same && bid[r] == b0;
      if (__all_sync(0xffffffffu, same)) {
#pragma unroll
        for (int r = 0; r < IT; ++r) lrank[r] = r * 32 + lane;
        if (lane == 0) my_cnt[b0] = (uint16_t)(32 * IT);
        __syncwarp();
      } else {
#pragma unroll
      for (int r = 0; r < IT; ++r) {
        const uint32_t b = bid[r];
        const bool v = b != 0xffffffffu;
        // peers = the lanes holding the same bucket: up to 32 buckets by
        // ballots over the bucket bits; beyond, every lane writes its lane id
        // to the warp's slot of its bucket and the id that stayed there (one
        // per distinct bucket) is compared instead
        uint32_t w = b;
        if (k > 32) {
          if (v) my_win[b] = (uint8_t)lane;
          __syncwarp();
          w = v ? my_win[b] : 0u;
          __syncwarp();
        }
        uint32_t peers = __ballot_sync(0xffffffffu, v);
        const bool alone = k > 32 && __all_sync(0xffffffffu, !v || w == (uint32_t)lane);
        if (alone) {
          peers &= 1u << lane;
        } else {
#pragma unroll
          for (int bit = 0; bit < 5; ++bit) {
            if (bit < nbits) {
              const bool one = (w >> bit) & 1u;
              const uint32_t m = __ballot_sync(0xffffffffu, one);
              peers &= one ? m : ~m;
            }
          }
        }
        const uint32_t c0 = v ? my_cnt[b] : 0;
        __syncwarp();
        if (v && lane == __ffs(peers) - 1) my_cnt[b] = (uint16_t)(c0 + __popc(peers));
        __syncwarp();
        lrank[r] = c0 + __popc(peers & ltmask);
      }
      }  // mixed window
      }  // STABLE
      __syncthreads();  // (A) every warp's counts are in; the old carry is in place
      // -- 2. per bucket: its elements t in this sub-tile (stable: the exclusive
      //    prefix over the warps' counts, in place), its virtual run (carry +
      //    t), the whole units u of that run and the elements w among t that
      //    fill them; one block scan of (u, w) places its elements in the
      //    sorted sub-tile and its units in the record list; its output state
      //    moves on by u units
      uint32_t loc = 0;  // w | u << 15
      auto shape = [&](uint32_t t, uint32_t cb, uint32_t& u, uint32_t& w) {
        u = (cb + t) / kUnit;
        w = u ? kUnit * u - cb : 0u;
      };
      if constexpr (!STABLE) {
        for (uint32_t b = bb0; b < bb1; ++b) {
          const uint32_t t = ucnt[b];
          ucnt[b] = 0;  // ready for the next sub-tile (its atomics follow barriers)
          uint32_t u, w;
          shape(t, meta[b] & 7u, u, w);
          info[b] = t;
          loc += w | (u << 15);
        }
      } else {
        uint32_t b = bb0;
        for (; (per & 1) == 0 && b + 1 < bb1; b += 2) {
          uint32_t tot2 = 0;
#pragma unroll
          for (int w = 0; w < NW; ++w) {
            uint32_t* cw = reinterpret_cast<uint32_t*>(wcnt + (size_t)w * kst + b);
            const uint32_t cnt2 = *cw;
            *cw = tot2;
            tot2 = __vadd2(tot2, cnt2);
          }
#pragma unroll
          for (int h = 0; h < 2; ++h) {
            const uint32_t t = h ? (tot2 >> 16) : (tot2 & 0xffffu);
            uint32_t u, w;
            shape(t, meta[b + h] & 7u, u, w);
            info[b + h] = t;
            loc += w | (u << 15);
          }
        }
        for (; b < bb1; ++b) {
          uint32_t t = 0;
#pragma unroll
          for (int w = 0; w < NW; ++w) {
            const uint32_t cnt = wcnt[(size_t)w * kst + b];
            wcnt[(size_t)w * kst + b] = (uint16_t)t;
            t += cnt;
          }
          uint32_t u, w;
          shape(t, meta[b] & 7u, u, w);
          info[b] = t;
          loc += w | (u << 15);
        }
      }
      uint32_t inc = loc;
#pragma unroll
      for (int o = 1; o < 32; o <<= 1) {
        const uint32_t y = __shfl_up_sync(0xffffffffu, inc, o);
        if (lane >= o) inc += y;
      }
      if (lane == 31) s_scan[warp] = inc;
      __syncthreads();  // (A2) warp sums
      uint32_t tot = 0, at = inc - loc;
#pragma unroll
      for (int q = 0; q < NW; ++q) {
        const uint32_t v = s_scan[q];
        at += q < warp ? v : 0u;
        tot += v;
      }
      {
        uint32_t run_w = at & 0x7fffu, run_u = at >> 15;
        for (uint32_t b = bb0; b < bb1; ++b) {
          const uint32_t t = info[b], m = meta[b], cb = m & 7u;
          uint32_t u, w;
          shape(t, cb, u, w);
          info[b] = (run_w & ((1u << kInfoSlotBits) - 1)) | (w << kInfoUnitShift) |
                    ((u ? 0u : cb) << kInfoCarryShift);
          // (an incomplete first unit keeps its phantoms)
          meta[b] = u ? (cb + t) % kUnit : (cb + t) | (m & 0x38u);
          if (u) {
            const uint32_t ob = obase[b];
            obase[b] = ob + kUnit * u;
            const uint32_t qv = (run_w + kUnit - cb) | (b << kRecBucketShift);
            const uint2 first = make_uint2(ob, qv | ((m & 0x3fu) << kRecFirstShift));
            if (u > (uint32_t)kUsDirectUnits) {
              s_bigs[atomicAdd(&s_nbig, 1u)] = make_uint4(run_u, u, first.x, first.y);
            } else {
              urec[run_u] = first;
              for (uint32_t d = 1; d < u; ++d)
                urec[run_u + d] = make_uint2(ob + kUnit * d, qv + kUnit * d);
            }
          }
          run_w += w;
          run_u += u;
        }
      }
      const uint32_t U = tot >> 15;
      __syncthreads();  // (B) bucket bases and records are in
      const uint32_t nbig = s_nbig;
      for (uint32_t i = warp; i < nbig; i += NW) {
        const uint4 e = s_bigs[i];
        for (uint32_t d = lane; d < e.y; d += 32)
          urec[e.x + d] = make_uint2(e.z + kUnit * d,
                                     (d ? e.w & ~(0x3fu << kRecFirstShift) : e.w) + kUnit * d);
      }
      // -- 3. elements that leave go to their sorted slots; the others keep
      //    their carry slot (lrank) and wait
      const uint32_t pos0 = (uint32_t)(cs + s * ST - sg.start) + q0;  // implicit positions
      if (conv) {
#pragma unroll
        for (int r = 0; r < IT; ++r) key[r] = conv_key(key[r], conv);
      }
#pragma unroll
      for (int r = 0; r < IT; ++r) {
        const uint32_t b = bid[r];
        uint32_t wait = 0xffffffffu;
        if (b != 0xffffffffu) {
          const uint32_t in = info[b];
          const uint32_t w = (in >> kInfoUnitShift) & 0x3fffu;
          const uint32_t rk = lrank[r] + (STABLE ? (uint32_t)my_cnt[b] : 0u);
          const uint32_t q = (in & ((1u << kInfoSlotBits) - 1)) + rk;
          if (rk < w) {
            skey[q] = key[r];
            sidx[q] = HAS_IDX ? idx[r] : pos0 + r * 32;
          } else {
            wait = ST + b * kCarry + (in >> kInfoCarryShift) + rk - w;
          }
        }
        lrank[r] = wait;
      }
      // the next sub-tile's bucket ids go out now (they are ranked first)
      load_bid(s + 1);
      __syncthreads();  // (C) the sorted sub-tile and the records are in
      if (tid == 0) s_nbig = 0;
      // -- 4. whole units out: 8 consecutive lanes store one unit (slots
      //    before the carry count come from the carry area, phantoms are
      //    skipped); one record lookup per slot
      {
        const uint32_t j = tid % kUnit;
#pragma unroll 2
        for (uint32_t u = tid / kUnit; u < U; u += NT / kUnit) {
          const uint2 rc = urec[u];
          const uint32_t cb = (rc.y >> kRecFirstShift) & 7u;
          const uint32_t ph = (rc.y >> (kRecFirstShift + 3)) & 7u;
          const uint32_t q = j < cb ? ST + (rc.y >> kRecBucketShift) * kCarry + j
                                    : (rc.y & ((1u << kRecFirstShift) - 1)) - kUnit + j;
          const uint64_t kv = skey[q];
          const uint32_t iv = sidx[q];
          if (j >= ph) {
            const uint32_t d = rc.x + j;  // (a bucket's first unit may start below 0)
            dst.key[d] = kv;
            dst.idx[d] = iv;
          }
        }
      }
      __syncthreads();  // (D) carry slots are read
      // -- 5. the elements that stay become their buckets' carry
#pragma unroll
      for (int r = 0; r < IT; ++r) {
        if (lrank[r] != 0xffffffffu) {
          skey[lrank[r]] = key[r];
          sidx[lrank[r]] = HAS_IDX ? idx[r] : pos0 + r * 32;
        }
      }
      load_key(s + 1);
    }
    __syncthreads();  // the last carry is in place
    // the chunk's last, incomplete unit of every bucket (the rest of its
    // sectors belongs to the next chunk's range)
    for (uint32_t b = tid; b < k; b += NT) {
      const uint32_t m = meta[b], ob = obase[b];
      const uint32_t cb = m & 7u, ph = m >> 3;
      for (uint32_t j = ph; j < cb; ++j) {
        dst.key[ob + j] = skey[ST + b * kCarry + j];
        dst.idx[ob + j] = sidx[ST + b * kCarry + j];
      }
    }
  }
}

template <int NT, int IT, bool HAS_IDX, bool STABLE>
__global__ void __launch_bounds__(NT, kUsThreads / NT)
k_scatter_units(const DevState* st, const LevelSeg* segs, Src src, const uint32_t* hist_scan,
                Dst dst, uint32_t kmax, int conv, uint32_t aoff, bool auto_order) {
  pdl_entry();
  // (level 1 with its order decided on the device: both forms are launched and
  // the one not chosen returns at once)
  if (auto_order && l1_auto_ordered(st) != STABLE) return;
  scatter_units<NT, IT, HAS_IDX, STABLE>(st, segs, src, hist_scan, dst, kmax, conv, aoff);
}

// Level 1 with its order decided on the device: either form, in one launch.  It
// spares a small call one launch; the two forms in one kernel cost registers
// and scheduling (2^28 keys: 2.06 -> 2.24 ms), so calls with long chunks launch
// both, the likelier first (the empty one's CTAs then start while it ends:
// 2*10^7 float64 keys 799 -> 791 us).  Its stable form keeps 8 elements a thread
// (48 served sorts of up to 2^22 keys: 1220 us, with 12 1245).
constexpr uint32_t kAutoOneLaunchW = kFineTile;
static_assert(kUsThreads * kUsItems == kFineTile, "fine chunks are one sub-tile");
constexpr int kUsItemsAuto = 8;  // of its stable form
__host__ inline size_t us_smem_bytes_auto(uint32_t kmax, uint32_t nt) {
  return umax64(us_smem_bytes(kmax, nt, kUsItemsAuto, true),
                us_smem_bytes(kmax, nt, kUsItems, false));
}
template <int NT>
__global__ void __launch_bounds__(NT, kUsThreads / NT)
k_scatter_units_auto(const DevState* st, const LevelSeg* segs, Src src, const uint32_t* hist_scan,
                     Dst dst, uint32_t kmax, int conv, uint32_t aoff) {
  pdl_entry();
  if (l1_auto_ordered(st))
    scatter_units<NT, kUsItemsAuto, false, true>(st, segs, src, hist_scan, dst, kmax, conv, aoff);
  else
    scatter_units<NT, kUsItems, false, false>(st, segs, src, hist_scan, dst, kmax, conv, aoff);
}

// ---------------------------------------------------------------------------
// Scatter of an unordered level (a full sort's levels after the first): the
// in-SM sort orders (key, position) pairs, so elements of a bucket may leave
// in any order.  Every element takes its rank from one shared-memory atomic
// on its bucket's counter -- no per-warp tables, no carries (a bucket's run
// per sub-tile is long at these fan-outs) -- so the kernel is small enough
// for several CTAs per SM to hide each other's latency.
// ---------------------------------------------------------------------------
constexpr int kSaThreads = 256;
constexpr int kSaItems = 8;
constexpr int kSaTile = kSaThreads * kSaItems;  // 2048 elements per sub-tile

__host__ __device__ inline size_t sa_smem_bytes(uint32_t kmax) {
  return (size_t)kSaTile * (8 + 4 + 2) + (size_t)kmax * 12;
}

template <int NT, bool HAS_IDX>
__global__ void __launch_bounds__(NT, 4)
k_scatter_atomic(const DevState* st, const LevelSeg* segs, Src src, const uint32_t* hist_scan,
                 Dst dst, uint32_t kmax, int conv) {
  pdl_entry();
  constexpr int IT = kSaItems;
  constexpr int ST = NT * IT;
  extern __shared__ __align__(16) unsigned char smem_raw[];
  unsigned char* p = smem_raw;
  uint64_t* skey = (uint64_t*)p; p += (size_t)ST * 8;
  uint32_t* sidx = (uint32_t*)p; p += (size_t)ST * 4;
  uint32_t* cnt = (uint32_t*)p; p += (size_t)kmax * 4;    // counts, then rank bases
  uint32_t* opos = (uint32_t*)p; p += (size_t)kmax * 4;   // running output position
  uint32_t* dlt = (uint32_t*)p; p += (size_t)kmax * 4;    // output position - sorted slot
  uint16_t* sb = (uint16_t*)p;                            // bucket of every sorted slot
  __shared__ uint64_t scan_sm[NT / 32];
  const uint64_t pol = l2_evict_first_policy();
  const uint64_t pol_keep = l2_evict_last_policy();
  const uint64_t total = st->total_chunks;
  const uint32_t G = st->cur_nseg;
  const uint32_t tid = threadIdx.x;
  const int lane = tid & 31, warp = tid >> 5;
  const uint32_t q0 = (uint32_t)warp * (IT * 32) + lane;
  for (uint64_t c = blockIdx.x; c < total; c += gridDim.x) {
    const uint32_t g = seg_of_chunk(src.chunk_seg, G, c);
    const LevelSeg sg = segs[g];
    const uint32_t k = sg.k;
    const uint64_t cl = c - sg.chunk_off;
    const uint64_t cs = sg.start + cl * sg.W;
    const uint64_t ce = umin64(cs + sg.W, sg.start + sg.m);
    const uint32_t per = (k + NT - 1) / NT;
    const uint32_t bb0 = min(tid * per, k), bb1 = min(bb0 + per, k);
    __syncthreads();  // the previous chunk is done with every shared array
    for (uint32_t b = tid; b < k; b += NT) {
      opos[b] = (uint32_t)(hist_scan[sg.hist_off + (uint64_t)b * sg.nunits + cl] + sg.delta);
      cnt[b] = 0;
    }
    for (uint64_t b0 = cs; b0 < ce; b0 += ST) {
      const uint32_t len = (uint32_t)umin64(ST, ce - b0);
      uint64_t key[IT];
      uint32_t idx[IT], bid[IT], rank[IT];
#pragma unroll
      for (int r = 0; r < IT; ++r) {
        const uint32_t q = q0 + r * 32;
        bid[r] = 0xffffffffu;
        if (q < len) {
          key[r] = ld_stream_u64(src.key + b0 + q, pol);
          idx[r] = HAS_IDX ? ld_stream_u32(src.idx + b0 + q, pol)
                           : (uint32_t)(b0 + q - sg.start);
          bid[r] = ld_stream_u16(src.bid + b0 + q, pol);
        }
      }
      __syncthreads();  // (A) counters cleared, previous sub-tile written out
      rank_by_atomics<IT>(bid, rank, cnt, lane, lanemask_lt());
      __syncthreads();  // (B) counts complete
      {
        uint32_t loc = 0;
        for (uint32_t b = bb0; b < bb1; ++b) loc += cnt[b];
        uint64_t tot;
        uint32_t run = (uint32_t)block_excl_scan_u64<NT>(loc, &tot, scan_sm);
        for (uint32_t b = bb0; b < bb1; ++b) {
          const uint32_t t = cnt[b];
          cnt[b] = run;                    // rank base of the bucket in the sub-tile
          dlt[b] = opos[b] - run;          // modulo 2^32: positions are below 2^32
          opos[b] += t;
          run += t;
        }
      }
      __syncthreads();  // (C) bases in place
#pragma unroll
      for (int r = 0; r < IT; ++r) {
        const uint32_t b = bid[r];
        if (b != 0xffffffffu) {
          const uint32_t q = cnt[b] + rank[r];
          skey[q] = conv_key(key[r], conv);
          sidx[q] = idx[r];
          sb[q] = (uint16_t)b;
        }
      }
      __syncthreads();  // (D) sub-tile sorted by bucket
      // runs of ~m/k elements per bucket: the sectors at their ends are
      // completed by the next sub-tile, so the stores ask the L2 to keep
      // them until then
      for (uint32_t q = tid; q < len; q += NT) {
        const uint32_t d = dlt[sb[q]] + q;
        st_keep_u64(dst.key + d, skey[q], pol_keep);
        st_keep_u32(dst.idx + d, sidx[q], pol_keep);
      }
      // counters back to zero for the next sub-tile (bases are no longer read)
      __syncthreads();
      for (uint32_t b = bb0; b < bb1; ++b) cnt[b] = 0;
    }
  }
}

// Dynamic shared memory limit of the unit scatter (0 until set or if refused).
size_t g_us_smem_max = 0;

}  // namespace

size_t classify_ids_smem_bytes(uint32_t kmax, int mode, bool bands = false) {
  const size_t Kp = next_pow2_u32(kmax);
  size_t b = (mode & 1) == 0 ? Kp * 8 : table_bytes((uint32_t)Kp);
  b += (size_t)kmax * (8 + 4 + 4 + 2 + (bands ? 4 : 0));
  return (b + 15) & ~(size_t)15;
}

bool unit_scatter_fits(uint32_t kmax) {
  return kmax <= (uint32_t)kUnitMaxK &&
         us_smem_bytes(kmax, kUsThreads, kUsItems, true) <= g_us_smem_max &&
         us_smem_bytes(kmax, kUsThreads, kUsItems, false) <= g_us_smem_max;
}

namespace {
template <int NT>
bool set_scatter_units_attributes(int limit) {
  auto set = [&](auto* f) {
    return cudaFuncSetAttribute(f, cudaFuncAttributeMaxDynamicSharedMemorySize, limit) ==
           cudaSuccess;
  };
  return set(k_scatter_units<NT, kUsItems, true, true>) &&
         set(k_scatter_units<NT, kUsItems, false, true>) &&
         set(k_scatter_units<NT, kUsItems, true, false>) &&
         set(k_scatter_units<NT, kUsItems, false, false>) && set(k_scatter_units_auto<NT>);
}
}  // namespace

namespace {
template <bool FINE, bool BANDS>
void set_classify_ids_attributes(uint32_t kmax) {
  const int smem = (int)umax64(FINE ? 0 : classify_ids_smem_bytes(kmax, 0, BANDS),
                               classify_ids_smem_bytes(kmax, 1, BANDS));
  auto set = [&](auto* f) {
    cudaFuncSetAttribute(f, cudaFuncAttributeMaxDynamicSharedMemorySize, smem);
  };
  set(k_classify_ids<256, true, false, FINE, BANDS>);
  set(k_classify_ids<256, true, true, FINE, BANDS>);
  set(k_classify_ids<256, false, false, FINE, BANDS>);
  set(k_classify_ids<256, false, true, FINE, BANDS>);
}
}  // namespace

void set_unit_scatter_attributes() {
  set_classify_ids_attributes<false, false>(kMaxK);
  set_classify_ids_attributes<false, true>(kMaxK);
  set_classify_ids_attributes<true, false>(kMaxFine);
  static_assert((size_t)kMaxFine * 2 + kUnitMaxK * 4 + 16 <= 48 * 1024, "k_map_ids' default limit");
  cudaFuncSetAttribute(k_classify_bulk<256>, cudaFuncAttributeMaxDynamicSharedMemorySize,
                       (int)classify_bulk_smem_bytes(umax64(classify_ids_smem_bytes(kMaxK, 0),
                                                            classify_ids_smem_bytes(kMaxK, 1))));
  int dev = 0, optin = 0;
  cudaGetDevice(&dev);
  cudaDeviceGetAttribute(&optin, cudaDevAttrMaxSharedMemoryPerBlockOptin, dev);
  cudaFuncAttributes fa{};
  size_t limit = 0;
  if (cudaFuncGetAttributes(&fa, k_scatter_units_auto<kUsThreads>) == cudaSuccess &&
      (size_t)optin > fa.sharedSizeBytes) {
    limit = (size_t)optin - fa.sharedSizeBytes;
    const size_t need = umax64(us_smem_bytes(kUnitMaxK, kUsThreads, kUsItems, true),
                               us_smem_bytes(kUnitMaxK, kUsThreads, kUsItems, false));
    if (limit > need) limit = need;
    if (!set_scatter_units_attributes<kUsThreads>((int)limit) ||
        !set_scatter_units_attributes<kUsThreadsSmall>((int)limit))
      limit = 0;
  }
  g_us_smem_max = limit;
  cudaFuncSetAttribute(k_scatter_atomic<kSaThreads, true>,
                       cudaFuncAttributeMaxDynamicSharedMemorySize, (int)sa_smem_bytes(kMaxK));
  cudaFuncSetAttribute(k_scatter_atomic<kSaThreads, false>,
                       cudaFuncAttributeMaxDynamicSharedMemorySize, (int)sa_smem_bytes(kMaxK));
  cudaGetLastError();
}

namespace {
// Resident CTAs per SM of k_classify_ids (0: its shared memory does not fit).
template <bool FINE, bool BANDS>
int classify_ids_blocks(uint32_t kmax, int mode) {
  int nb = 0;
  if (cudaOccupancyMaxActiveBlocksPerMultiprocessor(
          &nb, k_classify_ids<256, true, false, FINE, BANDS>, 256,
          classify_ids_smem_bytes(kmax, mode, BANDS)) != cudaSuccess) {
    cudaGetLastError();
    nb = 0;
  }
  return nb;
}

template <bool FINE, bool BANDS>
void launch_classify_ids_as(const LaunchEnv& e, uint64_t chunk_cap, int nb, DevState* st,
                            const LevelSeg* segs, const Src& src, const uint64_t* ssk,
                            const uint32_t* ssi, uint32_t* hist, uint32_t kmax, int mode, bool eq,
                            uint32_t over) {
  const size_t smem = classify_ids_smem_bytes(kmax, mode, BANDS);
  const uint64_t grid = umin64(chunk_cap, (uint64_t)e.num_sms * (nb < 1 ? 1 : nb));
  const int g = (int)(grid ? grid : 1);
  auto go = [&](auto* kernel) {
    launch_kernel(e, kernel, g, 256, smem, st, segs, src, ssk, ssi, hist, kmax, mode, eq, over);
  };
  // 16-byte pair loads need a 16-byte aligned key array
  const bool vec = ((uintptr_t)src.key & 15) == 0;
  if (vec && src.map_f64)
    go(k_classify_ids<256, true, true, FINE, BANDS>);
  else if (vec)
    go(k_classify_ids<256, true, false, FINE, BANDS>);
  else if (src.map_f64)
    go(k_classify_ids<256, false, true, FINE, BANDS>);
  else
    go(k_classify_ids<256, false, false, FINE, BANDS>);
}

}  // namespace

void launch_classify_ids(const LaunchEnv& e, const LevelParams& P, DevState* st,
                         const LevelSeg* segs, Src src, const uint64_t* ssk, const uint32_t* ssi,
                         uint32_t* hist, uint32_t kmax, int mode, bool bands, const char* name) {
  if (P.bulk_classify && ((uintptr_t)src.key & 15) == 0) {
    // keys staged by bulk copies (needs a 16-byte aligned key array)
    const size_t common = classify_ids_smem_bytes(kmax, mode);
    const size_t smem = classify_bulk_smem_bytes(common);
    int nb = 0;
    cudaOccupancyMaxActiveBlocksPerMultiprocessor(&nb, k_classify_bulk<256>, 256 + 32, smem);
    if (nb < 1) nb = 1;
    const uint64_t grid = umin64(P.chunk_cap, (uint64_t)e.num_sms * nb);
    Scope sc(e, name);
    launch_kernel(e, k_classify_bulk<256>, (int)(grid ? grid : 1), 256 + 32, smem, st, segs, src,
                  ssk, ssi, hist, kmax, mode, common, P.stable == kOrderAuto);
    return;
  }
  Scope sc(e, name);
  // bands where the room for them costs no resident CTA
  const bool eq = P.stable == kOrderAuto;
  const int nb = classify_ids_blocks<false, false>(kmax, mode);
  if (bands && (mode & 3) == 1 && classify_ids_blocks<false, true>(kmax, mode) >= nb)
    launch_classify_ids_as<false, true>(e, P.chunk_cap, nb, st, segs, src, ssk, ssi, hist, kmax,
                                        mode, eq, 0);
  else
    launch_classify_ids_as<false, false>(e, P.chunk_cap, nb, st, segs, src, ssk, ssi, hist, kmax,
                                         mode, eq, 0);
}

bool fine_ids_fit(uint32_t K) { return classify_ids_blocks<true, false>(K, 1) >= 2; }

void launch_fine_ids(const LaunchEnv& e, const LevelParams& P, DevState* st, const LevelSeg* segs,
                     Src src, const uint64_t* ssk, const uint32_t* ssi, const Overpart& op,
                     const char* name) {
  Scope sc(e, name);
  const uint32_t K = op.k * op.over;
  const int mode = 1 | (P.no_tie_break ? 2 : 0);
  launch_classify_ids_as<true, false>(e, P.chunk_cap, classify_ids_blocks<true, false>(K, mode),
                                      st, segs, src, ssk, ssi, op.fine_cnt, K, mode, false,
                                      op.over);
}

void launch_map_ids(const LaunchEnv& e, const LevelParams& P, const DevState* st,
                    const LevelSeg* segs, Src src, const Overpart& op, uint32_t* hist,
                    const char* name) {
  const size_t smem = map_ids_smem_bytes(op.k * op.over, op.k);
  int nb = 0;
  cudaOccupancyMaxActiveBlocksPerMultiprocessor(&nb, k_map_ids, kMapThreads, smem);
  const uint64_t grid = umin64(P.chunk_cap, (uint64_t)e.num_sms * (nb < 1 ? 1 : nb));
  Scope sc(e, name);
  launch_kernel(e, k_map_ids, (int)(grid ? grid : 1), kMapThreads, smem, st, segs, src,
                op.fine_cnt, op.over, hist, op.k);
}

void launch_scatter_atomic(const LaunchEnv& e, const LevelParams& P, DevState* st,
                           const LevelSeg* segs, Src src, const uint32_t* hist_scan, Dst dst,
                           uint32_t kmax, int unmap_out, const char* name) {
  const int conv = (src.map_f64 && !unmap_out) ? 1 : ((!src.map_f64 && unmap_out) ? 2 : 0);
  const size_t smem = sa_smem_bytes(kmax);
  int nb = 0;
  if (src.idx)
    cudaOccupancyMaxActiveBlocksPerMultiprocessor(&nb, k_scatter_atomic<kSaThreads, true>,
                                                  kSaThreads, smem);
  else
    cudaOccupancyMaxActiveBlocksPerMultiprocessor(&nb, k_scatter_atomic<kSaThreads, false>,
                                                  kSaThreads, smem);
  if (nb < 1) nb = 1;
  const uint64_t grid = umin64(P.chunk_cap, (uint64_t)e.num_sms * nb);
  Scope sc(e, name);
  if (src.idx)
    launch_kernel(e, k_scatter_atomic<kSaThreads, true>, (int)(grid ? grid : 1), kSaThreads, smem,
                  st, segs, src, hist_scan, dst, kmax, conv);
  else
    launch_kernel(e, k_scatter_atomic<kSaThreads, false>, (int)(grid ? grid : 1), kSaThreads, smem,
                  st, segs, src, hist_scan, dst, kmax, conv);
}

bool atomic_scatter_fits(uint32_t kmax) {
  return kmax <= (uint32_t)kMaxK && sa_smem_bytes(kmax) <= sa_smem_bytes(kMaxK);
}

namespace {
template <int NT>
void launch_scatter_units_nt(const LaunchEnv& e, const LevelParams& P, DevState* st,
                             const LevelSeg* segs, const Src& src, const uint32_t* hist_scan,
                             const Dst& dst, uint32_t kmax, int conv, uint32_t aoff) {
  const uint64_t grid = umin64(P.chunk_cap, (uint64_t)e.num_sms * (kUsThreads / NT));
  const int g = (int)(grid ? grid : 1);
  const size_t smem_s = us_smem_bytes(kmax, NT, kUsItems, true);
  const size_t smem_a = us_smem_bytes(kmax, NT, kUsItems, false);
  const bool autoo = P.stable == kOrderAuto;  // (level 1: no stored positions)
  if (autoo && P.W <= kAutoOneLaunchW) {
    launch_kernel(e, k_scatter_units_auto<NT>, g, NT, us_smem_bytes_auto(kmax, NT), st, segs, src,
                  hist_scan, dst, kmax, conv, aoff);
    return;
  }
  if (P.stable != 1 || autoo) {
    if (src.idx)
      launch_kernel(e, k_scatter_units<NT, kUsItems, true, false>, g, NT, smem_a, st, segs, src,
                    hist_scan, dst, kmax, conv, aoff, autoo);
    else
      launch_kernel(e, k_scatter_units<NT, kUsItems, false, false>, g, NT, smem_a, st, segs, src,
                    hist_scan, dst, kmax, conv, aoff, autoo);
  }
  if (autoo && e.launches) ++*e.launches;
  if (P.stable == 1 || autoo) {
    if (src.idx)
      launch_kernel(e, k_scatter_units<NT, kUsItems, true, true>, g, NT, smem_s, st, segs, src,
                    hist_scan, dst, kmax, conv, aoff, autoo);
    else
      launch_kernel(e, k_scatter_units<NT, kUsItems, false, true>, g, NT, smem_s, st, segs, src,
                    hist_scan, dst, kmax, conv, aoff, autoo);
  }
}
}  // namespace

void launch_scatter_units(const LaunchEnv& e, const LevelParams& P, DevState* st,
                          const LevelSeg* segs, Src src, const uint32_t* hist_scan, Dst dst,
                          uint32_t kmax, int unmap_out, const char* name) {
  const int conv = (src.map_f64 && !unmap_out) ? 1 : ((!src.map_f64 && unmap_out) ? 2 : 0);
  // units start where the output key address is 64-byte aligned
  const uint32_t aoff = (uint32_t)(((64 - ((uintptr_t)dst.key & 63)) & 63) / 8);
  Scope sc(e, name);
  if (kmax <= kUsSmallK)
    launch_scatter_units_nt<kUsThreadsSmall>(e, P, st, segs, src, hist_scan, dst, kmax, conv, aoff);
  else
    launch_scatter_units_nt<kUsThreads>(e, P, st, segs, src, hist_scan, dst, kmax, conv, aoff);
}

}  // namespace rsort
