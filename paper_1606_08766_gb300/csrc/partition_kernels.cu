// partition_kernels.cu -- one level of the robust multi-level sample sort
// (Appendix "Robust Multi-Level Sample Sort" of Axtmann & Sanders,
// arXiv 1606.08766) over a device-resident list of segments:
//
//   plan -> sample and sort the sample -> classify + per-chunk histograms ->
//   exclusive scan -> scatter -> collect the buckets
//
// The scatter keeps input order inside every bucket (the partition step's
// layout) unless the level is a full sort's deeper level, which may rank by
// shared-memory atomics instead (the in-SM sort orders (key, position) pairs).
//
// Every segment of the level is partitioned independently; all segments share
// the launches, so one level of a plain sort (one segment) and of a batched
// segmented sort (thousands of segments) run the same kernels.  The paper's
// processing elements are virtual partitions of HBM: the k buckets of a
// segment are its k virtual partitions, and the MPI_Alltoallv data exchange of
// the paper's sample sort becomes the scan + scatter through HBM.
#include <cstdio>
#include <type_traits>

#include "async_copy.cuh"
#include "cta_sort.cuh"
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

// ---------------------------------------------------------------------------
// Kernels
// ---------------------------------------------------------------------------

// Control block of a call, before its first level.
__device__ __forceinline__ void reset_state(DevState* st, const LocalPlan& local) {
  st->local = local;
  st->nseg[0] = st->nseg[1] = 0;
  for (int c = 0; c < kNumLists; ++c) {
    st->nfinal_c[c] = 0;
    st->cursor_c[c] = 0;
  }
  for (int c = 0; c < kNumClasses; ++c) st->class_elems[c] = 0;
  st->cursor_rest = 0;
  for (int a = 0; a < kNumAlgos; ++a) st->algo_elems[a] = 0;
  st->error = 0;
  st->max_bucket_l1 = 0;
  st->levels_used = 0;
  st->cur_nseg = 0;
  st->total_samples = st->total_chunks = st->total_hist = 0;
  st->total_schunks = st->total_buckets = 0;
  st->big_items = 0;
  for (int i = 0; i < 4; ++i) st->level_elems[i] = 0;
  st->l1_eq = st->l1_nb = st->l1_ordered = 0;
}

// Start of a call on a list of segments (n == 0), or of a sort of n keys that
// one CTA sorts.
__global__ void k_init_plain(DevState* st, FinalItem* items, uint64_t n, uint64_t final_cap,
                             LocalPlan local) {
  pdl_entry();
  if (threadIdx.x != 0 || blockIdx.x != 0) return;
  reset_state(st, local);
  if (n == 0) return;
  FinalItem f;
  f.start = 0;
  f.aux = 0;
  f.size = (uint32_t)n;
  f.where = kWhereInput;
  f.kind = n == 1 ? kKindCopy : kKindSort;
  f.bits = kBitsUnknown;
  push_final(st, items, final_cap, f, kErrFinalCap);
}

__device__ __forceinline__ void fill_segment(LevelSeg& s, uint64_t start, uint32_t m, uint32_t k,
                                             uint32_t S, uint32_t nch, const LevelParams& P,
                                             uint32_t known, const KeyRange& range) {
  s.start = start;
  s.seed = P.level == 1 ? P.seed : splitmix64_at(P.seed, ((uint64_t)P.level << 40) ^ start);
  s.m = m;
  s.k = k;
  s.S = S;
  s.nchunks = nch;
  s.nschunks = (S + P.sample_chunk - 1) / P.sample_chunk;
  s.nunits = nch;
  // equal chunks inside the segment (the level's W bounds their size)
  s.W = nch ? (uint32_t)(((uint64_t)m + nch - 1) / nch) : P.W;
  s.known = known;
  s.range = range;
}

// Per-segment parameters and prefix sums of one level.  CTA t takes segments
// [t, t + 1) * kPlanThreads.  With one CTA k_level_plan does everything; a level
// that may have more segments runs k_plan_sums first, which leaves every CTA's
// sums in plan_sums, and each CTA of k_level_plan adds up those before its
// own (33,000 segments: one CTA in a loop over tiles 197 us, a run of segments
// per thread 256, the two launches 30).
constexpr int kPlanThreads = 1024;

// Samples, chunks, histogram counters, sample chunks, buckets and elements of
// segment g of list_in (zeros past the end).
__device__ __forceinline__ SegIn plan_shape(const SegIn* list_in, uint32_t g, uint32_t G,
                                            const LevelParams& P, uint32_t kmax_level,
                                            uint64_t (&v)[6]) {
  SegIn in{};
#pragma unroll
  for (int i = 0; i < 6; ++i) v[i] = 0;
  if (g >= G) return in;
  in = list_in[g];
  const uint32_t cls = ceil_log2_dev(in.m);
  const uint32_t tb = (cls <= 32 && P.target_by_class[cls]) ? P.target_by_class[cls]
                                                            : P.target_bucket;
  const uint32_t want = in.m / tb + (in.m % tb ? 1u : 0u);
  const uint32_t k = max(2u, min(want, kmax_level));
  const uint32_t S = (uint32_t)umin64(umin64(in.m, (uint64_t)kDeepOversample * k), P.samp_max);
  const uint32_t nch = in.m / P.W + (in.m % P.W ? 1u : 0u);
  v[0] = S;
  v[1] = nch;
  v[2] = (uint64_t)k * nch;
  v[3] = (S + kSampleChunk - 1) / kSampleChunk;
  v[4] = k;
  v[5] = in.m;
  return in;
}

// The six sums in four scans.  Samples, chunks, sample chunks and elements are
// each at most one per element (below 2^32); buckets are not bounded like that,
// but each brings a histogram counter, whose sum keeps 64 bits and fails its
// capacity first.
constexpr int kPlanScans = 4;
__device__ __forceinline__ void pack_plan(const uint64_t (&v)[6], uint64_t (&pk)[kPlanScans]) {
  pk[0] = v[0] | (v[1] << 32);
  pk[1] = v[2];
  pk[2] = v[3] | (v[4] << 32);
  pk[3] = v[5];
}
__device__ __forceinline__ void unpack_plan(const uint64_t (&pk)[kPlanScans], uint64_t (&v)[6]) {
  v[0] = pk[0] & 0xffffffffu;
  v[1] = pk[0] >> 32;
  v[2] = pk[1];
  v[3] = pk[2] & 0xffffffffu;
  v[4] = pk[2] >> 32;
  v[5] = pk[3];
}

__global__ void __launch_bounds__(kPlanThreads)
k_plan_sums(const DevState* st, const SegIn* list_in, LevelParams P, int par_in,
            uint32_t kmax_level, uint64_t* plan_sums) {
  pdl_entry();
  __shared__ uint64_t sm[kPlanThreads / 32];
  const uint32_t G = st->nseg[par_in];
  if (G > P.seg_cap || (uint64_t)blockIdx.x * kPlanThreads >= G) return;
  uint64_t v[6], pk[kPlanScans];
  plan_shape(list_in, blockIdx.x * kPlanThreads + threadIdx.x, G, P, kmax_level, v);
  pack_plan(v, pk);
#pragma unroll
  for (int i = 0; i < kPlanScans; ++i) {
    uint64_t tot;
    block_excl_scan_u64<kPlanThreads>(pk[i], &tot, sm);
    if (threadIdx.x == 0) plan_sums[blockIdx.x * kPlanScans + i] = tot;
  }
}

__global__ void __launch_bounds__(kPlanThreads)
k_level_plan(DevState* st, const SegIn* list_in, LevelSeg* segs, LevelParams P, int par_in,
             uint32_t kmax_level, const uint64_t* plan_sums, uint32_t* chunk_seg) {
  pdl_entry();
  __shared__ uint64_t sm[kPlanThreads / 32];
  const uint32_t G0 = st->nseg[par_in];
  // (segments that may overlap are not partitioned: the ids and outputs of one
  // would be overwritten by another's while its counts are its own)
  const bool over = G0 > P.seg_cap || (st->error & kErrUnordered) != 0;
  const uint32_t G = over ? 0u : G0;
  const uint32_t ncta = max(1u, (G + kPlanThreads - 1) / kPlanThreads);
  const uint32_t t = blockIdx.x;
  if (t >= ncta) return;
  if (P.fit_chunks && gridDim.x == 1) {
    // few elements may have come this far (duplicate-heavy input): they are
    // spread over as many chunks as all elements would be (the chunk and
    // histogram capacities count those chunks and one more per segment)
    const uint32_t gm = threadIdx.x;
    uint64_t sum;
    block_excl_scan_u64<kPlanThreads>(gm < G ? list_in[gm].m : 0u, &sum, sm);
    const uint64_t w = (sum + P.fit_chunks - 1) / P.fit_chunks;
    P.W = (uint32_t)umin64(P.W, umax64(kMinDeepChunk,
                                       (w + kMinDeepChunk - 1) / kMinDeepChunk * kMinDeepChunk));
  }
  uint64_t before[kPlanScans];
#pragma unroll
  for (int i = 0; i < kPlanScans; ++i) {
    uint64_t x = 0;
    for (uint32_t q = threadIdx.x; q < t; q += kPlanThreads) x += plan_sums[q * kPlanScans + i];
    before[i] = 0;
    if (t > 0) block_excl_scan_u64<kPlanThreads>(x, &before[i], sm);
  }
  const uint32_t g = t * kPlanThreads + threadIdx.x;
  uint64_t v[6], pk[kPlanScans], ex[6], tot[6];
  const SegIn in = plan_shape(list_in, g, G, P, kmax_level, v);
  pack_plan(v, pk);
  {
    uint64_t sum[kPlanScans];
#pragma unroll
    for (int i = 0; i < kPlanScans; ++i) {
      pk[i] = before[i] + block_excl_scan_u64<kPlanThreads>(pk[i], &sum[i], sm);
      sum[i] += before[i];
    }
    unpack_plan(pk, ex);
    unpack_plan(sum, tot);
  }
  // (every CTA's totals up to its own tile: beyond a capacity, the last CTA's
  // check fails too and the level is not run)
  uint32_t err = 0;
  if (tot[0] > P.samp_cap) err |= kErrSampleCap;
  if (tot[1] > P.chunk_cap) err |= kErrChunkCap;
  if (tot[2] > P.hist_cap) err |= kErrHistCap;
  if (tot[3] > P.schunk_cap) err |= kErrSchunkCap;
  if (tot[4] > P.bucket_cap) err |= kErrBucketCap;
  if (g < G) {
    LevelSeg s;
    fill_segment(s, in.start, in.m, (uint32_t)v[4], (uint32_t)v[0], (uint32_t)v[1], P, in.known,
                 in.range);
    s.samp_off = ex[0];
    s.chunk_off = ex[1];
    s.hist_off = ex[2];
    s.schunk_off = ex[3];
    s.bkt_off = ex[4];
    s.delta = in.start - ex[5];
    segs[g] = s;
  }
  if (err == 0) {
    // the segment of every chunk: a thread its segment's few, a warp the many
    const uint32_t nch = (uint32_t)v[1];
    const bool many = nch > 8;
    if (!many)
      for (uint32_t c = 0; c < nch; ++c) chunk_seg[ex[1] + c] = g;
    uint32_t left = __ballot_sync(0xffffffffu, many);
    while (left) {
      const int l = __ffs(left) - 1;
      left &= left - 1;
      const uint64_t c0 = __shfl_sync(0xffffffffu, ex[1], l);
      const uint32_t n = __shfl_sync(0xffffffffu, nch, l);
      const uint32_t gl = __shfl_sync(0xffffffffu, g, l);
      for (uint32_t c = threadIdx.x & 31; c < n; c += 32) chunk_seg[c0 + c] = gl;
    }
  }
  if (threadIdx.x != 0 || t + 1 != ncta) return;
  st->nseg[par_in ^ 1] = 0;
  if (G0 > P.seg_cap) err |= kErrSegCap;
  if (over && err == 0) err = kErrUnordered;
  if (err) {
    atomicOr(&st->error, err);
    st->cur_nseg = 0;
    st->total_samples = st->total_chunks = st->total_hist = 0;
    st->total_schunks = st->total_buckets = 0;
  } else {
    st->cur_nseg = G;
    st->total_samples = tot[0];
    st->total_chunks = tot[1];
    st->total_hist = tot[2];
    st->total_schunks = tot[3];
    st->total_buckets = tot[4];
    if (G) st->levels_used = P.level;
    if (P.level == 1) st->l1_nb = (uint32_t)umin64(tot[4], 0xffffffffull);
    if (P.level >= 1 && P.level <= 4) st->level_elems[P.level - 1] = tot[5];
  }
}

// Sample positions of a segment of m elements with S samples: sample j comes
// from positions [floor(j*m/S), floor((j+1)*m/S)) at offset splitmix64(seed, j)
// mod size.  The quotients need no 64-bit division per sample: with m = q S + r,
// floor(j*m/S) = j q + floor(j r / S), and j r < S^2 is divided by a multiply
// with ceil(2^64 / S) (exact while S < 2^21: j r S < 2^63); a stratum holds q
// or q + 1 positions, whose remainders come from a multiply with
// floor((2^64 - 1) / size), at most two too small.
struct SampleDraw {
  uint64_t inv, magic0, magic1, seed;
  uint32_t q, r, S;
  __device__ __forceinline__ SampleDraw(uint32_t m, uint32_t S_, uint64_t seed_)
      : seed(seed_), S(S_) {
    q = m / S;
    r = m - q * S;
    inv = ~0ULL / S + 1;  // (S = 1 wraps to 0: r is 0 then)
    magic0 = ~0ULL / q;   // q >= 1 (S <= m)
    magic1 = ~0ULL / (q + 1);
  }
  __device__ __forceinline__ uint32_t position(uint32_t j) const {
    const uint64_t x = (uint64_t)j * r;
    const uint32_t f0 = (uint32_t)__umul64hi(x, inv);
    const uint32_t f1 = (uint32_t)__umul64hi(x + r, inv);
    const uint32_t size = q + (f1 - f0);
    const uint64_t z = splitmix64_at(seed, j);
    uint64_t rem = z - __umul64hi(z, f1 != f0 ? magic1 : magic0) * size;
    if (rem >= size) rem -= size;
    if (rem >= size) rem -= size;
    return j * q + f0 + (uint32_t)rem;
  }
};
static_assert(16u * 11 * kMaxK < (1u << 21), "sample counts the exact division covers");

// Start of a one-segment call, made by the first launch itself (n == 0: the
// level's segments come from its plan).
struct PlainStart {
  uint64_t n = 0;
  uint32_t k = 0;     // buckets
  uint32_t S = 0;     // samples
  uint32_t nch = 0;   // chunks
  LocalPlan local;
};

// Steps 1 and 2a: stratified random samples, each carrying its position, drawn
// straight into the registers of the CTA that sorts them.  Sample chunk c of
// nschunks takes samples c, c + nschunks, ...: every chunk represents the whole
// segment (the merge below takes its ranges from one chunk), in position order
// when the segment's level input is (in_order).  A segment with one chunk is
// done here.  Serves the chunks of more than min_len samples.  A one-segment
// call's control block and segment are written here too.
template <int NT, int IT, int MINB>
__global__ void __launch_bounds__(NT, MINB)
k_sample_sort(DevState* st, LevelSeg* segs, Src src, uint64_t* samp_key, uint32_t* samp_idx,
              uint64_t* ssamp_key, uint32_t* ssamp_idx, int in_order, uint32_t min_len,
              PlainStart ps, LevelParams P) {
  pdl_entry();
  constexpr uint32_t kCap = NT * IT;
  extern __shared__ __align__(16) unsigned char smem_raw[];
  CtaSortSmem s;
  s.k = (uint64_t*)smem_raw;
  s.i = (uint32_t*)(s.k + kCap);
  s.hist = s.i + kCap;
  __shared__ uint64_t red[2 * NT / 32];
  __shared__ uint64_t scan_sm[NT / 32];
  LevelSeg sg;
  if (ps.n) {
    fill_segment(sg, 0, (uint32_t)ps.n, ps.k, ps.S, ps.nch, P, 0, KeyRange{0, ~0ULL});
    sg.samp_off = sg.chunk_off = sg.hist_off = sg.schunk_off = sg.bkt_off = sg.delta = 0;
    if (blockIdx.x == 0 && threadIdx.x == 0) {
      reset_state(st, ps.local);
      segs[0] = sg;
      st->levels_used = P.level;
      st->cur_nseg = 1;
      st->total_samples = sg.S;
      st->total_chunks = sg.nchunks;
      st->total_hist = (uint64_t)sg.k * sg.nunits;
      st->total_schunks = sg.nschunks;
      st->total_buckets = sg.k;
      st->l1_nb = sg.k;
      st->level_elems[0] = sg.m;
    }
  }
  const uint64_t total = ps.n ? sg.nschunks : st->total_schunks;
  for (uint64_t c = blockIdx.x; c < total; c += gridDim.x) {
    if (!ps.n) sg = segs[c];  // (one sample chunk a segment)
    const uint32_t cl = (uint32_t)(c - sg.schunk_off);
    const uint32_t each = sg.S / sg.nschunks, more = sg.S % sg.nschunks;
    const uint32_t len = each + (cl < more ? 1u : 0u);
    if (len <= min_len || len > kCap) continue;
    const uint64_t base = sg.samp_off + (uint64_t)cl * each + min(cl, more);
    const SampleDraw draw(sg.m, sg.S, sg.seed);
    uint64_t key[IT];
    uint32_t idx[IT];
#pragma unroll
    for (int r = 0; r < IT; ++r) {
      const uint32_t e = r * NT + threadIdx.x;
      if (e < len) {
        const uint32_t pos = draw.position(cl + e * sg.nschunks);
        const uint64_t at = sg.start + pos;
        key[r] = load_key(src, at);
        idx[r] = src.idx ? src.idx[at] : pos;
      }
    }
    cta_sort_pairs<NT, IT>(key, idx, len,
                           [&] { return in_order == kOrderAuto ? st->l1_ordered != 0
                                                               : in_order != 0; },
                           s, red, scan_sm, nullptr);
    uint64_t* ok = sg.nschunks == 1 ? ssamp_key : samp_key;
    uint32_t* oi = sg.nschunks == 1 ? ssamp_idx : samp_idx;
    for (uint32_t t = threadIdx.x; t < len; t += NT) {
      ok[base + t] = s.k[t];
      oi[base + t] = s.i[t];
    }
    __syncthreads();
  }
}

// Step 2b: merge the sorted chunks of a one-segment level.  CTA i takes the
// pairs between two quantiles of chunk 0 (chunks are alike, so about S/gridDim
// pairs): a binary search per chunk finds their runs, the sum of the runs'
// starts is their place in the sorted sample (the rank of an element is its
// rank in its own sorted sequence plus its ranks in the others, Appendix "Fast
// Work-Inefficient Ranking"), and the CTA sorts them in shared memory.  A range
// that does not fit is placed pair by pair by its ranks.
//   163,840 samples: ranking every pair in every other chunk
//   81 us, this form 19 us.
constexpr int kMergeThreads = 512;
constexpr int kMergeItems = 8;
constexpr uint32_t kMergeRange = 1024;   // pairs a CTA is given on average
constexpr uint32_t kMaxSampleChunks = 96;
constexpr uint32_t kMinSplitSample = 5120;   // (larger samples are cut into chunks)
static_assert(16u * 11 * kMaxK <= kMaxSampleChunks * kSampleChunk / 2, "a run per sample chunk");
__global__ void __launch_bounds__(kMergeThreads, 2)
k_sample_merge(const LevelSeg* segs, const uint64_t* samp_key, const uint32_t* samp_idx,
               uint64_t* ssamp_key, uint32_t* ssamp_idx) {
  pdl_entry();
  constexpr int NT = kMergeThreads, IT = kMergeItems;
  constexpr uint32_t kCap = NT * IT;
  extern __shared__ __align__(16) unsigned char smem_raw[];
  CtaSortSmem s;
  s.k = (uint64_t*)smem_raw;
  s.i = (uint32_t*)(s.k + kCap);
  s.hist = s.i + kCap;
  __shared__ uint64_t red[2 * NT / 32];
  __shared__ uint64_t scan_sm[NT / 32];
  __shared__ uint32_t s_lo[kMaxSampleChunks];       // first pair of every chunk's run
  __shared__ uint32_t s_at[kMaxSampleChunks + 1];   // runs' starts in the range
  const LevelSeg& sg = segs[0];
  const uint32_t nch = sg.nschunks, S = sg.S, tid = threadIdx.x;
  const uint32_t each = S / nch, more = S % nch;
  auto chunk_len = [&](uint32_t c) { return each + (c < more ? 1u : 0u); };
  auto chunk_at = [&](uint32_t c) { return sg.samp_off + (uint64_t)c * each + min(c, more); };
  // pairs of chunk c below the pair (k, i)
  auto rank_in = [&](uint32_t c, uint64_t k, uint32_t i) {
    const uint64_t b = chunk_at(c);
    uint32_t lo = 0, hi = chunk_len(c);
    while (lo < hi) {
      const uint32_t mid = (lo + hi) >> 1;
      const uint64_t km = samp_key[b + mid];
      if (km < k || (km == k && samp_idx[b + mid] < i)) lo = mid + 1;
      else hi = mid;
    }
    return lo;
  };
  const uint32_t l0 = chunk_len(0);
  const uint32_t q0 = (uint32_t)(((uint64_t)blockIdx.x * l0) / gridDim.x);
  const uint32_t q1 = (uint32_t)(((uint64_t)(blockIdx.x + 1) * l0) / gridDim.x);
  const bool last = blockIdx.x + 1 == gridDim.x;
  if (tid < 2 * nch) {  // both ends of every run at once
    const uint32_t c = tid >> 1, q = tid & 1 ? q1 : q0;
    uint32_t r;
    if (tid & 1 ? last : blockIdx.x == 0) r = tid & 1 ? chunk_len(c) : 0u;
    else r = rank_in(c, samp_key[chunk_at(0) + q], samp_idx[chunk_at(0) + q]);
    if (tid & 1) s_at[c + 1] = r;
    else s_lo[c] = r;
  }
  __syncthreads();
  if (tid == 0) {
    uint32_t run = 0;
    s_at[0] = 0;
    for (uint32_t c = 0; c < nch; ++c) {
      run += s_at[c + 1] - s_lo[c];
      s_at[c + 1] = run;
    }
  }
  __syncthreads();
  const uint32_t cnt = s_at[nch];
  uint64_t out = sg.samp_off;
  for (uint32_t c = 0; c < nch; ++c) out += s_lo[c];
  auto source = [&](uint32_t e) {  // slot of the range's pair e
    uint32_t lo = 0, hi = nch;
    while (hi - lo > 1) {
      const uint32_t mid = (lo + hi) >> 1;
      if (s_at[mid] <= e) lo = mid;
      else hi = mid;
    }
    return chunk_at(lo) + s_lo[lo] + (e - s_at[lo]);
  };
  if (cnt == 0) return;
  if (cnt > kCap) {
    for (uint32_t e = tid; e < cnt; e += NT) {
      const uint64_t at = source(e);
      const uint64_t k = samp_key[at];
      const uint32_t i = samp_idx[at];
      uint64_t r = sg.samp_off;
      for (uint32_t c = 0; c < nch; ++c) r += rank_in(c, k, i);
      ssamp_key[r] = k;
      ssamp_idx[r] = i;
    }
    return;
  }
  uint64_t key[IT];
  uint32_t idx[IT];
#pragma unroll
  for (int r = 0; r < IT; ++r) {
    const uint32_t e = r * NT + tid;
    if (e < cnt) {
      const uint64_t at = source(e);
      key[r] = samp_key[at];
      idx[r] = samp_idx[at];
    }
  }
  cta_sort_pairs<NT, IT>(key, idx, cnt, [] { return false; }, s, red, scan_sm, nullptr);
  for (uint32_t t = tid; t < cnt; t += NT) {
    ssamp_key[out + t] = s.k[t];
    ssamp_idx[out + t] = s.i[t];
  }
}

// Shared-memory carve-up of the classify / scatter kernels.
constexpr int kCT = 2048;                       // keys per classify pipeline stage
constexpr int kCStages = 3;                     // classify stages at level 1 (2 in flight)
constexpr int kCStagesDeep = 2;                 // deeper levels: fewer stages, more CTAs per SM
constexpr int kCItems = kCT / kPartThreads;     // 8 keys per lane per stage

struct PartSmem {
  Splitters sp;
  uint32_t* hist;      // [K]   classify: counts;  scatter: running offsets
  uint32_t* sbase;     // [K+1] scatter: sub-tile bucket starts
  uint16_t* wcnt;      // [kPartWarps][cnt_stride(K)] scatter: per-warp counts / bases
  uint32_t* dlt;       // scatter: [K] output position minus sub-tile run start, per bucket
  uint8_t* wwin;       // [kPartWarps][K] scatter: per-warp winner lane of each bucket
  unsigned char* buf;  // classify: kCStages key stages; scatter: two sub-tile buffers
};

// mode: bit 0 the classifier (0 tree, 1 table), bit 1 no tie-breaking.
__host__ __device__ inline size_t part_common_bytes(uint32_t kmax, int mode) {
  const size_t Kp = next_pow2_u32(kmax);
  size_t b = (mode & 1) == 0 ? Kp * 8 : table_bytes((uint32_t)Kp);
  b += (size_t)kmax * 8 + (size_t)kmax * 4 + (size_t)kmax * 2 + (size_t)kmax * 4;
  return (b + 15) & ~(size_t)15;
}

__host__ __device__ inline size_t classify_smem_bytes(uint32_t kmax, int mode, int stages) {
  return part_common_bytes(kmax, mode) + (size_t)stages * kCT * 8;
}

__device__ inline PartSmem carve(unsigned char* base, uint32_t kmax, int mode) {
  PartSmem s;
  const size_t Kp = next_pow2_u32(kmax);
  unsigned char* p = base;
  s.sp.mode = mode & 1;
  s.sp.ntb = (mode >> 1) & 1;
  s.sp.tree = nullptr;
  s.sp.tbl = nullptr;
  if (s.sp.mode == 0) {
    s.sp.tree = (uint64_t*)p;
    p += Kp * 8;
  } else {
    s.sp.tbl = (uint16_t*)p;
    p += table_bytes((uint32_t)Kp);
  }
  s.sp.key = (uint64_t*)p; p += (size_t)kmax * 8;
  s.sp.idx = (uint32_t*)p; p += (size_t)kmax * 4;
  s.hist = (uint32_t*)p; p += (size_t)kmax * 4;
  s.sp.rend = (uint16_t*)p; p += (size_t)kmax * 2;
  p = base + part_common_bytes(kmax, mode);
  s.sbase = nullptr;
  s.wcnt = nullptr;
  s.dlt = nullptr;
  s.wwin = nullptr;
  s.buf = p;
  return s;
}

// Dynamic shared memory the wide (512-thread, 4096-key) scatter may use: the
// device's opt-in limit minus the kernel's static shared memory, found when
// the kernel attributes are set (0 until then, or if CUDA refused).  The wide
// scatter runs only when its carve-up fits.
static size_t g_wide_scatter_smem_max = 0;

// Shared memory of the staged scatter with NW warps and ST-key sub-tiles.
// The stable scatter keeps per-warp counters and winner slots per bucket; the
// unstable one a single 32-bit counter per bucket (in place of the former).
__host__ __device__ inline size_t scatter_smem_bytes(uint32_t kmax, int mode, int nw, int st,
                                                     bool stable = true) {
  size_t b = part_common_bytes(kmax, mode);
  b += (size_t)(kmax + 1) * 4 + 4;
  b += stable ? (size_t)nw * cnt_stride(kmax) * 2 : (size_t)kmax * 4;
  b += (size_t)kmax * 4;
  b += stable ? (size_t)nw * kmax : 0;
  b = (b + 15) & ~(size_t)15;
  return b + 2 * ((size_t)st * (8 + 4 + 2) + 16);
}

__device__ inline PartSmem carve_scatter(unsigned char* base, uint32_t kmax, int mode, int nw,
                                         bool stable = true) {
  PartSmem s = carve(base, kmax, mode);
  unsigned char* p = base + part_common_bytes(kmax, mode);
  s.sbase = (uint32_t*)p;
  p += (size_t)(kmax + 1) * 4 + 4;
  s.wcnt = (uint16_t*)p;
  p += stable ? (size_t)nw * cnt_stride(kmax) * 2 : (size_t)kmax * 4;
  s.dlt = (uint32_t*)p;
  p += (size_t)kmax * 4;
  s.wwin = (uint8_t*)p;
  p += stable ? (size_t)nw * kmax : 0;
  s.buf = (unsigned char*)(((uintptr_t)p + 15) & ~(uintptr_t)15);
  return s;
}

// Steps 4 + 5a: classify every element and count, per chunk of W elements,
// how many fall into each bucket.  hist is laid out per segment bucket-major:
// hist[hist_off + b * nchunks + chunk].  The chunk's keys stream through a
// STAGES-deep cp.async pipeline of kCT-key stages in shared memory.  Level 1
// (few long chunks) runs 3 stages at 3 CTAs per SM; deeper levels (many
// short chunks, each loading its segment's splitters) measured faster with 2
// stages at 4 CTAs per SM.
template <int STAGES>
__global__ void __launch_bounds__(kPartThreads, STAGES == 2 ? 4 : 3)
k_classify_count(const DevState* st, const LevelSeg* segs, Src src, const uint64_t* ssk,
                 const uint32_t* ssi, uint32_t* hist, uint32_t W, uint32_t kmax, int mode) {
  pdl_entry();
  extern __shared__ __align__(16) unsigned char smem_raw[];
  PartSmem sm = carve(smem_raw, kmax, mode);
  uint64_t* stage = (uint64_t*)sm.buf;
  const uint64_t pol = l2_evict_first_policy();
  const uint64_t total = st->total_chunks;
  const uint32_t G = st->cur_nseg;
  const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
  uint32_t cur_g = 0xffffffffu;
  for (uint64_t c = blockIdx.x; c < total; c += gridDim.x) {
    const uint32_t g = seg_of_chunk(src.chunk_seg, G, c);
    const LevelSeg sg = segs[g];
    __syncthreads();
    if (g != cur_g) {
      load_splitters<kPartThreads>(sg, ssk, ssi, sm.sp);
      cur_g = g;
    }
    for (uint32_t b = threadIdx.x; b < sg.k; b += kPartThreads) sm.hist[b] = 0;
    const uint64_t cl = c - sg.chunk_off;
    const uint64_t cs = sg.start + cl * sg.W;
    const uint64_t ce = umin64(cs + sg.W, sg.start + sg.m);
    const uint64_t nst = (ce - cs + kCT - 1) / kCT;
    auto issue = [&](uint64_t s) {
      if (s < nst) {
        const uint64_t b0 = cs + s * kCT;
        const uint32_t len = (uint32_t)umin64(kCT, ce - b0);
        uint64_t* dst = stage + (s % STAGES) * kCT;
        for (uint32_t t = threadIdx.x; t < len; t += kPartThreads)
          cp_async_8(dst + t, src.key + b0 + t, pol);
      }
      cp_async_commit();
    };
#pragma unroll
    for (int s = 0; s < STAGES - 1; ++s) issue(s);
    for (uint64_t s = 0; s < nst; ++s) {
      cp_async_wait<STAGES - 2>();
      __syncthreads();
      issue(s + STAGES - 1);
      const uint64_t b0 = cs + s * kCT;
      const uint32_t len = (uint32_t)umin64(kCT, ce - b0);
      const uint64_t* stg = stage + (s % STAGES) * kCT;
      const uint32_t q0 = (uint32_t)warp * (kCItems * 32) + lane;
      uint64_t key[kCItems];
#pragma unroll
      for (int r = 0; r < kCItems; ++r) {
        const uint32_t q = q0 + r * 32;
        const uint64_t k = q < len ? stg[q] : 0;
        key[r] = src.map_f64 ? f64_to_ordered(k) : k;
      }
      uint32_t bk[kCItems];
      // positions are read only when a key ties with a splitter key, and
      // never past the stage (a padding slot's key 0 may tie; its result is
      // discarded)
      classify_batch<kCItems>(key, bk, [&](int r) {
        const uint32_t q = q0 + r * 32;
        if (q >= len) return 0u;
        const uint64_t pos = b0 + q;
        return src.idx ? src.idx[pos] : (uint32_t)(pos - sg.start);
      }, sm.sp);
      if (src.bid) {
#pragma unroll
        for (int r = 0; r < kCItems; ++r)
          if (q0 + r * 32 < len) src.bid[b0 + q0 + r * 32] = (uint16_t)bk[r];
      }
      // runs of one bucket across the warp (duplicate-heavy inputs) take one
      // atomic per warp and slot; otherwise one atomic per key
      const uint32_t bw = __shfl_sync(0xffffffffu, bk[0], 0);
      if (__popc(__ballot_sync(0xffffffffu, bk[0] == bw)) > 8) {
#pragma unroll
        for (int r = 0; r < kCItems; ++r) {
          const bool v = q0 + r * 32 < len;
          const uint32_t b = bk[r];
          const uint32_t bl = __shfl_sync(0xffffffffu, b, 0);
          if (__all_sync(0xffffffffu, v && b == bl)) {
            if (lane == 0) atomicAdd(&sm.hist[bl], 32u);
          } else if (v) {
            atomicAdd(&sm.hist[b], 1u);
          }
        }
      } else {
#pragma unroll
        for (int r = 0; r < kCItems; ++r)
          if (q0 + r * 32 < len) atomicAdd(&sm.hist[bk[r]], 1u);
      }
    }
    cp_async_wait<0>();
    __syncthreads();
    for (uint32_t b = threadIdx.x; b < sg.k; b += kPartThreads)
      hist[sg.hist_off + (uint64_t)b * sg.nunits + cl] = sm.hist[b];
  }
}

// Step 5b: exclusive scan of the histogram counters: sums of tiles of
// kScanTile, then every CTA adds up the sums before its tile (a few thousand
// words at most) and scans the tile.
__global__ void __launch_bounds__(1024)
k_scan_reduce(const DevState* st, const uint32_t* a, uint32_t* sums) {
  pdl_entry();
  __shared__ uint64_t sm[32];
  const uint64_t total = st->total_hist;
  const uint64_t base = (uint64_t)blockIdx.x * kScanTile;
  if (base >= total) return;
  uint64_t v = 0;
  for (int r = 0; r < 4; ++r) {
    const uint64_t i = base + threadIdx.x * 4 + r;
    if (i < total) v += a[i];
  }
  uint64_t tot;
  block_excl_scan_u64<1024>(v, &tot, sm);
  if (threadIdx.x == 0) sums[blockIdx.x] = (uint32_t)tot;
}

// One tile of the scan by 1024 threads; returns the tile's sum.
__device__ __forceinline__ uint32_t scan_tile(uint32_t* a, uint64_t base, uint64_t total,
                                              uint32_t before, uint64_t* sm) {
  uint32_t x[4];
  uint64_t v = 0;
  for (int r = 0; r < 4; ++r) {
    const uint64_t i = base + threadIdx.x * 4 + r;
    x[r] = i < total ? a[i] : 0;
    v += x[r];
  }
  uint64_t tot;
  uint64_t run = block_excl_scan_u64<1024>(v, &tot, sm) + before;
  for (int r = 0; r < 4; ++r) {
    const uint64_t i = base + threadIdx.x * 4 + r;
    if (i < total) a[i] = (uint32_t)run;
    run += x[r];
  }
  return (uint32_t)tot;
}

__global__ void __launch_bounds__(1024)
k_scan_down(const DevState* st, uint32_t* a, const uint32_t* sums) {
  pdl_entry();
  __shared__ uint64_t sm[32];
  const uint64_t total = st->total_hist;
  const uint64_t base = (uint64_t)blockIdx.x * kScanTile;
  if (base >= total) return;
  uint64_t pre = 0, before;
  for (uint32_t t = threadIdx.x; t < blockIdx.x; t += 1024) pre += sums[t];
  block_excl_scan_u64<1024>(pre, &before, sm);
  scan_tile(a, base, total, (uint32_t)before, sm);
}

// Step 5c: scatter.  Every chunk streams through two ST-key sub-tile buffers
// (cp.async: sub-tile s+1 loads while s is processed).  Every element gets a
// rank among the elements of its bucket in the sub-tile; the sub-tile is then
// counting-sorted by bucket into its own buffer and every bucket's run is
// written out contiguously (write-combining through shared memory).
//   STABLE   warp w owns IT*32 consecutive elements; ranks come from
//            warp-synchronous peer counting (warp order, then lane order =
//            input order), so buckets keep input order -- the layout of the
//            partition step.
//   unstable one shared-memory atomic per element on its bucket's counter:
//            buckets come out in no particular order, which a full sort's
//            deeper levels may do (the in-SM sort orders (key, position)
//            pairs).
template <int NT, int ST, bool STABLE>
__global__ void __launch_bounds__(NT, (NT <= 256 ? 2 : 1))
k_scatter(const DevState* st, const LevelSeg* segs, Src src, const uint64_t* ssk,
          const uint32_t* ssi, const uint32_t* hist_scan, Dst dst, uint32_t W, uint32_t kmax,
          int unmap_out, int mode) {
  pdl_entry();
  constexpr int NW = NT / 32;
  constexpr int IT = ST / NT;
  static_assert(IT * 32 * NW == ST, "warp w owns IT*32 consecutive keys of a sub-tile");
  // keys, positions, bucket ids (+16 bytes: the staged ids start at an even
  // position, one before the sub-tile when it starts at an odd one)
  constexpr size_t BUFB = (size_t)ST * (8 + 4 + 2) + 16;
  extern __shared__ __align__(16) unsigned char smem_raw[];
  PartSmem sm = carve_scatter(smem_raw, kmax, mode, NW, STABLE);
  uint32_t* cntu = reinterpret_cast<uint32_t*>(sm.wcnt);  // unstable: one counter per bucket
  if constexpr (!STABLE) {
    for (uint32_t b = threadIdx.x; b < kmax; b += NT) cntu[b] = 0;
  }
  __shared__ uint64_t scan_sm[NW];
  // sub-tile buffer i: keys, positions, bucket ids (addressed arithmetically so
  // that no descriptor array lives in local memory)
  struct Buf {
    uint64_t* key;
    uint32_t* idx;
    uint16_t* b;
  };
  auto buf_of = [&](uint64_t i) {
    unsigned char* p = sm.buf + (size_t)(i & 1) * BUFB;
    Buf r;
    r.key = (uint64_t*)p;
    r.idx = (uint32_t*)(p + (size_t)ST * 8);
    r.b = (uint16_t*)(p + (size_t)ST * 12);
    return r;
  };
  const uint64_t pol = l2_evict_first_policy();
  const uint64_t pol_keep = l2_evict_last_policy();
  const uint64_t total = st->total_chunks;
  const uint32_t G = st->cur_nseg;
  const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
  const uint32_t ltmask = lanemask_lt();
  const uint32_t kst = cnt_stride(kmax);
  uint16_t* my_cnt = sm.wcnt + (size_t)warp * kst;
  uint8_t* my_win = sm.wwin + (size_t)warp * kmax;
  uint32_t cur_g = 0xffffffffu;
  for (uint64_t c = blockIdx.x; c < total; c += gridDim.x) {
    const uint32_t g = seg_of_chunk(src.chunk_seg, G, c);
    const LevelSeg sg = segs[g];
    __syncthreads();
    if (g != cur_g) {
      load_splitters<NT>(sg, ssk, ssi, sm.sp);
      cur_g = g;
    }
    const uint32_t k = sg.k;
    const int nbits = k > 32 ? 5 : (int)ceil_log2_dev(k);
    const uint64_t cl = c - sg.chunk_off;
    for (uint32_t b = threadIdx.x; b < k; b += NT)
      sm.hist[b] = (uint32_t)(hist_scan[sg.hist_off + (uint64_t)b * sg.nunits + cl] + sg.delta);
    const uint64_t cs = sg.start + cl * sg.W;
    const uint64_t ce = umin64(cs + sg.W, sg.start + sg.m);
    const uint64_t nst = (ce - cs + ST - 1) / ST;
    auto issue = [&](uint64_t s) {
      if (s < nst) {
        const uint64_t b0 = cs + s * ST;
        const uint32_t len = (uint32_t)umin64(ST, ce - b0);
        const Buf B = buf_of(s);
        for (uint32_t t = threadIdx.x; t < len; t += NT) {
          cp_async_8(B.key + t, src.key + b0 + t, pol);
          if (src.idx) cp_async_4(B.idx + t, src.idx + b0 + t, pol);
        }
        if (src.bid) {  // bucket ids as 4-byte pairs from the even position at or below b0
          const uint64_t w0 = b0 >> 1;
          const uint32_t nw = (uint32_t)(((b0 + len + 1) >> 1) - w0);
          const uint32_t* gw = reinterpret_cast<const uint32_t*>(src.bid) + w0;
          for (uint32_t t = threadIdx.x; t < nw; t += NT)
            cp_async_4(reinterpret_cast<uint32_t*>(B.b) + t, gw + t, pol);
        }
      }
      cp_async_commit();
    };
    issue(0);
    for (uint64_t s = 0; s < nst; ++s) {
      cp_async_wait<0>();
      __syncthreads();
      issue(s + 1);
      const Buf B = buf_of(s);
      const uint64_t b0 = cs + s * ST;
      const uint32_t len = (uint32_t)umin64(ST, ce - b0);
      const uint32_t q0 = (uint32_t)warp * (IT * 32) + lane;
      uint64_t key[IT];
      uint32_t idx[IT];
      uint32_t bk[IT];
      uint32_t lrank[IT];
#pragma unroll
      for (int r = 0; r < IT; ++r) {
        const uint32_t q = q0 + r * 32;
        const bool v = q < len;
        const uint64_t kv = v ? B.key[q] : 0;
        key[r] = src.map_f64 ? f64_to_ordered(kv) : kv;
        idx[r] = v ? (src.idx ? B.idx[q] : (uint32_t)(b0 + q - sg.start)) : 0;
      }
      if (src.bid) {
        const uint16_t* bh = B.b + (b0 & 1);
#pragma unroll
        for (int r = 0; r < IT; ++r) {
          const uint32_t q = q0 + r * 32;
          bk[r] = q < len ? bh[q] : 0u;
        }
      } else {
        classify_batch<IT>(key, bk, [&](int r) { return idx[r]; }, sm.sp);
      }
      if constexpr (!STABLE) {
#pragma unroll
        for (int r = 0; r < IT; ++r) {
          const bool v = q0 + r * 32 < len;
          bk[r] = v ? bk[r] : 0xffffffffu;
          lrank[r] = v ? atomicAdd(&cntu[bk[r]], 1u) : 0u;
        }
      } else {
      for (uint32_t q = lane; q < (k + 1) / 2; q += 32) ((uint32_t*)my_cnt)[q] = 0;
      __syncwarp();
#pragma unroll
      for (int r = 0; r < IT; ++r) {
        const bool v = q0 + r * 32 < len;
        const uint32_t b = v ? bk[r] : 0xffffffffu;
        bk[r] = b;
        // peers = the lanes holding the same bucket.  Up to 32 buckets the
        // bucket bits are compared by ballots; beyond, every lane first writes
        // its lane id to the warp's slot of its bucket, and the lane id that
        // stayed there (one per distinct bucket) is compared instead: 5
        // ballots whatever k is.
        uint32_t w = b;
        if (k > 32) {
          if (v) my_win[b] = (uint8_t)lane;
          __syncwarp();
          w = v ? my_win[b] : 0u;
          __syncwarp();
        }
        uint32_t peers = __ballot_sync(0xffffffffu, v);
        // every lane kept its own slot: the warp's buckets are distinct, so
        // each lane is its bucket's only peer (the common case for k >> 32)
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
      }  // STABLE
      __syncthreads();
      {  // per bucket (each thread a run of buckets): exclusive prefix over the
         // warps' counts, in place; an exclusive scan of the bucket totals then
         // places every bucket's run in the sub-tile, and the running output
         // offsets advance by the totals
        const uint32_t per = (k + NT - 1) / NT;
        const uint32_t bb0 = threadIdx.x * per;
        const uint32_t bb1 = bb0 + per < k ? bb0 + per : k;
        uint32_t loc = 0;
        uint32_t b0s = bb0;
        if constexpr (STABLE) {
          // two buckets at a time: their 16-bit counters share a 32-bit word
          // (rows have even length, bb0 is even when per is), and no count or
          // prefix exceeds the sub-tile, so halfword adds never carry
          for (; (per & 1) == 0 && b0s + 1 < bb1; b0s += 2) {
            uint32_t tot2 = 0;
#pragma unroll
            for (int w = 0; w < NW; ++w) {
              uint32_t* cw = reinterpret_cast<uint32_t*>(sm.wcnt + (size_t)w * kst + b0s);
              const uint32_t cnt2 = *cw;
              *cw = tot2;
              tot2 = __vadd2(tot2, cnt2);
            }
            sm.sbase[b0s] = tot2 & 0xffffu;
            sm.sbase[b0s + 1] = tot2 >> 16;
            loc += (tot2 & 0xffffu) + (tot2 >> 16);
          }
        }
        for (uint32_t b = b0s; b < bb1; ++b) {
          uint32_t tot = 0;
          if constexpr (STABLE) {
#pragma unroll
            for (int w = 0; w < NW; ++w) {
              const uint32_t cnt = sm.wcnt[(size_t)w * kst + b];
              sm.wcnt[(size_t)w * kst + b] = (uint16_t)tot;
              tot += cnt;
            }
          } else {
            tot = cntu[b];
            cntu[b] = 0;  // ready for the next sub-tile (its atomics follow barriers)
          }
          sm.sbase[b] = tot;
          loc += tot;
        }
        uint64_t tot;
        uint32_t run = (uint32_t)block_excl_scan_u64<NT>(loc, &tot, scan_sm);
        for (uint32_t b = bb0; b < bb1; ++b) {
          const uint32_t t = sm.sbase[b];
          sm.sbase[b] = run;
          sm.dlt[b] = sm.hist[b] - run;  // modulo 2^32: positions are below 2^32
          sm.hist[b] += t;
          run += t;
        }
      }
      __syncthreads();
      // counting-sort the sub-tile by bucket into its own buffer
#pragma unroll
      for (int r = 0; r < IT; ++r) {
        const uint32_t b = bk[r];
        if (b != 0xffffffffu) {
          const uint32_t q = sm.sbase[b] + (STABLE ? (uint32_t)my_cnt[b] : 0u) + lrank[r];
          B.key[q] = key[r];
          B.idx[q] = idx[r];
          B.b[q] = (uint16_t)b;
        }
      }
      __syncthreads();
      for (uint32_t q = threadIdx.x; q < len; q += NT) {
        const uint32_t b = B.b[q];
        const uint64_t d = (uint32_t)(sm.dlt[b] + q);
        const uint64_t kv = B.key[q];
        st_keep_u64(dst.key + d, unmap_out ? ordered_to_f64(kv) : kv, pol_keep);
        st_keep_u32(dst.idx + d, B.idx[q], pol_keep);
      }
    }
    cp_async_wait<0>();
  }
}

// Collect the buckets of the level: bucket sizes follow from the scanned
// histogram.  Buckets that fit one SM, equality buckets of a stable level on
// input in position order (both bounding splitters share one key, so every
// element has that key and the stable scatter left them in position order)
// and empty ones are final; the rest become segments of the next level.
// Otherwise an equality bucket is a bucket like any other, and its elements
// arrive at the in-SM sort in no particular order.
__device__ __forceinline__ void collect_buckets(DevState* st, const LevelSeg* segs,
                                                const uint64_t* ssk, const uint32_t* hist_scan,
                                                SegIn* list_out, int par_out, FinalItem* items,
                                                const LevelParams& P, uint16_t where,
                                                int last_level, int emit_final,
                                                uint64_t* offsets_out) {
  const uint64_t total = st->total_buckets;
  const uint32_t G = st->cur_nseg;
  // buckets keep position order only if the level is stable and its input
  // was in position order (level 1 records this for the levels below)
  const bool stable = P.stable == kOrderAuto ? l1_auto_ordered(st) : P.stable != 0;
  const bool in_order = P.in_order == kOrderAuto ? st->l1_ordered != 0 : P.in_order != 0;
  const bool ordered = stable && in_order;
  if (P.level == 1 && blockIdx.x == 0 && threadIdx.x == 0) st->l1_ordered = ordered ? 1u : 0u;
  for (uint64_t f = (uint64_t)blockIdx.x * blockDim.x + threadIdx.x; f < total;
       f += (uint64_t)gridDim.x * blockDim.x) {
    const uint32_t g = find_seg(segs, G, f, [](const LevelSeg& x) { return x.bkt_off; });
    const LevelSeg& sg = segs[g];
    const uint32_t b = (uint32_t)(f - sg.bkt_off);
    const uint64_t start = hist_scan[sg.hist_off + (uint64_t)b * sg.nunits] + sg.delta;
    const uint64_t end = (b + 1 < sg.k)
                             ? hist_scan[sg.hist_off + (uint64_t)(b + 1) * sg.nunits] + sg.delta
                             : sg.start + sg.m;
    const uint32_t size = (uint32_t)(end - start);
    if (offsets_out) {
      offsets_out[b] = start - sg.start;
      if (b == 0) offsets_out[sg.k] = sg.m;
    }
    if (P.level == 1) atomicMax(&st->max_bucket_l1, size);
    if (!emit_final || size == 0) continue;
    // its keys lie between its splitters (the segment's bounds at the ends)
    KeyRange kr = sg.range;
    uint32_t known = sg.known;
    if (b >= 1) {
      kr.lo = ssk[sg.samp_off + ((uint64_t)b * sg.S) / sg.k];
      known |= 1u;
    }
    if (b + 1 < sg.k) {
      kr.hi = ssk[sg.samp_off + ((uint64_t)(b + 1) * sg.S) / sg.k];
      known |= 2u;
    }
    const bool eq = ordered && b >= 1 && b + 1 < sg.k && kr.lo == kr.hi;
    if (eq || size <= kBucketCap || last_level) {
      FinalItem it;
      it.start = start;
      it.aux = kr.lo;
      it.bits = known != 3u          ? kBitsUnknown
                : kr.hi == kr.lo     ? (uint8_t)0
                                     : (uint8_t)(64 - __clzll((long long)(kr.hi - kr.lo)));
      it.size = size;
      it.where = where;
      it.kind = (eq || size == 1)      ? kKindCopy
                : size > kBucketCap    ? kKindBig
                : ordered              ? kKindSort
                                       : kKindSortAny;
      if (it.kind == kKindBig) atomicAdd((unsigned long long*)&st->big_items, 1ull);
      push_final(st, items, P.final_cap, it, kErrFinalCap,
                 P.refine && it.bits >= kRefineBits && it.bits != kBitsUnknown &&
                     size > st->local.rank_max);
    } else {
      SegIn s;
      s.start = start;
      s.m = size;
      s.known = known;
      s.range = kr;
      const uint32_t slot = atomicAdd(&st->nseg[par_out], 1u);
      if (slot < P.seg_cap) list_out[slot] = s;
      else atomicOr(&st->error, kErrSegCap);
    }
  }
}

__global__ void __launch_bounds__(256)
k_collect(DevState* st, const LevelSeg* segs, const uint64_t* ssk, const uint32_t* hist_scan,
          SegIn* list_out, int par_out, FinalItem* items, LevelParams P, uint16_t where,
          int last_level, int emit_final, uint64_t* offsets_out) {
  pdl_entry();
  collect_buckets(st, segs, ssk, hist_scan, list_out, par_out, items, P, where, last_level,
                  emit_final, offsets_out);
}

// Scan and collect of a one-segment level with few counters, by one CTA in one
// launch instead of three.
constexpr uint64_t kSmallScan = 4 * kScanTile;
__global__ void __launch_bounds__(1024)
k_scan_collect(DevState* st, const LevelSeg* segs, const uint64_t* ssk, uint32_t* hist,
               SegIn* list_out, int par_out, FinalItem* items, LevelParams P, uint16_t where,
               int last_level, int emit_final, uint64_t* offsets_out) {
  pdl_entry();
  __shared__ uint64_t sm[32];
  const uint64_t total = st->total_hist;
  uint32_t before = 0;
  for (uint64_t base = 0; base < total; base += kScanTile)
    before += scan_tile(hist, base, total, before, sm);
  __syncthreads();
  collect_buckets(st, segs, ssk, hist, list_out, par_out, items, P, where, last_level, emit_final,
                  offsets_out);
}

// ---------------------------------------------------------------------------
// AMS-sort overpartitioning of a one-segment step (Section 3, AMS-sort;
// Appendix "Implementation Details": b = 2 / ((1 + eps)^(1/l) - 1)).
//
//   k_fine_count    exact sizes of the K = b*k fine partitions of the same
//                   sample (fine splitter j = sorted sample floor(j*S/K)),
//                   counted per CTA in shared memory
//   k_group_*       the smallest load bound L for which the in-order greedy
//                   scan needs at most k groups (candidate bounds checked by
//                   every thread of the GPU per round), then that scan; the
//                   k-1 group boundaries are written after the sample as the
//                   splitters of the ordinary k-way step, and the segment is
//                   pointed at them
// ---------------------------------------------------------------------------
constexpr int kFineThreads = 1024;
constexpr int kFineItems = 4;
constexpr int kGreedyThreads = 1024;

__host__ __device__ inline size_t fine_smem_bytes(uint32_t K) {
  const uint32_t Kp = next_pow2_u32(K);
  return table_bytes(Kp) + (size_t)K * (8 + 4 + 4 + 2);
}

__host__ __device__ inline size_t greedy_smem_bytes(uint32_t K, uint32_t k) {
  return (size_t)(K + 1) * 4 + (size_t)(k + 1) * 4 + (size_t)(K + 1) * 4;
}

__global__ void __launch_bounds__(kFineThreads, 1)
k_fine_count(const LevelSeg* segs, Src src, const uint64_t* ssk, const uint32_t* ssi,
             uint32_t over, int ntb, uint32_t* fine_cnt) {
  pdl_entry();
  extern __shared__ __align__(16) unsigned char smem_raw[];
  LevelSeg sg = segs[0];
  const uint32_t K = sg.k * over;
  // no sample (S = 0, the sample-size rule for k = 1): no fine splitters, so
  // every element counts for fine partition 0
  sg.k = sg.S > 0 ? K : 1;
  Splitters sp;
  sp.mode = 1;
  sp.ntb = ntb;
  sp.tree = nullptr;
  unsigned char* p = smem_raw;
  sp.tbl = (uint16_t*)p;
  p += table_bytes(next_pow2_u32(K));
  sp.key = (uint64_t*)p;
  p += (size_t)K * 8;
  sp.idx = (uint32_t*)p;
  p += (size_t)K * 4;
  uint32_t* cnt = (uint32_t*)p;
  p += (size_t)K * 4;
  sp.rend = (uint16_t*)p;
  load_splitters<kFineThreads>(sg, ssk, ssi, sp);
  for (uint32_t b = threadIdx.x; b < K; b += kFineThreads) cnt[b] = 0;
  __syncthreads();
  constexpr uint64_t kSpan = (uint64_t)kFineThreads * kFineItems;
  const uint64_t m = sg.m;
  for (uint64_t base = (uint64_t)blockIdx.x * kSpan; base < m;
       base += (uint64_t)gridDim.x * kSpan) {
    uint64_t x[kFineItems];
    uint32_t b[kFineItems];
#pragma unroll
    for (int r = 0; r < kFineItems; ++r) {
      const uint64_t q = base + (uint64_t)r * kFineThreads + threadIdx.x;
      x[r] = q < m ? load_key(src, sg.start + q) : 0;
    }
    // level 1 of a one-segment step: the position is the offset in the segment
    classify_batch<kFineItems>(x, b, [&](int r) {
      return (uint32_t)(base + (uint64_t)r * kFineThreads + threadIdx.x);
    }, sp);
#pragma unroll
    for (int r = 0; r < kFineItems; ++r)
      if (base + (uint64_t)r * kFineThreads + threadIdx.x < m) atomicAdd(&cnt[b[r]], 1u);
  }
  __syncthreads();
  for (uint32_t b = threadIdx.x; b < K; b += kFineThreads)
    if (cnt[b]) atomicAdd(&fine_cnt[b], cnt[b]);
}

// End of the greedy group that starts at fine partition j0: the largest
// j in (j0, K] with P[j] - P[j0] <= L (P: prefix sums, every size <= L).
__device__ __forceinline__ uint32_t greedy_next(const uint32_t* P, uint32_t K, uint32_t j0,
                                                uint64_t L, uint32_t guess) {
  // the group starting at fine partition j0 ends after the last j with
  // P[j] - P[j0] <= L (it takes at least one partition); prefix sums are
  // below 2^32, so the target saturates there
  const uint64_t t64 = (uint64_t)P[j0] + L;
  const uint32_t target = t64 > 0xffffffffull ? 0xffffffffu : (uint32_t)t64;
  const uint32_t first = j0 + 1;
  if (first >= K || P[first] > target) return first;
  // answer in [first, K]: start at the guess and gallop to a bracket a < b
  // with P[a] <= target < P[b] (b = K + 1 stands for "past the end")
  uint32_t g = j0 + guess;
  g = g < first ? first : (g > K ? K : g);
  uint32_t a, b;
  if (P[g] <= target) {
    a = g;
    uint32_t d = 1;
    while (a + d <= K && P[a + d] <= target) {
      a += d;
      d <<= 1;
    }
    b = a + d <= K ? a + d : K + 1;
  } else {
    b = g;
    uint32_t d = 1;
    while (b - first > d && P[b - d] > target) {
      b -= d;
      d <<= 1;
    }
    a = b - first > d ? b - d : first;
  }
  while (b - a > 1) {
    const uint32_t mid = (a + b) >> 1;
    if (P[mid] <= target) a = mid; else b = mid;
  }
  return a;
}

// link[j] = link[link[j]] in the other of two arrays, for all j <= K: after i of
// these a link leads 2^i groups on.  Following single links is a chain of as
// many dependent shared-memory reads as there are groups (256 groups: 4.4 us a
// launch), doubling them takes log2 of that many short passes.
__device__ __forceinline__ void double_links(uint16_t*& link, uint16_t*& spare, uint32_t K,
                                             uint32_t nt) {
#pragma unroll 4
  for (uint32_t j = threadIdx.x; j <= K; j += nt) spare[j] = link[link[j]];
  __syncthreads();
  uint16_t* t = link;
  link = spare;
  spare = t;
}

// The greedy's bound L is searched by the whole GPU.  k_group_prep (one CTA)
// writes the prefix sums P of the fine sizes and the first bracket
// [lo, hi] (hi always feasible); every k_group_search launch spreads
// gridDim candidate bounds over the bracket the earlier rounds left, one per
// CTA, each checked by a greedy scan over P in shared memory, and keeps the
// smallest feasible candidate of the round; the next launch follows the rounds
// to the bracket below it.  Four rounds of 3 CTAs per SM narrow any bracket below
// 2^33 to one value, the smallest feasible bound; k_group_finish (one CTA) runs
// the greedy scan with it.
// search[0] = lo, search[1] = hi, search[2 + r] = smallest feasible candidate of
// round r.
constexpr int kSearchThreads = 256;
constexpr int kSearchRounds = 4;

__global__ void __launch_bounds__(kGreedyThreads, 1)
k_group_prep(const LevelSeg* segs, Overpart op) {
  pdl_entry();
  __shared__ uint64_t scan_sm[kGreedyThreads / 32];
  const LevelSeg sg = segs[0];
  const uint32_t k = sg.k, K = k * op.over;
  uint32_t* P = op.prefix;
  const uint32_t tid = threadIdx.x;
  // prefix sums of the fine sizes, one run of fine partitions per thread
  const uint32_t per = (K + kGreedyThreads - 1) / kGreedyThreads;
  const uint32_t j0 = tid * per, j1 = j0 + per < K ? j0 + per : K;
  uint64_t loc = 0, mx = 0;
  for (uint32_t j = j0; j < j1; ++j) {
    const uint64_t c = op.fine_cnt[j];
    loc += c;
    mx = c > mx ? c : mx;
    if (op.fine_out) op.fine_out[j] = c;
  }
  uint64_t n;
  uint64_t run = block_excl_scan_u64<kGreedyThreads>(loc, &n, scan_sm);
  if (tid == 0) P[0] = 0;
  for (uint32_t j = j0; j < j1; ++j) {
    run += op.fine_cnt[j];
    P[j + 1] = (uint32_t)run;  // sums below 2^32
  }
  // largest fine size (max-reduce through the scan scratch)
#pragma unroll
  for (int o = 16; o > 0; o >>= 1) {
    const uint64_t y = __shfl_xor_sync(0xffffffffu, mx, o);
    mx = y > mx ? y : mx;
  }
  if ((tid & 31) == 0) scan_sm[tid >> 5] = mx;
  __syncthreads();
  if (tid == 0) {
    uint64_t maxc = 0;
    for (int w = 0; w < kGreedyThreads / 32; ++w) maxc = scan_sm[w] > maxc ? scan_sm[w] : maxc;
    // every group holds at least ceil(n/k) in the worst case and at least the
    // largest fine partition; ceil(n/k) + maxc always needs at most k groups
    const uint64_t avg = (n + k - 1) / k;
    const uint64_t lo = avg > maxc ? avg : maxc;
    op.search[0] = lo;
    op.search[1] = avg + maxc > lo ? avg + maxc : lo;
    for (int r = 0; r < kSearchRounds; ++r) op.search[2 + r] = ~0ull;
  }
}

// The bracket after `rounds` rounds of T candidates.
__device__ __forceinline__ void group_bracket(const Overpart& op, int rounds, uint64_t T,
                                              uint64_t& lo, uint64_t& hi) {
  lo = op.search[0];
  hi = op.search[1];
  for (int r = 0; r < rounds && lo < hi; ++r) {
    const uint64_t t = op.search[2 + r];  // < T: the candidate hi is feasible
    const uint64_t span = hi - lo;
    hi = lo + (span * (t + 1)) / T;
    lo = t == 0 ? lo : lo + (span * t) / T + 1;
  }
}

__global__ void __launch_bounds__(kSearchThreads)
k_group_search(const LevelSeg* segs, Overpart op, int round) {
  pdl_entry();
  extern __shared__ __align__(16) unsigned char smem_raw[];
  uint64_t lo, hi;
  group_bracket(op, round, gridDim.x, lo, hi);
  if (lo >= hi) return;  // settled (the same for every CTA of this launch)
  const uint32_t k = segs[0].k, K = k * op.over;
  uint32_t* P = (uint32_t*)smem_raw;   // [K + 1]
  uint16_t* nxt = (uint16_t*)(P + K + 1);  // [K + 1]
  uint16_t* spare = nxt + K + 1;           // [K + 1]
  for (uint32_t j = threadIdx.x; j <= K; j += kSearchThreads) P[j] = op.prefix[j];
  __syncthreads();
  // this CTA's candidate bound (the last CTA's is hi): the end of the group
  // that would start at every fine partition (the end links to itself); the
  // bound holds if k groups from partition 0 reach the end
  const uint64_t t = blockIdx.x, T = gridDim.x;
  const uint64_t L = lo + ((hi - lo) * (t + 1)) / T;
  for (uint32_t j = threadIdx.x; j < K; j += kSearchThreads)
    nxt[j] = (uint16_t)greedy_next(P, K, j, L, op.over);
  if (threadIdx.x == 0) nxt[K] = (uint16_t)K;
  __syncthreads();
  uint32_t at = 0;  // the same in every thread
  for (uint32_t left = k; left != 0; left >>= 1) {
    if (left & 1) at = nxt[at];
    if (at == K) break;
    if (left > 1) double_links(nxt, spare, K, kSearchThreads);
  }
  if (threadIdx.x == 0 && at == K)
    atomicMin((unsigned long long*)&op.search[2 + round], (unsigned long long)t);
}

__global__ void __launch_bounds__(kGreedyThreads, 1)
k_group_finish(LevelSeg* segs, uint64_t* ssk, uint32_t* ssi, Overpart op, uint64_t T) {
  pdl_entry();
  extern __shared__ __align__(16) unsigned char smem_raw[];
  const LevelSeg sg = segs[0];
  const uint32_t k = sg.k, K = k * op.over;
  uint32_t* P = (uint32_t*)smem_raw;                 // [K + 1]
  uint32_t* first = P + K + 1;                       // [k + 1]
  uint16_t* nxt = (uint16_t*)(first + k + 1);        // [K + 1] (K <= kMaxFine < 2^16)
  uint16_t* spare = nxt + K + 1;                     // [K + 1]
  const uint32_t tid = threadIdx.x;
  for (uint32_t j = tid; j <= K; j += kGreedyThreads) P[j] = op.prefix[j];
  __syncthreads();
  // the end of the group that would start at every fine partition, in
  // parallel; the scan from partition 0 then only follows these links: the
  // starts of groups [2^i, 2^(i + 1)) are 2^i groups on from those before
  uint64_t lo, L;  // equal once settled; L is always feasible
  group_bracket(op, kSearchRounds, T, lo, L);
  for (uint32_t j = tid; j < K; j += kGreedyThreads)
    nxt[j] = (uint16_t)greedy_next(P, K, j, L, op.over);
  if (tid == 0) {
    nxt[K] = (uint16_t)K;
    first[0] = 0;
  }
  __syncthreads();
  for (uint32_t d = 1; d <= k; d <<= 1) {
    for (uint32_t g = d + tid; g < 2 * d && g <= k; g += kGreedyThreads) first[g] = nxt[first[g - d]];
    double_links(nxt, spare, K, kGreedyThreads);  // (its barrier also ends this step)
  }
  // group boundaries become the splitters of the k-way step, stored after the
  // sample: entry g (g = 1..k-1) is fine splitter first[g] (an element-free
  // sentinel above every pair when the group is empty and past the end)
  const uint64_t extra = sg.samp_off + sg.S;
  for (uint32_t g = tid + 1; g < k; g += kGreedyThreads) {
    const uint32_t f = first[g];
    uint64_t key = ~0ULL;
    uint32_t idx = ~0u;
    if (f < K) {
      const uint64_t r = ((uint64_t)f * sg.S) / K;
      key = ssk[sg.samp_off + r];
      idx = ssi[sg.samp_off + r];
    }
    ssk[extra + g] = key;
    ssi[extra + g] = idx;
  }
  if (op.first_out)
    for (uint32_t g = tid; g <= k; g += kGreedyThreads) op.first_out[g] = first[g];
  // the group of every fine partition (the sizes are no longer needed)
  for (uint32_t g = tid; g < k; g += kGreedyThreads) {
    const uint32_t end = g + 1 < k ? first[g + 1] : K;
    for (uint32_t j = first[g]; j < end; ++j) op.fine_cnt[j] = g;
  }
  __syncthreads();
  if (tid == 0) {
    segs[0].samp_off = extra;
    segs[0].S = k;
  }
}

// Without overpartitioning the fine partitions are the outputs themselves.
__global__ void k_plain_groups(const uint64_t* offsets, uint32_t k, uint64_t* fine_out,
                               uint32_t* first_out) {
  pdl_entry();
  for (uint32_t g = blockIdx.x * blockDim.x + threadIdx.x; g <= k; g += gridDim.x * blockDim.x) {
    if (fine_out && g < k) fine_out[g] = offsets[g + 1] - offsets[g];
    if (first_out) first_out[g] = g;
  }
}

inline int grid_for(uint64_t work, int per_block, int max_blocks) {
  uint64_t b = (work + per_block - 1) / per_block;
  if (b < 1) b = 1;
  return (int)umin64(b, (uint64_t)max_blocks);
}

}  // namespace

namespace {

constexpr uint32_t kBandMinW = 8192;

void launch_overpartition(const LaunchEnv& e, const LevelParams& P, DevState* st, LevelSeg* segs,
                          Src src, uint64_t* ssk, uint32_t* ssi, const Overpart& op,
                          bool fine_ids) {
  const uint32_t k = op.k, K = op.k * op.over;
  cudaMemsetAsync(op.fine_cnt, 0, (size_t)K * 4, e.stream);
  if (fine_ids) {
    launch_fine_ids(e, P, st, segs, src, ssk, ssi, op, "L1.fine_count");
  } else {
    Scope sc(e, "L1.fine_count");
    launch_kernel(e, k_fine_count, e.num_sms, kFineThreads, fine_smem_bytes(K), segs, src, ssk, ssi,
                  op.over, P.no_tie_break, op.fine_cnt);
  }
  {
    Scope sc(e, "L1.group");
    launch_kernel(e, k_group_prep, 1, kGreedyThreads, 0, segs, op);
    const int grid = e.num_sms * 3;
    for (int r = 0; r < kSearchRounds; ++r)
      launch_kernel(e, k_group_search, grid, kSearchThreads, (size_t)(K + 1) * 8,
                    segs, op, r);
    launch_kernel(e, k_group_finish, 1, kGreedyThreads, greedy_smem_bytes(K, k), segs, ssk, ssi, op,
                  (uint64_t)grid);
  }
}

}  // namespace

void launch_plain_groups(const LaunchEnv& e, const uint64_t* offsets, uint32_t k,
                         uint64_t* fine_out, uint32_t* first_out) {
  Scope sc(e, "L1.group");
  launch_kernel(e, k_plain_groups, (k + 256) / 256, 256, 0, offsets, k, fine_out, first_out);
}

void launch_init_plain(const LaunchEnv& e, DevState* st, FinalItem* items, uint64_t n,
                       uint64_t final_cap) {
  Scope sc(e, "init");
  launch_kernel(e, k_init_plain, 1, 32, 0, st, items, n, final_cap, e.local);
}

template <int NT, int IT, int MINB>
void set_sample_sort_attributes() {
  cudaFuncSetAttribute(k_sample_sort<NT, IT, MINB>, cudaFuncAttributeMaxDynamicSharedMemorySize,
                       (int)BinSort<NT, IT>::kSmem);
}

void set_partition_kernel_attributes() {
  set_sample_sort_attributes<128, 8, 8>();
  set_sample_sort_attributes<512, 8, 2>();
  set_sample_sort_attributes<512, 8, 1>();
  set_sample_sort_attributes<512, 16, 1>();
  set_sample_sort_attributes<1024, 8, 1>();
  cudaFuncSetAttribute(k_sample_merge, cudaFuncAttributeMaxDynamicSharedMemorySize,
                       (int)BinSort<kMergeThreads, kMergeItems>::kSmem);
  const size_t c = umax64(classify_smem_bytes(kMaxK, 0, kCStages),
                          classify_smem_bytes(kMaxK, 1, kCStages));
  cudaFuncSetAttribute(k_classify_count<kCStages>, cudaFuncAttributeMaxDynamicSharedMemorySize,
                       (int)c);
  cudaFuncSetAttribute(k_classify_count<kCStagesDeep>,
                       cudaFuncAttributeMaxDynamicSharedMemorySize,
                       (int)umax64(classify_smem_bytes(kMaxKDeep, 0, kCStagesDeep),
                                   classify_smem_bytes(kMaxKDeep, 1, kCStagesDeep)));
  cudaFuncSetAttribute(k_scatter<kPartThreads, 2048, true>,
                       cudaFuncAttributeMaxDynamicSharedMemorySize,
                       (int)umax64(scatter_smem_bytes(kMaxK, 0, kPartWarps, 2048),
                                   scatter_smem_bytes(kMaxK, 1, kPartWarps, 2048)));
  cudaFuncSetAttribute(k_scatter<kPartThreads, 2048, false>,
                       cudaFuncAttributeMaxDynamicSharedMemorySize,
                       (int)umax64(scatter_smem_bytes(kMaxK, 0, kPartWarps, 2048, false),
                                   scatter_smem_bytes(kMaxK, 1, kPartWarps, 2048, false)));
  {
    int dev = 0, optin = 0;
    cudaGetDevice(&dev);
    cudaDeviceGetAttribute(&optin, cudaDevAttrMaxSharedMemoryPerBlockOptin, dev);
    cudaFuncAttributes fa{};
    size_t limit = 0;
    if (cudaFuncGetAttributes(&fa, k_scatter<512, 4096, true>) == cudaSuccess &&
        (size_t)optin > fa.sharedSizeBytes) {
      limit = (size_t)optin - fa.sharedSizeBytes;
      if (cudaFuncSetAttribute(k_scatter<512, 4096, true>,
                               cudaFuncAttributeMaxDynamicSharedMemorySize,
                               (int)limit) != cudaSuccess ||
          cudaFuncSetAttribute(k_scatter<512, 4096, false>,
                               cudaFuncAttributeMaxDynamicSharedMemorySize,
                               (int)limit) != cudaSuccess)
        limit = 0;
    }
    g_wide_scatter_smem_max = limit;
  }
  cudaFuncSetAttribute(k_fine_count, cudaFuncAttributeMaxDynamicSharedMemorySize,
                       (int)fine_smem_bytes(kMaxFine));
  cudaFuncSetAttribute(k_group_search, cudaFuncAttributeMaxDynamicSharedMemorySize,
                       (kMaxFine + 1) * 8);
  cudaFuncSetAttribute(k_group_finish, cudaFuncAttributeMaxDynamicSharedMemorySize,
                       (int)greedy_smem_bytes(kMaxFine, kMaxK));
  cudaGetLastError();  // a refused attribute only disables the variant
}

// Resident CTAs per SM of the classify and of the 2048-key scatter for a bucket
// bound.
int classify_blocks_per_sm(uint32_t kmax, int mode) {
  int nb = 0;
  cudaOccupancyMaxActiveBlocksPerMultiprocessor(&nb, k_classify_count<kCStages>, kPartThreads,
                                                classify_smem_bytes(kmax, mode, kCStages));
  return nb > 0 ? nb : 1;
}

int scatter_blocks_per_sm(uint32_t kmax, int mode, bool stable) {
  int nb = 0;
  const size_t smem = scatter_smem_bytes(kmax, mode, kPartWarps, 2048, stable);
  if (stable)
    cudaOccupancyMaxActiveBlocksPerMultiprocessor(&nb, k_scatter<kPartThreads, 2048, true>,
                                                  kPartThreads, smem);
  else
    cudaOccupancyMaxActiveBlocksPerMultiprocessor(&nb, k_scatter<kPartThreads, 2048, false>,
                                                  kPartThreads, smem);
  return nb > 0 ? nb : 1;
}

int classify_deep_blocks_per_sm(uint32_t kmax, int mode) {
  int nb = 0;
  cudaOccupancyMaxActiveBlocksPerMultiprocessor(&nb, k_classify_count<kCStagesDeep>, kPartThreads,
                                                classify_smem_bytes(kmax, mode, kCStagesDeep));
  return nb > 0 ? nb : 1;
}

int wide_scatter_blocks_per_sm(uint32_t kmax, int mode, bool stable) {
  int nb = 0;
  if (stable)
    cudaOccupancyMaxActiveBlocksPerMultiprocessor(&nb, k_scatter<512, 4096, true>, 512,
                                                  scatter_smem_bytes(kmax, mode, 16, 4096));
  else
    cudaOccupancyMaxActiveBlocksPerMultiprocessor(&nb, k_scatter<512, 4096, false>, 512,
                                                  scatter_smem_bytes(kmax, mode, 16, 4096, false));
  return nb > 0 ? nb : 1;
}

// Segmented input: every segment [offsets[s], offsets[s+1]) is checked and
// routed by size: empty ones are skipped, those that fit one CTA go straight
// to the in-SM sort (original positions relative to the segment start), the
// rest become level-1 segments of the sample sort.  Bad offsets raise a
// device error flag instead of being followed; where they decrease, segments may
// overlap, and the plan leaves the level-1 segments out (the others are read from
// the input and written in their own range).
__global__ void __launch_bounds__(256)
k_init_segments(DevState* st, const uint64_t* offsets, uint32_t nseg, uint64_t n,
                SegIn* list_l1, FinalItem* items, uint64_t seg_cap, uint64_t final_cap,
                int f64) {
  pdl_entry();
  for (uint64_t s = (uint64_t)blockIdx.x * blockDim.x + threadIdx.x; s < nseg;
       s += (uint64_t)gridDim.x * blockDim.x) {
    const uint64_t a = offsets[s], b = offsets[s + 1];
    if (b < a || b > n || (b - a) > 0xFFFFFFFFull) {
      atomicOr(&st->error, kErrBadOffsets | (b < a ? kErrUnordered : 0u));
      continue;
    }
    const uint64_t m = b - a;
    if (m == 0) continue;
    if (m <= (uint64_t)kBucketCap) {
      FinalItem f;
      f.start = a;
      f.aux = a;
      f.size = (uint32_t)m;
      f.where = kWhereInput;
      f.kind = m == 1 ? kKindCopy : kKindSort;
      f.bits = kBitsUnknown;
      push_final(st, items, final_cap, f, kErrFinalCap, f64 != 0 && m > st->local.rank_max);
    } else {
      SegIn in;
      in.start = a;
      in.m = (uint32_t)m;
      in.known = 0;
      in.range = KeyRange{0, ~0ULL};
      const uint32_t slot = atomicAdd(&st->nseg[1], 1u);
      if (slot < seg_cap) list_l1[slot] = in;
      else atomicOr(&st->error, kErrSegCap);
    }
  }
}

void launch_init_segments(const LaunchEnv& e, DevState* st, const uint64_t* offsets,
                          uint32_t nseg, uint64_t n, SegIn* list_l1, FinalItem* items,
                          uint64_t seg_cap, uint64_t final_cap, int f64) {
  Scope sc(e, "init_segments");
  const int grid = (int)umin64((nseg + 255) / 256 + 1, (uint64_t)e.num_sms * 8);
  launch_kernel(e, k_init_segments, grid, 256, 0, st, offsets, nseg, n, list_l1, items, seg_cap,
                final_cap, f64);
}

namespace {

// Samples of a deeper level's segments: the expected segment decides the shape
// of the CTAs that draw and sort them (LevelParams::samp_max bounds the rest).
template <int NT, int IT, int MINB>
void launch_sample_sort(const LaunchEnv& e, const char* name, uint64_t chunks, DevState* st,
                        LevelSeg* segs, const Src& src, uint64_t* samp_key, uint32_t* samp_idx,
                        uint64_t* ssamp_key, uint32_t* ssamp_idx, uint32_t min_len,
                        const PlainStart& ps, const LevelParams& P) {
  Scope sc(e, name);
  launch_kernel(e, k_sample_sort<NT, IT, MINB>, grid_for(chunks, 1, e.num_sms * MINB), NT,
                BinSort<NT, IT>::kSmem, st, segs, src, samp_key, samp_idx, ssamp_key, ssamp_idx,
                P.in_order, min_len, ps, P);
}

}  // namespace

// k_plain: buckets of a call's only segment, [0, n_total) of the input (level 1
// of a sort or partition, started by this launch); 0: the segments of list_in.
void launch_level(const LaunchEnv& e, const LevelParams& P, DevState* st, const SegIn* list_in,
                  SegIn* list_out, LevelSeg* segs, Src src, Dst dst, uint16_t dst_where,
                  uint64_t* samp_key, uint32_t* samp_idx, uint64_t* ssamp_key,
                  uint32_t* ssamp_idx, uint32_t* hist, uint32_t* block_sums, FinalItem* items,
                  int kmax_level, int last_level, int emit_final, uint64_t* offsets_out,
                  uint64_t n_total, int unmap_out, const Overpart* op, uint32_t k_plain,
                  uint64_t* plan_sums) {
  const int par_in = P.level & 1;
  const int sms = e.num_sms;
  static const char* kNames[kMaxLevels + 1][8] = {
      {"L?.plan", "L?.sample_sort", "L?.sample_merge", "L?.classify", "L?.scan_reduce",
       "L?.scan_down", "L?.scatter", "L?.collect"},
      {"L1.plan", "L1.sample_sort", "L1.sample_merge", "L1.classify", "L1.scan_reduce",
       "L1.scan_down", "L1.scatter", "L1.collect"},
      {"L2.plan", "L2.sample_sort", "L2.sample_merge", "L2.classify", "L2.scan_reduce",
       "L2.scan_down", "L2.scatter", "L2.collect"},
      {"L3.plan", "L3.sample_sort", "L3.sample_merge", "L3.classify", "L3.scan_reduce",
       "L3.scan_down", "L3.scatter", "L3.collect"}};
  const char* const* nm = kNames[(P.level >= 1 && P.level <= kMaxLevels) ? P.level : 0];
  LevelParams PS = P;  // of the sample
  PlainStart ps;
  uint64_t plain_hist = 0;  // counters of a one-segment level
  if (k_plain) {
    ps.n = n_total;
    ps.k = k_plain;
    ps.nch = (uint32_t)((n_total + P.W - 1) / P.W);
    uint32_t lg = 0;
    while ((1ull << lg) < k_plain) ++lg;
    const uint64_t a = P.hinted ? 16ull * lg : (uint64_t)P.oversample;
    ps.S = (uint32_t)umin64(umin64(n_total, a * k_plain), P.samp_max);
    ps.local = e.local;
    plain_hist = (uint64_t)k_plain * ps.nch;
    // Chunks sorted side by side and a merge take less than one CTA's sort of
    // them all: 8192 float64 samples 41 -> 15 + 15 us, 6144 23 -> 11 + 11 (the
    // merge's launch overlaps); at 4608 samples the two are even and below one
    // CTA wins (partition of 2^20 keys, 2560 samples: 44.7 us, two chunks 49.7).
    // 163,840 samples in chunks of 2048 instead of 4096: 23 + 17 -> 17 + 18 us, an
    // overpartitioned step of 2^24 keys 349 -> 340.
    if (ps.S > kMaxSampleChunks * 2048u) PS.sample_chunk = 4096;
    else if (ps.S > (uint32_t)kSampleChunk) PS.sample_chunk = 2048;
    else if (ps.S > kMinSplitSample) PS.sample_chunk = 1024;
    const uint64_t nsch = (ps.S + PS.sample_chunk - 1) / PS.sample_chunk;
    auto draw = [&](auto nt, auto it) {
      launch_sample_sort<decltype(nt)::value, decltype(it)::value, 1>(
          e, nm[1], umax64(nsch, 1), st, segs, src, samp_key, samp_idx, ssamp_key, ssamp_idx, 0,
          ps, PS);
    };
    // one CTA a chunk: the more threads the shorter
    if (ps.S <= 4096 || nsch > 1)
      draw(std::integral_constant<int, 512>(), std::integral_constant<int, 8>());
    else
      draw(std::integral_constant<int, 1024>(), std::integral_constant<int, 8>());
    if (nsch > 1) {
      Scope sc(e, nm[2]);
      const size_t smem = BinSort<kMergeThreads, kMergeItems>::kSmem;
      launch_kernel(e, k_sample_merge, (int)((ps.S + kMergeRange - 1) / kMergeRange), kMergeThreads,
                    smem, segs, samp_key, samp_idx, ssamp_key, ssamp_idx);
    }
  } else {
    {
      Scope sc(e, nm[0]);
      const int ctas = grid_for(umin64(P.seg_cap, P.max_segs), kPlanThreads, 1 << 22);
      if (ctas > 1) {
        launch_kernel(e, k_plan_sums, ctas, kPlanThreads, 0, st, list_in, P, par_in,
                      (uint32_t)kmax_level, plan_sums);
        if (e.launches) ++*e.launches;
      }
      launch_kernel(e, k_level_plan, ctas, kPlanThreads, 0, st, list_in, segs, P, par_in,
                    (uint32_t)kmax_level, plan_sums, src.chunk_seg);
    }
    // (every segment has at most kMaxKDeep buckets, so one sample chunk)
    static_assert(kMaxKDeep * kDeepOversample <= kSampleChunk, "one sample chunk a segment");
    if (P.samp_max <= 1024) {
      launch_sample_sort<128, 8, 8>(e, nm[1], P.schunk_cap, st, segs, src, samp_key, samp_idx,
                                    ssamp_key, ssamp_idx, 0, ps, P);
    } else if (P.samp_max <= 4096) {
      // (twice the threads of 256 x 16 on the same shared memory: 1024 samples of
      // about 2700 pairs 157 -> 145 us)
      launch_sample_sort<512, 8, 2>(e, nm[1], P.schunk_cap, st, segs, src, samp_key, samp_idx,
                                    ssamp_key, ssamp_idx, 0, ps, P);
    } else {
      // segments of any size: small samples by small CTAs, the others by large
      launch_sample_sort<128, 8, 8>(e, nm[1], P.schunk_cap, st, segs, src, samp_key, samp_idx,
                                    ssamp_key, ssamp_idx, 0, ps, P);
      launch_sample_sort<512, 16, 1>(e, nm[1], P.schunk_cap, st, segs, src, samp_key, samp_idx,
                                     ssamp_key, ssamp_idx, 1024, ps, P);
    }
  }
  const int mode = P.classifier | (P.no_tie_break ? 2 : 0);
  const size_t smem_c = classify_smem_bytes((uint32_t)kmax_level, mode, kCStages);
  // deeper levels take the 2-stage classify when their buckets fit its shared memory
  const bool deep_c = P.level > 1 && (uint32_t)kmax_level <= (uint32_t)kMaxKDeep;
  const size_t smem_cd = classify_smem_bytes((uint32_t)kmax_level, mode, kCStagesDeep);
  const int grid_c = grid_for(
      P.chunk_cap, 1,
      sms * (deep_c ? classify_deep_blocks_per_sm((uint32_t)kmax_level, mode)
                    : classify_blocks_per_sm((uint32_t)kmax_level, mode)));
  const bool stable = P.stable == 1;
  const int grid_s = grid_for(P.chunk_cap, 1,
                              sms * scatter_blocks_per_sm((uint32_t)kmax_level, mode, stable));
  const bool wide = kmax_level >= P.wide_scatter_k &&
                    scatter_smem_bytes((uint32_t)kmax_level, mode, 16, 4096, stable) <=
                        g_wide_scatter_smem_max;
  // A level with at most kUnitMaxK buckets classifies once, storing every
  // element's bucket id, and scatters whole 8-element units (unit_scatter.cu).
  // Otherwise stored bucket ids spare the staged scatter its second
  // classification, except at 1024+ buckets, where its L2-resident write
  // frontiers were the bottleneck and the extra id stream measured slower.
  // With atomic_scatter, an unordered level (a full sort's levels after the
  // first) keeps the ids of its classify pass and ranks by shared-memory
  // atomics in the small-footprint scatter (measured slower than the staged
  // scatter at 2^28 keys with ~171 buckets per segment; a tuner candidate).
  // (a level that need not keep input order -- a full sort's levels -- has
  // the unit scatter rank by shared-memory atomics)
  const bool units = P.unit_scatter && src.bid != nullptr &&
                     kmax_level > 32 && unit_scatter_fits((uint32_t)kmax_level);
  const bool atomics = !units && P.atomic_scatter && !stable &&
                       src.bid != nullptr && atomic_scatter_fits((uint32_t)kmax_level);
  if (!units && !atomics && kmax_level >= 1024) src.bid = nullptr;
  // the ids of an overpartitioned step's fine partitions are stored instead, and
  // mapped to buckets after the greedy has grouped them
  const bool fine_ids = op && units && stable && !P.bulk_classify &&
                        n_total >= kFineIdsMin * op->k * op->over &&
                        fine_ids_fit(op->k * op->over);
  // A level of one segment and long chunks has the classify look for runs of
  // equal splitters and place ties by bands: both cost a pass over the splitters
  // a chunk (below kBandMinW keys a chunk, and per segment, it showed: 10^5 keys
  // 38.8 -> 39.5 us, 100,000 segments 6.92 -> 6.99 ms).
  const bool bands = k_plain > 0 && src.idx == nullptr && P.W >= kBandMinW;
  if (op) launch_overpartition(e, P, st, segs, src, ssamp_key, ssamp_idx, *op, fine_ids);
  if (fine_ids) {
    launch_map_ids(e, P, st, segs, src, *op, hist, nm[3]);
  } else if (units) {
    launch_classify_ids(e, P, st, segs, src, ssamp_key, ssamp_idx, hist, (uint32_t)kmax_level,
                        mode, bands, nm[3]);
  } else {
    Scope sc(e, nm[3]);
    if (deep_c)
      launch_kernel(e, k_classify_count<kCStagesDeep>, grid_c, kPartThreads, smem_cd, st, segs, src,
                    ssamp_key, ssamp_idx, hist, P.W, (uint32_t)kmax_level, mode);
    else
      launch_kernel(e, k_classify_count<kCStages>, grid_c, kPartThreads, smem_c, st, segs, src,
                    ssamp_key, ssamp_idx, hist, P.W, (uint32_t)kmax_level, mode);
  }
  const bool small_scan = k_plain && plain_hist <= kSmallScan;
  if (small_scan) {
    Scope sc(e, nm[5]);
    launch_kernel(e, k_scan_collect, 1, 1024, 0, st, segs, ssamp_key, hist, list_out, par_in ^ 1,
                  items, P, dst_where, last_level, emit_final, offsets_out);
  } else {
    const uint64_t most = k_plain ? plain_hist : P.hist_cap;
    const int scan_grid = (int)umax64((most + kScanTile - 1) / kScanTile, 1);
    {
      Scope sc(e, nm[4]);
      launch_kernel(e, k_scan_reduce, scan_grid, 1024, 0, st, hist, block_sums);
    }
    {
      Scope sc(e, nm[5]);
      launch_kernel(e, k_scan_down, scan_grid, 1024, 0, st, hist, block_sums);
    }
  }
  if (units) {
    launch_scatter_units(e, P, st, segs, src, hist, dst, (uint32_t)kmax_level, unmap_out, nm[6]);
  } else if (atomics) {
    launch_scatter_atomic(e, P, st, segs, src, hist, dst, (uint32_t)kmax_level, unmap_out, nm[6]);
  } else {
    Scope sc(e, nm[6]);
    if (wide && stable)
      launch_kernel(e, k_scatter<512, 4096, true>,
                    grid_for(P.chunk_cap, 1, sms * wide_scatter_blocks_per_sm((uint32_t)kmax_level, mode, true)),
                    512, scatter_smem_bytes((uint32_t)kmax_level, mode, 16, 4096), st, segs, src,
                    ssamp_key, ssamp_idx, hist, dst, P.W, (uint32_t)kmax_level, unmap_out, mode);
    else if (wide)
      launch_kernel(e, k_scatter<512, 4096, false>,
                    grid_for(P.chunk_cap, 1, sms * wide_scatter_blocks_per_sm((uint32_t)kmax_level, mode, false)),
                    512, scatter_smem_bytes((uint32_t)kmax_level, mode, 16, 4096, false), st, segs,
                    src, ssamp_key, ssamp_idx, hist, dst, P.W, (uint32_t)kmax_level, unmap_out,
                    mode);
    else if (stable)
      launch_kernel(e, k_scatter<kPartThreads, 2048, true>, grid_s, kPartThreads,
                    scatter_smem_bytes((uint32_t)kmax_level, mode, kPartWarps, 2048), st, segs, src,
                    ssamp_key, ssamp_idx, hist, dst, P.W, (uint32_t)kmax_level, unmap_out, mode);
    else
      launch_kernel(e, k_scatter<kPartThreads, 2048, false>, grid_s, kPartThreads,
                    scatter_smem_bytes((uint32_t)kmax_level, mode, kPartWarps, 2048, false), st,
                    segs, src, ssamp_key, ssamp_idx, hist, dst, P.W, (uint32_t)kmax_level,
                    unmap_out, mode);
  }
  if (!small_scan) {
    Scope sc(e, nm[7]);
    launch_kernel(e, k_collect, grid_for(P.bucket_cap, 256, sms * 8), 256, 0, st, segs, ssamp_key,
                  hist, list_out, par_in ^ 1, items, P, dst_where, last_level, emit_final,
                  offsets_out);
  }
}

}  // namespace rsort
