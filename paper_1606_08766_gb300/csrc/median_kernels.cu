// median_kernels.cu -- the binary-tree median approximation of Section 3
// ("Approximate Median Selection with a Single Reduction") over a whole key
// array, by the whole GPU.
//
// Every CTA reduces a subtree of kTmLeaves leaves in shared memory
// (k_tm_leaves) and leaves the window of its root in scratch; further launches
// reduce groups of windows (k_tm_windows) until one CTA holds the tree's root.
//
// The lowest levels cut nothing: a node over at most K/2 leaves has at most K/2
// entries below every element (K/2 minus the coins that came up 1) and at most
// K/2 elements, so its window is its sorted leaves.  One thread sorts K/2
// leaves in registers and replaces log2(K/2) levels.  Above, a thread makes
// four consecutive entries of a node's window: a merge-path search finds where
// they start in the two children, four merge steps follow.
//   Bound by instructions in the first launch and by the latency of the levels
//   in the others.  2^20 keys, k = 16: one CTA reducing the tree through
//   global memory, a thread per node, took 7.94 ms; element-wise ranking of
//   every level in two launches 53 us; this form 32 us.
#include "rsort_internal.cuh"
#include "tree_median.cuh"

namespace rsort {

namespace {

constexpr int kTmThreads = 512;
constexpr uint32_t kTmLeaves = 2048;  // leaves of a CTA of the first launch
// window entries of a CTA of the others (one CTA per SM: the fewer launches,
// the better)
template <int K>
constexpr uint32_t kTmEntries = K >= 16 ? 8192 : 4096;

// Slots between two windows of cap entries: one more from 8 on, so that the
// windows a warp works on start in different banks.
__host__ __device__ __forceinline__ constexpr uint32_t tm_stride(uint32_t cap) {
  return cap >= 8 ? cap + 1 : cap;
}

// Two levels of windows in shared memory, ENT entries each in at most NODES
// windows: node j of a level holds nre[j] elements from slot j * tm_stride(cap)
// on, and neg[j] entries below every element.  A level is named by its side (0
// or 1), so that every access is a shared-memory one at a computed slot.
template <uint32_t ENT, uint32_t NODES>
struct TmSmem {
  static constexpr uint32_t kSlots = ENT + ENT / 8;
  static constexpr size_t kBytes = (size_t)2 * kSlots * 12 + (size_t)4 * NODES;
  uint64_t* key;  // [2][kSlots]
  uint32_t* pos;  // [2][kSlots]
  uint8_t* neg;   // [2][NODES]
  uint8_t* nre;   // [2][NODES]
  __device__ __forceinline__ explicit TmSmem(unsigned char* p) {
    key = (uint64_t*)p;
    pos = (uint32_t*)(key + 2 * kSlots);
    neg = (uint8_t*)(pos + 2 * kSlots);
    nre = neg + 2 * NODES;
  }
};

// Windows of one level in scratch, K slots each.
struct TmWindows {
  uint64_t* key;
  uint32_t* pos;
  uint8_t* neg;
  uint8_t* nre;
};

// Combines the windows of side `sd` pairwise into side sd ^ 1: `half` nodes of
// ncap slots from children of cap slots, E consecutive entries a thread.  The
// search and the merge steps run without branches: a level is bound by their
// latency, and lanes of a warp would take both sides of each.
template <int K, int E, typename S>
__device__ __forceinline__ void tm_level(const S& m, uint32_t sd, uint32_t half, uint32_t cap,
                                         uint32_t ncap, uint32_t nodes_cap) {
  constexpr int s = K / 2;  // first merged position a node keeps
  const uint32_t sa = tm_stride(cap), sb = tm_stride(ncap);
  const int lper = __ffs((int)(ncap / E)) - 1;  // log2 of the threads per node
  const uint64_t* ik = m.key + sd * S::kSlots;
  const uint32_t* ip = m.pos + sd * S::kSlots;
  const uint8_t* in = m.neg + sd * nodes_cap;
  const uint8_t* ir = m.nre + sd * nodes_cap;
  for (uint32_t x = threadIdx.x; x < half << lper; x += kTmThreads) {
    const uint32_t j = x >> lper, q = x & ((1u << lper) - 1);
    const uint32_t ca = 2 * j, cb = ca + 1;        // its children
    const int N = in[ca] + in[cb];                 // merged entries below every element
    const int nA = ir[ca], nB = ir[cb];
    const int R = nA + nB;                         // merged elements
    const int lo = s - N > 0 ? s - N : 0;          // first merged element kept
    const int hi = s + K - N < R ? s + K - N : R;  // one past the last
    if (q == 0) {
      const int nneg = N - s;
      m.neg[(sd ^ 1) * nodes_cap + j] = (uint8_t)(nneg < 0 ? 0 : (nneg > K ? K : nneg));
      m.nre[(sd ^ 1) * nodes_cap + j] = (uint8_t)(hi > lo ? hi - lo : 0);
    }
    const int t0 = lo + (int)q * E;
    if (t0 < hi) {
      const uint32_t A = ca * sa, B = cb * sa;
      // elements of A among the first t0 merged ones
      int l = t0 > nB ? t0 - nB : 0, h = t0 < nA ? t0 : nA;
#pragma unroll
      for (int w = K; w > 0; w >>= 1) {
        const bool act = l < h;
        const int mid = (l + h) >> 1;
        const uint32_t pa = A + (act ? mid : 0), pb = B + (act ? t0 - 1 - mid : 0);
        const bool less = pair_less(ik[pa], ip[pa], ik[pb], ip[pb]);
        l = act && less ? mid + 1 : l;
        h = act && !less ? mid : h;
      }
      int ia = l, ib = t0 - l;
      uint64_t ka = ik[A + (ia < nA ? ia : 0)], kb = ik[B + (ib < nB ? ib : 0)];
      uint32_t qa = ip[A + (ia < nA ? ia : 0)], qb = ip[B + (ib < nB ? ib : 0)];
      const uint32_t o = (sd ^ 1) * S::kSlots + j * sb + q * E;
#pragma unroll
      for (int e = 0; e < E; ++e) {
        const bool ta = ib >= nB || (ia < nA && pair_less(ka, qa, kb, qb));
        if (t0 + e < hi) {
          m.key[o + e] = ta ? ka : kb;
          m.pos[o + e] = ta ? qa : qb;
        }
        if (e + 1 < E) {
          ia += ta ? 1 : 0;
          ib += ta ? 0 : 1;
          const uint32_t nx = ta ? A + (ia < nA ? ia : 0) : B + (ib < nB ? ib : 0);
          const uint64_t kn = ik[nx];
          const uint32_t pn = ip[nx];
          ka = ta ? kn : ka;
          qa = ta ? pn : qa;
          kb = ta ? kb : kn;
          qb = ta ? qb : pn;
        }
      }
    }
  }
}

// Reduces `nodes` windows of `cap` slots (powers of two, cap >= K/2) on side 0
// to one; returns the side that holds it.  The caller has synchronised the CTA
// after filling side 0.
template <int K, typename S>
__device__ __forceinline__ uint32_t tm_reduce(const S& m, uint32_t nodes, uint32_t cap,
                                              uint32_t nodes_cap) {
  constexpr int E = K < 4 ? K : 4;
  uint32_t sd = 0;
  while (nodes > 1) {
    const uint32_t half = nodes / 2;
    const uint32_t ncap = 2 * cap < (uint32_t)K ? 2 * cap : (uint32_t)K;
    // four entries a thread while that fills the CTA, else one
    if (half * ncap > (uint32_t)kTmThreads) tm_level<K, E>(m, sd, half, cap, ncap, nodes_cap);
    else tm_level<K, 1>(m, sd, half, cap, ncap, nodes_cap);
    __syncthreads();
    sd ^= 1;
    nodes = half;
    cap = ncap;
  }
  return sd;
}

// Sorts H (key, position) pairs of one thread (bitonic network).
template <int H>
__device__ __forceinline__ void tm_sort_regs(uint64_t (&k)[H], uint32_t (&p)[H]) {
#pragma unroll
  for (int size = 2; size <= H; size <<= 1) {
#pragma unroll
    for (int st = size >> 1; st > 0; st >>= 1) {
#pragma unroll
      for (int r = 0; r < H; ++r) {
        if ((r & st) == 0 && pair_less(k[r + st], p[r + st], k[r], p[r]) == ((r & size) == 0)) {
          const uint64_t tk = k[r];
          const uint32_t tp = p[r];
          k[r] = k[r + st];
          p[r] = p[r + st];
          k[r + st] = tk;
          p[r + st] = tp;
        }
      }
    }
  }
}

// The root's window on side sd: the chosen element if this CTA holds the whole
// tree, else one window of the next launch.
template <int K, typename S>
__device__ __forceinline__ void tm_finish(const S& m, uint32_t sd, uint32_t nodes_cap,
                                          uint64_t seed, uint64_t leaves, const TmWindows& out,
                                          uint64_t* out_pos) {
  const uint32_t neg = m.neg[sd * nodes_cap], nre = m.nre[sd * nodes_cap];
  const uint64_t* k = m.key + sd * S::kSlots;
  const uint32_t* p = m.pos + sd * S::kSlots;
  if (gridDim.x == 1) {
    if (threadIdx.x == 0) {
      const int pick = tm_root_pick<K>((int)neg, (int)nre, seed, leaves);
      *out_pos = pick >= 0 ? p[pick] : 0u;
    }
    return;
  }
  const uint64_t g = blockIdx.x;
  if (threadIdx.x < nre) {
    out.key[g * K + threadIdx.x] = k[threadIdx.x];
    out.pos[g * K + threadIdx.x] = p[threadIdx.x];
  }
  if (threadIdx.x == 0) {
    out.neg[g] = (uint8_t)neg;
    out.nre[g] = (uint8_t)nre;
  }
}

template <int K>
using TmLeafSmem = TmSmem<kTmLeaves, kTmLeaves / (K / 2)>;
template <int K>
using TmWindowSmem = TmSmem<kTmEntries<K>, kTmEntries<K> / K>;

template <int K>
__global__ void __launch_bounds__(kTmThreads)
k_tm_leaves(const uint64_t* keys, uint32_t n, int f64, uint64_t seed, uint32_t leaves,
            TmWindows out, uint64_t* out_pos, uint32_t* error) {
  pdl_entry();
  extern __shared__ __align__(16) unsigned char smem_raw[];
  const TmLeafSmem<K> m(smem_raw);
  constexpr int H = K / 2;  // leaves a thread sorts
  constexpr uint32_t kNodes = kTmLeaves / H;
  if (blockIdx.x == 0 && threadIdx.x == 0) *error = 0;  // of the control block
  const uint32_t cnt = leaves < kTmLeaves ? leaves : kTmLeaves;
  const uint32_t groups = cnt > (uint32_t)H ? cnt / H : 1;
  for (uint32_t g = threadIdx.x; g < groups; g += kTmThreads) {
    const uint32_t i0 = blockIdx.x * kTmLeaves + g * H;
    uint64_t k[H];
    uint32_t p[H];
    int ones = 0, present = 0;
#pragma unroll
    for (int r = 0; r < H; ++r) {
      const uint32_t i = i0 + r;
      k[r] = ~0ULL;  // a leaf without an element sorts last
      p[r] = ~0u;
      if (i < n) {
        const uint64_t raw = keys[i];
        k[r] = f64 ? f64_to_ordered(raw) : raw;
        p[r] = i;
        ones += K / 2 - tm_leaf_neg<K>(true, seed, i);
        ++present;
      }
    }
    tm_sort_regs<H>(k, p);
#pragma unroll
    for (int r = 0; r < H; ++r) {
      m.key[g * tm_stride(H) + r] = k[r];
      m.pos[g * tm_stride(H) + r] = p[r];
    }
    m.neg[g] = (uint8_t)(K / 2 - ones);
    m.nre[g] = (uint8_t)present;
  }
  __syncthreads();
  const uint32_t sd = tm_reduce<K>(m, groups, H, kNodes);
  tm_finish<K>(m, sd, kNodes, seed, leaves, out, out_pos);
}

template <int K>
__global__ void __launch_bounds__(kTmThreads)
k_tm_windows(TmWindows in, uint32_t count, uint64_t seed, uint64_t leaves, TmWindows out,
             uint64_t* out_pos) {
  pdl_entry();
  extern __shared__ __align__(16) unsigned char smem_raw[];
  const TmWindowSmem<K> m(smem_raw);
  constexpr uint32_t kGroup = kTmEntries<K> / K;
  const uint32_t cnt = count < kGroup ? count : kGroup;
  const uint64_t first = (uint64_t)blockIdx.x * cnt;
  // (slots beyond a window's elements are copied unread)
#pragma unroll 4
  for (uint32_t t = threadIdx.x; t < cnt * K; t += kTmThreads) {
    const uint32_t at = (t / K) * tm_stride(K) + t % K;
    m.key[at] = in.key[first * K + t];
    m.pos[at] = in.pos[first * K + t];
  }
  for (uint32_t t = threadIdx.x; t < cnt; t += kTmThreads) {
    m.neg[t] = in.neg[first + t];
    m.nre[t] = in.nre[first + t];
  }
  __syncthreads();
  const uint32_t sd = tm_reduce<K>(m, cnt, K, kGroup);
  tm_finish<K>(m, sd, kGroup, seed, leaves, out, out_pos);
}

// Windows of the first launch (a power of two).
inline uint32_t tm_windows(uint32_t leaves) {
  return leaves > kTmLeaves ? leaves / kTmLeaves : 1;
}

template <int K>
void launch_k(const LaunchEnv& e, const uint64_t* keys, uint32_t n, int f64, uint64_t seed,
              uint32_t leaves, void* scratch, uint64_t* out) {
  uint32_t w = tm_windows(leaves);
  TmWindows lv[2];
  // the arena starts with the control block, whose error word is read back
  DevState* st = (DevState*)scratch;
  unsigned char* p = (unsigned char*)(st + 1);
  for (int i = 0; i < 2; ++i) {
    lv[i].key = (uint64_t*)p;
    p += (size_t)w * K * 8;
    lv[i].pos = (uint32_t*)p;
    p += (size_t)w * K * 4;
    lv[i].neg = (uint8_t*)p;
    p += w;
    lv[i].nre = (uint8_t*)p;
    p += w;
    p = (unsigned char*)(((uintptr_t)p + 15) & ~(uintptr_t)15);
  }
  launch_kernel(e, k_tm_leaves<K>, w, kTmThreads, TmLeafSmem<K>::kBytes, keys, n, f64, seed, leaves,
                lv[0], out, &st->error);
  for (int i = 0; w > 1; i ^= 1) {
    constexpr uint32_t kGroup = kTmEntries<K> / K;
    const uint32_t groups = w > kGroup ? w / kGroup : 1;
    launch_kernel(e, k_tm_windows<K>, groups, kTmThreads, TmWindowSmem<K>::kBytes, lv[i], w, seed,
                  leaves, lv[i ^ 1], out);
    if (e.launches) ++*e.launches;
    w = groups;
  }
}

template <int K>
void set_k_attributes() {
  cudaFuncSetAttribute(k_tm_leaves<K>, cudaFuncAttributeMaxDynamicSharedMemorySize,
                       (int)TmLeafSmem<K>::kBytes);
  cudaFuncSetAttribute(k_tm_windows<K>, cudaFuncAttributeMaxDynamicSharedMemorySize,
                       (int)TmWindowSmem<K>::kBytes);
}

}  // namespace

size_t tree_median_scratch_bytes(uint64_t n) {
  const uint32_t leaves = next_pow2_u32((uint32_t)(n > 0 ? n : 1));
  return sizeof(DevState) + 2 * ((size_t)tm_windows(leaves) * (32 * 12 + 2) + 16);
}

void set_median_kernel_attributes() {
  set_k_attributes<2>();
  set_k_attributes<4>();
  set_k_attributes<8>();
  set_k_attributes<16>();
  set_k_attributes<32>();
}

bool launch_tree_median(const LaunchEnv& e, const uint64_t* keys, uint32_t n, int f64,
                        uint32_t k, uint64_t seed, void* scratch, uint64_t* out_pos) {
  const uint32_t leaves = next_pow2_u32(n);
  struct Scope {
    const LaunchEnv& e;
    Scope(const LaunchEnv& env) : e(env) {
      if (e.timer) e.timer->begin("tree_median", e.stream);
    }
    ~Scope() {
      if (e.timer) e.timer->end(e.stream);
      if (e.launches) ++*e.launches;
    }
  } sc(e);
  switch (k) {
    case 2: launch_k<2>(e, keys, n, f64, seed, leaves, scratch, out_pos); return true;
    case 4: launch_k<4>(e, keys, n, f64, seed, leaves, scratch, out_pos); return true;
    case 8: launch_k<8>(e, keys, n, f64, seed, leaves, scratch, out_pos); return true;
    case 16: launch_k<16>(e, keys, n, f64, seed, leaves, scratch, out_pos); return true;
    case 32: launch_k<32>(e, keys, n, f64, seed, leaves, scratch, out_pos); return true;
    default: return false;
  }
}

}  // namespace rsort
