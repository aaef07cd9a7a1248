// Merge sort (Sec. 2.4, the parallel merge sort of Satish et al.): a
// comparison sort, stable, for keys that the radix passes do not take
// (128-bit keys) as well as 32- and 64-bit keys.
//   k_ms_tile   sorts each tile of kTile (4096) elements in one CTA, in shared
//               memory, by the key's bytes (those that differ in the tile);
//   k_ms_split  for a global merge of runs of width w, finds where each
//               output tile of the merged pair begins in the left run (the
//               merge path), one warp a tile: 32 probes of the tile's diagonal
//               at a time;
//   k_ms_merge  merges one output tile (kOutTile) per CTA from the two input
//               ranges its split delimits.
// The merge kernels are launched as the one before exits (pdl_wait).
// Ties always take the element of the left run, which holds the earlier
// input positions, so every merge (and the whole sort) is stable.  Values do
// not take part: 16-bit source positions are sorted and merged, and the values
// are gathered by them when a tile is written.
#include <algorithm>

#include "../../include/rs.h"
#include "rs_debug.cuh"
#include "rs_host.h"
#include "rs_kernels.cuh"

namespace rs {

namespace {

constexpr int kMsItems = 16;  // outputs a thread of a merge
constexpr int kTile = 4096;   // of the tile sort: the first runs

// Threads of a merge CTA, and its output tile.  Few 128-bit tiles fit an SM at
// once, so that the last wave of an array of a few million is mostly empty:
// tiles half the size lose half as much (4e6 keys with values, a pass: 54 us ->
// 51).
template <class K>
constexpr int kMsThreads = sizeof(K) == 16 ? 128 : 256;
template <class K>
constexpr int kOutTile = kMsThreads<K> * kMsItems;
constexpr int kOutTileLeast = 128 * kMsItems;

// A 128-bit unsigned key: value = lo + 2^64 * hi (little-endian words).
struct alignas(16) Key128 {
  uint64_t lo, hi;
};

__device__ __forceinline__ bool key_less(uint32_t a, uint32_t b) { return a < b; }
__device__ __forceinline__ bool key_less(uint64_t a, uint64_t b) { return a < b; }
__device__ __forceinline__ bool key_less(const Key128& a, const Key128& b) {
  return a.hi < b.hi || (a.hi == b.hi && a.lo < b.lo);
}

struct NoVal {};

// Shared-memory slot of element i: one pad slot after every 32 elements, so
// that a warp reading or writing each thread's kMsItems consecutive elements
// (stride kMsItems) spreads over the banks instead of hitting a few.
__device__ __forceinline__ uint32_t pad(uint32_t i) { return i + (i >> 5); }

// A run of elements in shared memory, indexed through pad().
template <class T>
struct Padded {
  T* base;
  uint32_t first;  // element index of run[0]
  __device__ __forceinline__ T& operator[](uint32_t i) const { return base[pad(first + i)]; }
};

// Elements taken from the left run a[0 .. na) at diagonal `diag` of the merge
// of a and b[0 .. nb): the largest i with a[i-1] <= b[diag-i] (ties: a first).
template <class A, class B>
__device__ __forceinline__ uint32_t merge_path(const A& a, uint32_t na, const B& b, uint32_t nb,
                                               uint32_t diag) {
  uint32_t lo = diag > nb ? diag - nb : 0u;
  uint32_t hi = min(diag, na);
  while (lo < hi) {
    const uint32_t mid = (lo + hi) >> 1;
    if (!key_less(b[diag - 1 - mid], a[mid])) lo = mid + 1;  // a[mid] <= b[...]: take it
    else hi = mid;
  }
  return lo;
}

// The first and one past the last element of a run inside a padded buffer.
struct Run {
  uint32_t at, end;
};

// Merge min(kMsItems, what is left) outputs of runs a and b (element indices
// into sk, a the left one) into registers, and their element indices into sp
// from element o on.  One key is read per output: the other run's head stays
// in a register.
template <bool HAS_V, class K>
__device__ __forceinline__ void merge_items(const K* sk, Run a, Run b, K (&k)[kMsItems],
                                            uint16_t* sp, uint32_t o) {
  K ka{}, kb{};
  if (a.at < a.end) ka = sk[pad(a.at)];
  if (b.at < b.end) kb = sk[pad(b.at)];
#pragma unroll
  for (int t = 0; t < kMsItems; ++t) {
    if (a.at >= a.end && b.at >= b.end) break;  // both used up (the last, partial tile)
    const bool take_a = b.at >= b.end || (a.at < a.end && !key_less(kb, ka));
    k[t] = take_a ? ka : kb;
    const uint32_t src = take_a ? a.at : b.at;
    if constexpr (HAS_V) sp[pad(o + t)] = uint16_t(src);
    const uint32_t next = src + 1u;
    if (take_a) a.at = next;
    else b.at = next;
    if (next < (take_a ? a.end : b.end)) {
      const K x = sk[pad(next)];
      if (take_a) ka = x;
      else kb = x;
    }
  }
}

// Shared memory of a merged tile: keys (with pad slots), 16-bit source
// positions, the values as loaded.
template <class K, class V, bool HAS_V>
struct MsSmem {
  static constexpr int SLOTS = kOutTile<K> + kOutTile<K> / 32;
  static constexpr int KEYS = 0;
  static constexpr int POS = (SLOTS * int(sizeof(K)) + 15) / 16 * 16;
  static constexpr int VALS = POS + (HAS_V ? SLOTS * 2 + 15 : 0) / 16 * 16;
  static constexpr int BYTES = VALS + (HAS_V ? kOutTile<K> * int(sizeof(V)) : 0);
  // resident CTAs to leave registers for: as many as the shared memory takes,
  // up to what 16 keys in registers allow.  (At two, with the registers that
  // allows, merges of 32- and 64-bit keys took 1.4 times as long.)
  static constexpr int FIT = 226 * 1024 / (BYTES + 1024);
  static constexpr int MOST = sizeof(K) == 4 ? 5 : sizeof(K) == 8 ? 4 : 6;
  static constexpr int MINB = FIT < MOST ? FIT : MOST;
};

// Shared memory of a tile sort: the keys by 32-bit word, so that a random
// key's word is a random bank, the positions, and the warps' counters.
template <class K>
struct MsTileSmem {
  // (fewer warps mean fewer counters to sweep; 128-bit keys need the warps, as
  // only two CTAs fit an SM)
  static constexpr int THREADS = sizeof(K) == 16 ? 512 : 256, MINB = sizeof(K) == 16 ? 2 : 4;
  static constexpr int ITEMS = kTile / THREADS, WARPS = THREADS / 32;
  static constexpr int WORDS = int(sizeof(K)) / 4;
  static constexpr int WH = 0;                              // u32 [2][WARPS][256], by pass parity
  static constexpr int TOT = WH + 2 * WARPS * 256 * 4;      // u32 [32]
  static constexpr int DIFF = TOT + 32 * 4;                 // u32 [WORDS] bits that differ in the tile
  static constexpr int KEYS = DIFF + 16;                    // u32 [WORDS][kTile]
  static constexpr int POS = KEYS + WORDS * kTile * 4;      // u16 [kTile]
  static constexpr int BYTES = POS + kTile * 2;
};

// One tile per CTA, sorted in place (src may equal dst): the keys stay where
// they were loaded and their positions are sorted, one stable counting sort per
// byte that is not the same in the whole tile.  A position's place comes from
// returning atomics (draw_rank); the result is checked and, out of order,
// sorted again with careful ranks.
//
// Bound by the shared-memory pipe (83-92 % busy): about 16 wavefronts per 32
// elements and byte.  The tile sort by merge rounds that this replaces read two
// keys per step of every thread's search in every round, which costs most for
// wide keys: 2^22 128-bit keys with values 315 us (now 203, all 16 bytes
// differing), 2^24 u32 keys 238 us (now 162).  Tiles of 8192 save one merge
// pass, but leave one CTA an SM for 128-bit keys: 275 us instead of 203.
template <class K, class V, bool HAS_V>
__global__ void __launch_bounds__(MsTileSmem<K>::THREADS, MsTileSmem<K>::MINB)
    k_ms_tile(const K* src, const V* vsrc, K* dst, V* vdst, uint32_t n,
              OrderTest order) {
  using S = MsTileSmem<K>;
  constexpr int THREADS = S::THREADS, ITEMS = S::ITEMS, WARPS = S::WARPS, WORDS = S::WORDS;
  extern __shared__ __align__(16) unsigned char smem[];
  uint32_t* s_tot = reinterpret_cast<uint32_t*>(smem + S::TOT);
  uint32_t* s_diff = reinterpret_cast<uint32_t*>(smem + S::DIFF);
  uint32_t* s_key = reinterpret_cast<uint32_t*>(smem + S::KEYS);
  uint16_t* s_pos = reinterpret_cast<uint16_t*>(smem + S::POS);
  const uint32_t base = blockIdx.x * uint32_t(kTile);
  const uint32_t len = min(uint32_t(kTile), n - base);
  const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
  union Words {
    K k;
    uint32_t w[WORDS];
    __device__ Words() {}
  };
  if (tid < WORDS) s_diff[tid] = 0u;
  __syncthreads();
  {
    Words x[ITEMS];
    Words x0;
    x0.k = src[base];
#pragma unroll
    for (int t = 0; t < ITEMS; ++t) {  // every load in flight before the first store
      const uint32_t i = uint32_t(t * THREADS + tid);
      x[t].k = i < len ? src[base + i] : x0.k;
    }
#pragma unroll
    for (int q = 0; q < WORDS; ++q) {
      uint32_t diff = 0u;
#pragma unroll
      for (int t = 0; t < ITEMS; ++t) {
        s_key[q * kTile + t * THREADS + tid] = x[t].w[q];
        diff |= x[t].w[q] ^ x0.w[q];
      }
      diff = __reduce_or_sync(kFull, diff);
      if (lane == 0 && diff != 0u) atomicOr(&s_diff[q], diff);
    }
  }
  for (int attempt = 0; attempt < 2; ++attempt) {
    const bool careful = attempt != 0;
    // item j of lane l of warp w is place (w * ITEMS + j) * 32 + l
    const uint32_t slot0 = uint32_t(warp * ITEMS * 32 + (order.mirror && !careful ? 31 - lane : lane));
#pragma unroll
    for (int t = 0; t < ITEMS; ++t) s_pos[t * THREADS + tid] = uint16_t(t * THREADS + tid);
    for (int i = tid; i < WARPS * 256 / 4; i += THREADS)
      reinterpret_cast<uint4*>(smem + S::WH)[i] = make_uint4(0u, 0u, 0u, 0u);
    __syncthreads();
    int parity = 0;
    for (int byte = 0; byte < int(sizeof(K)); ++byte) {
      const uint32_t shift = 8u * uint32_t(byte % 4);
      if ((s_diff[byte / 4] >> shift & 255u) == 0u) continue;  // CTA-uniform
      const uint32_t* word = s_key + byte / 4 * kTile;
      uint32_t* s_wh = reinterpret_cast<uint32_t*>(smem + S::WH) + parity * WARPS * 256;
      uint32_t* wh = s_wh + warp * 256;
      uint32_t pos[ITEMS], dr[ITEMS];  // digit << 16 | rank
#pragma unroll
      for (int j = 0; j < ITEMS; ++j) {
        const bool in = slot0 + j * 32 < len;
        pos[j] = in ? s_pos[slot0 + j * 32] : 0u;
      }
#pragma unroll
      for (int j = 0; j < ITEMS; ++j) dr[j] = word[pos[j]] >> shift & 255u;
#pragma unroll
      for (int j = 0; j < ITEMS; ++j)
        dr[j] = dr[j] << 16 | draw_rank(wh, dr[j], slot0 + j * 32 < len, careful, lane);
      __syncthreads();
      uint32_t c[WARPS], cnt = 0u;
      if (tid < 256) {
#pragma unroll
        for (int w = 0; w < WARPS; ++w) {
          c[w] = s_wh[w * 256 + tid];
          cnt += c[w];
        }
      }
      const uint32_t inc = warp_inclusive_scan(cnt, lane);
      if (lane == 31) s_tot[warp] = inc;
      __syncthreads();
      if (tid < 256) {
        uint32_t run = __reduce_add_sync(kFull, lane < 8 && lane < warp ? s_tot[lane] : 0u) + inc - cnt;
#pragma unroll
        for (int w = 0; w < WARPS; ++w) {
          s_wh[w * 256 + tid] = run;
          run += c[w];
        }
      }
      __syncthreads();
      uint32_t to[ITEMS];
#pragma unroll
      for (int j = 0; j < ITEMS; ++j) to[j] = wh[dr[j] >> 16] + (dr[j] & 0xffffu);
#pragma unroll
      for (int j = 0; j < ITEMS; ++j)
        if (slot0 + j * 32 < len) s_pos[to[j]] = uint16_t(pos[j]);
      parity ^= 1;
      uint4* zero = reinterpret_cast<uint4*>(smem + S::WH) + parity * WARPS * 256 / 4;
      for (int i = tid; i < WARPS * 256 / 4; i += THREADS) zero[i] = make_uint4(0u, 0u, 0u, 0u);
      __syncthreads();
    }
    bool bad = false;
#pragma unroll
    for (int t = 0; t < ITEMS; ++t) {
      const uint32_t i = uint32_t(t * THREADS + tid);
      if (i + 1u >= len) continue;
      const uint32_t a = s_pos[i], b = s_pos[i + 1];
      bool ordered = a < b;  // of equal keys the earlier first
#pragma unroll
      for (int q = 0; q < WORDS; ++q) {  // the top word decides last
        const uint32_t x = s_key[q * kTile + a], y = s_key[q * kTile + b];
        ordered = x < y || (x == y && ordered);
      }
      bad = bad || !ordered;
    }
    if (!__syncthreads_or(bad)) break;
    if (!careful && tid == 0) count_repair(order);
  }
  // in place: every value is read before the first is written
  V v[HAS_V ? ITEMS : 1];
  if constexpr (HAS_V) {
#pragma unroll
    for (int t = 0; t < ITEMS; ++t) {
      const uint32_t i = uint32_t(t * THREADS + tid);
      if (i < len) v[t] = vsrc[base + s_pos[i]];
    }
    __syncthreads();
  }
#pragma unroll
  for (int t = 0; t < ITEMS; ++t) {
    const uint32_t i = uint32_t(t * THREADS + tid);
    if (i >= len || !dbg_ok(uint64_t(base) + i, n, kSiteMergeTile)) continue;
    Words x;
#pragma unroll
    for (int q = 0; q < WORDS; ++q) x.w[q] = s_key[q * kTile + s_pos[i]];
    dst[base + i] = x.k;
    if constexpr (HAS_V) vdst[base + i] = v[t];
  }
}

// Elements taken from the left run a[0 .. na) at diagonal `diag`, as
// merge_path, by a whole warp: 32 probes at a time, so that a run of 2^22
// takes 5 dependent reads instead of 22.
template <class K>
__device__ __forceinline__ uint32_t merge_path_warp(const K* __restrict__ a, uint32_t na,
                                                    const K* __restrict__ b, uint32_t nb,
                                                    uint32_t diag) {
  const uint32_t lane = threadIdx.x & 31u;
  uint32_t lo = diag > nb ? diag - nb : 0u;
  uint32_t hi = min(diag, na);
  while (lo < hi) {  // the same in every lane
    const uint32_t span = hi - lo;
    const bool last = span <= 32u;
    const uint32_t mid = last ? lo + lane : lo + uint32_t(uint64_t(span) * (lane + 1u) / 33u);
    bool take = false;  // a[mid] comes before b[diag - 1 - mid]: true up to some mid, false after
    if (mid < hi) take = !key_less(b[diag - 1u - mid], a[mid]);
    const uint32_t c = uint32_t(__popc(__ballot_sync(0xffffffffu, take)));
    if (last) return lo + c;
    const uint32_t below = __shfl_sync(0xffffffffu, mid, int(c ? c - 1u : 0u));
    const uint32_t above = __shfl_sync(0xffffffffu, mid, int(c < 32u ? c : 31u));
    if (c < 32u) hi = above;
    if (c > 0u) lo = below + 1u;
  }
  return lo;
}

// Runs of width w (a multiple of kTile) are merged in pairs; output tile c
// starts at p = c * kOutTile inside the pair [base, base + 2w).  split[c] = how
// many of the pair's left-run elements precede that tile.  One warp a tile.
template <class K>
__global__ void k_ms_split(const K* __restrict__ src, uint32_t n, uint32_t w,
                           uint32_t* __restrict__ split, uint32_t tiles) {
  pdl_wait();
  const uint32_t c = (blockIdx.x * blockDim.x + threadIdx.x) / 32u;
  if (c >= tiles) return;
  const uint64_t p = uint64_t(c) * kOutTile<K>;
  const uint64_t base = p / (2ull * w) * (2ull * w);
  const uint32_t na = uint32_t(min(uint64_t(w), n - base));
  const uint32_t nb = uint32_t(n - base - na < w ? n - base - na : w);
  const uint32_t at = merge_path_warp(src + base, na, src + base + na, nb, uint32_t(p - base));
  if ((threadIdx.x & 31u) == 0u && dbg_ok(c, tiles, kSiteMergeSplit)) split[c] = at;
}

// Bound by latency: loads, a search of 12 dependent steps, 16 outputs one
// after another, each a shared-memory read.  2^24 u32 keys a pass: 46 us with
// the loads one after another and two reads an output, 41 now (u32 pairs 70 ->
// 55, u64 keys 81 -> 60, 2^22 128-bit keys with values 67 -> 52); the split
// 10-21 us a pass with one thread a tile, 5-8 now.
template <class K, class V, bool HAS_V>
__global__ void __launch_bounds__(kMsThreads<K>, MsSmem<K, V, HAS_V>::MINB) k_ms_merge(const K* __restrict__ src,
                                                            const V* __restrict__ vsrc,
                                                            K* __restrict__ dst,
                                                            V* __restrict__ vdst, uint32_t n,
                                                            uint32_t w,
                                                            const uint32_t* __restrict__ split) {
  using S = MsSmem<K, V, HAS_V>;
  extern __shared__ __align__(16) unsigned char smem[];
  K* sk = reinterpret_cast<K*>(smem + S::KEYS);
  uint16_t* sp = reinterpret_cast<uint16_t*>(smem + S::POS);
  V* sv = reinterpret_cast<V*>(smem + S::VALS);
  pdl_wait();
  const uint32_t c = blockIdx.x;
  const uint64_t p0 = uint64_t(c) * kOutTile<K>;
  const uint64_t p1 = min(p0 + kOutTile<K>, uint64_t(n));
  const uint64_t base = p0 / (2ull * w) * (2ull * w);  // kOutTile<K> divides 2w: one pair per CTA
  const uint32_t na = uint32_t(min(uint64_t(w), n - base));
  const uint32_t nb = uint32_t(n - base - na < w ? n - base - na : w);
  const uint32_t d0 = uint32_t(p0 - base), d1 = uint32_t(p1 - base);
  const uint32_t i0 = split[c];
  const uint32_t i1 = (p1 < base + na + nb) ? split[c + 1] : na;  // the pair's end: all of a
  const uint32_t j0 = d0 - i0, j1 = d1 - i1;
  const uint32_t la = i1 - i0, lb = j1 - j0;
  const uint32_t total = la + lb;
  const int tid = threadIdx.x;
  // the tile's elements: la from a + i0, then lb from b + j0; every load in
  // flight before the first store (one after another they took 16 us a tile)
  const uint64_t from_a = base + i0, from_b = base + na + j0 - la;
  K k[kMsItems];
  {
    V v[HAS_V ? kMsItems : 1];
#pragma unroll
    for (int t = 0; t < kMsItems; ++t) {
      const uint32_t i = uint32_t(t * kMsThreads<K> + tid);
      const uint64_t at = (i < la ? from_a : from_b) + i;
      if (i < total) {
        k[t] = src[at];
        if constexpr (HAS_V) v[t] = vsrc[at];
      }
    }
#pragma unroll
    for (int t = 0; t < kMsItems; ++t) {
      const uint32_t i = uint32_t(t * kMsThreads<K> + tid);
      if (i < total) {
        sk[pad(i)] = k[t];
        if constexpr (HAS_V) sv[i] = v[t];
      }
    }
  }
  __syncthreads();
  const uint32_t o = uint32_t(tid) * kMsItems;
  if (o < total) {
    const uint32_t i = merge_path(Padded<K>{sk, 0u}, la, Padded<K>{sk, la}, lb, o);
    merge_items<HAS_V>(sk, Run{i, la}, Run{la + o - i, total}, k, sp, o);
  }
  __syncthreads();
#pragma unroll
  for (int t = 0; t < kMsItems; ++t) {
    if (o + t < total) sk[pad(o + t)] = k[t];
  }
  __syncthreads();
#pragma unroll
  for (int t = 0; t < kMsItems; ++t) {
    const uint32_t i = uint32_t(t * kMsThreads<K> + tid);
    if (i >= total || !dbg_ok(p0 + i, n, kSiteMergeOut)) continue;
    dst[p0 + i] = sk[pad(i)];
    if constexpr (HAS_V) vdst[p0 + i] = sv[sp[pad(i)]];
  }
}

template <class K, class V, bool HAS_V>
struct MergeSort {
  using S = MsSmem<K, V, HAS_V>;

  static uint32_t tiles(size_t n) { return uint32_t((n + kOutTile<K> - 1) / kOutTile<K>); }
  // for every type alike: the smallest tiles
  static size_t workspace(size_t n) {
    return align_up(((n + kOutTileLeast - 1) / kOutTileLeast + 1) * 4, 256);
  }

  static cudaError_t run(void* keys, void* vals, void* keys_alt, void* vals_alt, size_t n,
                         void* ws, cudaStream_t s, int* in_alt) {
    auto tile_k = &k_ms_tile<K, V, HAS_V>;
    auto merge_k = &k_ms_merge<K, V, HAS_V>;
    using T = MsTileSmem<K>;
    if (prepare_kernel(reinterpret_cast<const void*>(tile_k), T::THREADS, T::BYTES) <= 0 ||
        prepare_kernel(reinterpret_cast<const void*>(merge_k), kMsThreads<K>, S::BYTES) <= 0)
      return cudaErrorInvalidConfiguration;
    K* bufk[2] = {static_cast<K*>(keys), static_cast<K*>(keys_alt)};
    V* bufv[2] = {static_cast<V*>(vals), static_cast<V*>(vals_alt)};
    const uint32_t nt = tiles(n);
    prof_before(s);
    tile_k<<<unsigned((n + kTile - 1) / kTile), T::THREADS, T::BYTES, s>>>(bufk[0], bufv[0], bufk[0], bufv[0], uint32_t(n),
                                            knobs_now().order);
    cudaError_t e = cudaGetLastError();
    prof_after(s, RS_KERNEL_MERGE, 2.0 * double(n) * double(sizeof(K) + (HAS_V ? sizeof(V) : 0)));
    if (e != cudaSuccess) return e;
    int cur = 0;
    uint32_t* split = static_cast<uint32_t*>(ws);
    for (uint64_t w = kTile; w < n; w *= 2) {
      auto launch = [&](auto kernel, unsigned blocks, int threads, int smem_bytes, auto... args) {
        cudaLaunchConfig_t cfg = {};
        cfg.gridDim = dim3(blocks);
        cfg.blockDim = dim3(unsigned(threads));
        cfg.dynamicSmemBytes = size_t(smem_bytes);
        cfg.stream = s;
        cudaLaunchAttribute attr[1];
        attr[0].id = cudaLaunchAttributeProgrammaticStreamSerialization;
        attr[0].val.programmaticStreamSerializationAllowed = 1;
        cfg.attrs = attr;
        cfg.numAttrs = pdl_enabled() ? 1 : 0;
        return cudaLaunchKernelEx(&cfg, kernel, args...);
      };
      const K* from = bufk[cur];
      const V* vfrom = bufv[cur];
      e = launch(&k_ms_split<K>, (nt + 7) / 8, 256, 0, from, uint32_t(n), uint32_t(w), split, nt);
      if (e != cudaSuccess) return e;
      prof_before(s);
      e = launch(merge_k, nt, kMsThreads<K>, S::BYTES, from, vfrom, bufk[cur ^ 1], bufv[cur ^ 1],
                 uint32_t(n), uint32_t(w), static_cast<const uint32_t*>(split));
      prof_after(s, RS_KERNEL_MERGE,
                 2.0 * double(n) * double(sizeof(K) + (HAS_V ? sizeof(V) : 0)));
      if (e != cudaSuccess) return e;
      cur ^= 1;
    }
    *in_alt = cur;
    return cudaSuccess;
  }
};

bool merge_types(int kb, int vb) {
  return (kb == 4 && (vb == 0 || vb == 4)) || (kb == 8 && (vb == 0 || vb == 8)) ||
         (kb == 16 && (vb == 0 || vb == 8));
}

size_t merge_workspace(size_t n) { return MergeSort<uint32_t, NoVal, false>::workspace(n); }

}  // namespace

}  // namespace rs

using namespace rs;

extern "C" {

rs_status rs_merge_workspace_bytes(int key_bytes, int val_bytes, size_t n, size_t* bytes) {
  if (!bytes || !merge_types(key_bytes, val_bytes) || n > RS_MAX_N) return RS_ERR_INVALID;
  *bytes = n <= 1 ? 0 : merge_workspace(n);
  return RS_OK;
}

rs_status rs_merge_sort(int key_bytes, int val_bytes, void* keys, void* vals, void* keys_alt,
                        void* vals_alt, size_t n, void* ws, size_t ws_bytes, rs_stream_t stream,
                        int* result_in_alt) {
  if (!result_in_alt || !merge_types(key_bytes, val_bytes) || n > RS_MAX_N)
    return RS_ERR_INVALID;
  *result_in_alt = 0;
  if (n <= 1) return RS_OK;
  auto al = [](const void* p, size_t a) { return reinterpret_cast<uintptr_t>(p) % a == 0; };
  if (!keys || !keys_alt || keys == keys_alt || !al(keys, size_t(key_bytes)) ||
      !al(keys_alt, size_t(key_bytes)))
    return RS_ERR_INVALID;
  if (val_bytes) {
    if (!vals || !vals_alt || vals == vals_alt || !al(vals, size_t(val_bytes)) ||
        !al(vals_alt, size_t(val_bytes)))
      return RS_ERR_INVALID;
  } else if (vals || vals_alt) {
    return RS_ERR_INVALID;
  }
  if (!ws || ws_bytes < merge_workspace(n) || !al(ws, 256)) return RS_ERR_WORKSPACE;
  cudaStream_t s = reinterpret_cast<cudaStream_t>(stream);
  int in_alt = 0;
  cudaError_t e;
  if (key_bytes == 4 && val_bytes == 0)
    e = MergeSort<uint32_t, NoVal, false>::run(keys, vals, keys_alt, vals_alt, n, ws, s, &in_alt);
  else if (key_bytes == 4)
    e = MergeSort<uint32_t, uint32_t, true>::run(keys, vals, keys_alt, vals_alt, n, ws, s,
                                                 &in_alt);
  else if (key_bytes == 8 && val_bytes == 0)
    e = MergeSort<uint64_t, NoVal, false>::run(keys, vals, keys_alt, vals_alt, n, ws, s, &in_alt);
  else if (key_bytes == 8)
    e = MergeSort<uint64_t, uint64_t, true>::run(keys, vals, keys_alt, vals_alt, n, ws, s,
                                                 &in_alt);
  else if (val_bytes == 0)
    e = MergeSort<Key128, NoVal, false>::run(keys, vals, keys_alt, vals_alt, n, ws, s, &in_alt);
  else
    e = MergeSort<Key128, uint64_t, true>::run(keys, vals, keys_alt, vals_alt, n, ws, s, &in_alt);
  if (e != cudaSuccess) return RS_ERR_CUDA;
  *result_in_alt = in_alt;
  return RS_OK;
}

}  // extern "C"
