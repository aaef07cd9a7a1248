// Batched segmented sort: the counting-sort passes of Sec. 2.6 applied
// independently to every segment [off[s], off[s+1]) of one array, for all
// segments in one persistent launch.
//
//   k_seg_plan        classifies segments (tiny ones fit one warp, short ones
//                     one CTA, long ones are tiled), numbers the work items
//                     and maps every histogram chunk to its segment.
//   k_seg_small       short segments, each sorted whole in one CTA's shared
//                     memory (every pass) or by one warp; once more, with
//                     larger CTAs, for the medium ones;
//   k_seg_hist        the digit histograms of the long segments, chunk by
//                     chunk; each segment's last chunk scans them and writes
//                     the descriptors of the segment's pass tiles;
//   k_seg_persistent  SMs x resident CTAs, each looping over one global work
//                     queue (an atomic counter) in this order:
//                       [pass 0 tiles of long segments] ... [pass P-1 tiles]
//                     (kept apart from the short segments so that it needs
//                     few registers and four CTAs fit on an SM)
//                     A tile reads its descriptor (written by the histogram
//                     kernel, launched before); a tile of pass p > 0 waits
//                     (bounded) until every tile of pass p-1 of its segment is
//                     written.  Every wait is on items taken from the queue
//                     earlier, which are held by running CTAs, so the queue
//                     always makes progress.
#pragma once

#include "rs_kernels.cuh"

namespace rs {

constexpr uint32_t kDevInvalid = 1;  // RS_ERR_INVALID seen on the device

struct SegDesc {
  uint64_t off;    // first element
  uint32_t len;    // elements
  uint32_t tile0;  // first global pass tile
  uint32_t chunk0; // first global histogram chunk
  uint32_t seg;    // segment id
  uint32_t pad[2];
};
static_assert(sizeof(SegDesc) == 32, "SegDesc is 32 bytes");

// Everything a pass tile needs to start, in one 32-byte read: written for
// every tile of a long segment by the segment's last histogram chunk, so the
// tile needs no dependent read of a tile map, a segment descriptor and the
// segment's state before it can load its keys.
struct TileDesc {
  uint64_t off;    // the segment's first element
  uint32_t len;    // the segment's elements
  uint32_t li;     // long-segment index (state, counts, offsets)
  uint32_t tile0;  // the segment's first global pass tile
  uint32_t exec;   // passes of the segment that move data (after the parity rule)
  uint32_t pad[2];
};
static_assert(sizeof(TileDesc) == 32, "TileDesc is 32 bytes");

// Per long segment: histogram ticket, done counters.
constexpr int kSegStateWords = 16;
enum SegStateField { kSegTicket = 0, kSegDone0 = 3 };

// Plan results in Ctrl::tile_counter[]
enum SegCtrlField {
  kQueue = 0,    // work-queue ticket
  kNSmall = 1,
  kNLarge = 2,
  kNTiles = 3,   // pass tiles of all long segments (one pass)
  kNChunks = 4,  // histogram chunks of all long segments
  kNTiny = 6,    // segments of 1 to 32 elements
  kSmallQueue = 7,  // work-queue ticket of the short segments
  kNMedium = 8,
  kMediumQueue = 9  // and of the medium ones
};
constexpr uint32_t kTinyMax = 32;

struct SegLayout {
  size_t small_ids, medium_ids, descs, tdesc, chunk_seg, state, counts, offsets, status, total;
  size_t tiles_max, chunks_max;
};

inline SegLayout seg_layout(size_t n, size_t nseg, int passes, int radix_bits, int tile,
                            int chunk) {
  SegLayout L{};
  const size_t radix = size_t(1) << radix_bits;
  L.tiles_max = align_up((n + tile - 1) / tile + nseg, 4);
  L.chunks_max = (n + chunk - 1) / chunk + nseg;
  L.state = 256;
  L.counts = align_up(L.state + nseg * kSegStateWords * 4, 256);
  L.offsets = align_up(L.counts + nseg * passes * radix * 4, 256);
  L.small_ids = align_up(L.offsets + nseg * passes * radix * 4, 256);
  L.medium_ids = align_up(L.small_ids + nseg * 4, 256);
  L.descs = align_up(L.medium_ids + nseg * 4, 256);
  L.tdesc = align_up(L.descs + nseg * sizeof(SegDesc), 256);
  L.chunk_seg = align_up(L.tdesc + L.tiles_max * sizeof(TileDesc), 256);
  L.status = align_up(L.chunk_seg + L.chunks_max * 4, 256);
  L.total = align_up(L.status + size_t(passes) * L.tiles_max * radix * 4, 256);
  return L;
}

struct SegArgs {
  const uint64_t* off;
  int begin_bit, end_bit, passes;
  Ctrl* ctrl;
  const uint32_t* small_ids;
  const uint32_t* medium_ids;
  const SegDesc* descs;
  TileDesc* tdesc;    // [tiles_max]
  const uint32_t* chunk_seg;
  uint32_t* state;    // [nseg][kSegStateWords]
  uint32_t* counts;   // [nseg][passes][RADIX]
  uint32_t* offsets;  // [nseg][passes][RADIX]
  uint32_t* status;   // [passes][tiles_max][RADIX]
  uint64_t tiles_max;
  uint64_t nseg;      // segments (debug bounds checks)
  Knobs knobs;
};

// Numbers the work, one segment a thread.  Segments longer than medium_max are
// "long"; of the others, those of 1 to 32 elements are "tiny" (listed from the
// end of small_ids), those of up to small_max "small", the rest "medium"; empty
// ones are left out.  Where one CTA sees every segment (up to THREADS of them)
// and one is long, none is medium: so few medium ones leave SMs idle, one
// after the other with the long ones' tiles, which they can fill instead (108
// segments of up to 24,000 u64 keys 175 us with medium ones and 115 without;
// up to 18,000 u64 pairs 191 and 130; 300 and more took the same or less with
// them).  The order
// inside the lists is of no consequence, so each CTA takes its places from
// global counters: with one CTA scanning all segments in order, 20,000 of them
// took 87 us.  The state of long segments, and the digit counts of those of
// several chunks, are cleared here: clearing every segment's took 80 MB of
// stores for 20,000.  Bad offsets are reported; the kernels that follow then
// do nothing.
template <int THREADS, int RADIX>
__global__ void __launch_bounds__(THREADS)
    k_seg_plan(uint64_t n, uint32_t small_max, uint32_t medium_max, uint32_t tile, uint32_t chunk, uint64_t chunks_max,
               uint32_t* __restrict__ small_ids, uint32_t* __restrict__ medium_ids,
               SegDesc* __restrict__ descs, uint32_t* __restrict__ chunk_seg, SegArgs a) {
  constexpr int COUNTS = 6, WARPS = THREADS / 32;
  const int field[COUNTS] = {kNTiny, kNSmall, kNLarge, kNTiles, kNChunks, kNMedium};
  __shared__ uint32_t s_tot[COUNTS][WARPS];
  const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
  const uint64_t s = uint64_t(blockIdx.x) * THREADS + tid;
  uint64_t from = 0;
  uint32_t len = 0u;
  bool bad = s == 0 && (a.off[0] != 0ull || a.off[a.nseg] != n);
  if (s < a.nseg) {
    from = a.off[s];
    const uint64_t to = a.off[s + 1];
    if (to < from || to > n || to - from > uint64_t((1u << 30) - 1u)) bad = true;
    else len = uint32_t(to - from);
  }
  const uint32_t line =
      gridDim.x == 1u && __syncthreads_or(len > medium_max) ? small_max : medium_max;
  const bool tiny = len >= 1u && len <= kTinyMax, lng = len > line;
  const bool small = len > kTinyMax && len <= small_max, medium = len > small_max && !lng;
  const uint32_t nt = lng ? (len + tile - 1u) / tile : 0u, nc = lng ? (len + chunk - 1u) / chunk : 0u;
  const uint32_t mine[COUNTS] = {tiny, small, lng, nt, nc, medium};
  uint32_t at[COUNTS];
#pragma unroll
  for (int q = 0; q < COUNTS; ++q) {
    const uint32_t inc = warp_inclusive_scan(mine[q], lane);
    if (lane == 31) s_tot[q][warp] = inc;
    at[q] = inc - mine[q];
  }
  __syncthreads();
  if (tid < COUNTS) {  // thread q: the warps' places among count q
    uint32_t sum = 0u;
    for (int w = 0; w < WARPS; ++w) sum += s_tot[tid][w];
    uint32_t run = sum ? atomicAdd(&a.ctrl->tile_counter[field[tid]], sum) : 0u;
    for (int w = 0; w < WARPS; ++w) {
      const uint32_t x = s_tot[tid][w];
      s_tot[tid][w] = run;
      run += x;
    }
  }
  __syncthreads();
#pragma unroll
  for (int q = 0; q < COUNTS; ++q) at[q] += s_tot[q][warp];
  const uint64_t slot = tiny ? a.nseg - 1u - at[0] : at[1];
  if ((tiny || small) && dbg_ok(slot, a.nseg, kSiteSegPlan)) small_ids[slot] = uint32_t(s);
  if (medium && dbg_ok(at[5], a.nseg, kSiteSegPlan)) medium_ids[at[5]] = uint32_t(s);
  const uint32_t li = at[2], c0 = at[4];
  bool map_ok = false;
  if (lng) {
    SegDesc d;
    d.off = from;
    d.len = len;
    d.tile0 = at[3];
    d.chunk0 = c0;
    d.seg = uint32_t(s);
    d.pad[0] = d.pad[1] = 0u;
    if (dbg_ok(li, a.nseg, kSiteSegPlan)) descs[li] = d;
    map_ok = uint64_t(d.tile0) + nt <= a.tiles_max && uint64_t(c0) + nc <= chunks_max;
    if (!map_ok) bad = true;
  }
  if (bad) report_error(a.ctrl, kDevInvalid, 0u);
  // each warp writes its lanes' long segments one after another, consecutive
  // entries per store: the chunk map, the state, the counts
  for (uint32_t m = __ballot_sync(kFull, map_ok); m != 0u; m &= m - 1u) {
    const int src = __ffs(int(m)) - 1;
    const uint32_t sli = __shfl_sync(kFull, li, src), sc0 = __shfl_sync(kFull, c0, src);
    const uint32_t snc = __shfl_sync(kFull, nc, src);
    for (uint32_t i = uint32_t(lane); i < snc; i += 32)
      if (dbg_ok(uint64_t(sc0) + i, chunks_max, kSiteSegPlan)) chunk_seg[sc0 + i] = sli;
    if (!dbg_ok(sli, a.nseg, kSiteSegState)) continue;
    if (lane < kSegStateWords) a.state[size_t(sli) * kSegStateWords + lane] = 0u;
    if (snc > 1u) {
      uint32_t* cnt = a.counts + size_t(sli) * a.passes * RADIX;
      for (int i = lane; i < a.passes * RADIX; i += 32) cnt[i] = 0u;
    }
  }
}

// SMALL_ITEMS: keys per thread of the short-segment sort, whose tile bounds a
// short segment.
template <class K, int VB, int RADIX_BITS, int THREADS, int ITEMS, int CHUNK_TILES,
          int SMALL_ITEMS = ITEMS, bool INDEX = true>
struct SegKernelCfg {
  static constexpr int RADIX = 1 << RADIX_BITS;
  static constexpr int TILE = THREADS * ITEMS;
  static constexpr int SMALL_TILE = THREADS * SMALL_ITEMS;
  static constexpr int CHUNK = TILE * CHUNK_TILES;
  static constexpr int MAXP = (8 * int(sizeof(K)) + RADIX_BITS - 1) / RADIX_BITS;
  // histogram kernel: [pass][digit][16 lane slots] u32 counters, 1024 threads
  static constexpr int HIST_THREADS = 1024;
  static constexpr int HIST_SLOTS = 16;
  static constexpr int HIST_BYTES = MAXP * RADIX * HIST_SLOTS * 4;
  // two CTAs per SM while their counters fit (32-bit keys), else one
  static constexpr int HIST_MINB = HIST_BYTES <= 100 * 1024 ? 2 : 1;
  using OS = OnesweepSmem<K, VB, RADIX_BITS, THREADS, ITEMS, INDEX>;
  static constexpr int MISC = (OS::BYTES + 15) / 16 * 16;  // u32 [8]
  static constexpr int BYTES = MISC + 32;
};

// One segment of at most 32 elements, sorted by one warp: an element's place
// is the number of elements that are smaller, or equal and earlier.
template <class K, int VB>
__device__ __forceinline__ void seg_warp_sort(const K* kin, const ValT<VB>* vin, K* kout,
                                              ValT<VB>* vout, uint32_t len, K looked) {
  const uint32_t lane = threadIdx.x & 31u;
  K k = K(0);
  ValT<VB> v = 0;
  if (lane < len) {
    k = kin[lane];
    if constexpr (VB > 0) v = vin[lane];
  }
  const K mine = k & looked;
  uint32_t place = 0u;
  for (uint32_t j = 0; j < len; ++j) {
    const K other = __shfl_sync(kFull, mine, int(j));
    place += (other < mine || (other == mine && j < lane)) ? 1u : 0u;
  }
  // (every load of the warp has completed: its key was shuffled, its value
  // is ordered by the warp barrier)
  __syncwarp();
  if (lane < len && dbg_ok(place, len, kSiteSegSmallOut)) {
    kout[place] = k;
    if constexpr (VB > 0) vout[place] = v;
  }
}

// The short segments: those of up to 32 elements one warp each, the others
// one CTA each, taken from a queue (the next one is asked for while the
// current one is sorted), so that long and short ones even out.  MEDIUM: the
// medium list alone, on CTAs of 1024 threads: one read and one write of a
// segment instead of a histogram and a tile or two in every pass (20,000
// log-uniform segments of 2^26 pairs: the tiled passes take 36 % less).
template <class K, int VB, int RADIX_BITS, int THREADS, int ITEMS, bool INDEX, int MINB,
          bool MEDIUM = false>
__global__ void __launch_bounds__(THREADS, MINB)
    k_seg_small(K* __restrict__ k0, ValT<VB>* __restrict__ v0, K* __restrict__ k1,
                ValT<VB>* __restrict__ v1, SegArgs a) {
  extern __shared__ __align__(16) unsigned char smem[];
  __shared__ uint32_t s_next[2];
  const int passes = a.passes;
  K* kout = (passes & 1) ? k1 : k0;  // where the pass count parity puts the result
  ValT<VB>* vout = (passes & 1) ? v1 : v0;
  pdl_wait();  // the planner (and what is before this kernel) is complete
  if (a.ctrl->error != 0u) return;  // bad offsets: nothing is written
  constexpr int QUEUE = MEDIUM ? kMediumQueue : kSmallQueue;
  const uint32_t* ids = MEDIUM ? a.medium_ids : a.small_ids;
  const uint32_t n_small = a.ctrl->tile_counter[MEDIUM ? kNMedium : kNSmall];
  uint32_t n_tiny = 0u;
  if constexpr (!MEDIUM) n_tiny = a.ctrl->tile_counter[kNTiny];
  const K looked = (a.end_bit - a.begin_bit == 8 * int(sizeof(K)))
                       ? ~K(0)
                       : K(((K(1) << (a.end_bit - a.begin_bit)) - K(1)) << a.begin_bit);
  if (threadIdx.x == 0) s_next[0] = atomicAdd(&a.ctrl->tile_counter[QUEUE], 1u);
  __syncthreads();
  for (uint32_t it = 0;; ++it) {
    const uint32_t i = s_next[it & 1u];
    if (i >= n_small) break;
    if (threadIdx.x == 0) s_next[(it + 1u) & 1u] = atomicAdd(&a.ctrl->tile_counter[QUEUE], 1u);
    const uint32_t s = ids[i];
    const uint64_t b = a.off[s];
    const uint32_t len = uint32_t(a.off[s + 1] - b);
    cta_sort<K, VB, RADIX_BITS, THREADS, ITEMS, INDEX>(k0 + b, v0 + b, kout + b, vout + b, len,
                                                       a.begin_bit, a.end_bit, smem,
                                                       KeyXf<K>{}, a.knobs.order);
    __syncthreads();
  }
  const uint32_t warps = gridDim.x * (THREADS / 32);
  for (uint32_t i = (blockIdx.x * THREADS + threadIdx.x) / 32u; i < n_tiny; i += warps) {
    const uint32_t s = a.small_ids[a.nseg - 1u - i];  // listed from the end
    const uint64_t b = a.off[s];
    const uint32_t len = uint32_t(a.off[s + 1] - b);
    seg_warp_sort<K, VB>(k0 + b, v0 + b, kout + b, vout + b, len, looked);
  }
}

// Digit histograms of the long segments, every pass (Sec. 2.6, the counting
// step), one chunk of CHUNK keys at a time, grid-stride over the chunks.  As in
// the whole-array upsweep: 16-byte loads, every pass's digit counted into
// per-lane-slot shared counters, then the chunk's counts added to its
// segment's.  The chunk also clears the look-back words of its tiles.  The
// last chunk of a segment (ticket; most segments are one chunk, and need no
// counts in memory) scans the segment's histograms, chooses the passes that
// move data and writes the descriptors of the segment's pass tiles.
//
// Bound by latency for segments of a tile or two: adding every chunk up in
// memory and scanning one pass after another took 218 us for the 3,500
// segments of over 4,096 of 2^26 pairs in 20,000 segments; the 85 us now are
// for those over 20,480.
template <class K, int RADIX_BITS, int THREADS, int MAXP, int SLOTS, int CHUNK, int TILE,
          int CHUNK_TILES, int MINB = 2>
__global__ void __launch_bounds__(THREADS, MINB)
    k_seg_hist(const K* __restrict__ k0, SegArgs a) {
  constexpr int RADIX = 1 << RADIX_BITS;
  constexpr int VEC = 16 / int(sizeof(K));
  static_assert(THREADS == 1024 && RADIX % 32 == 0, "32 warps' sums, whole warps per pass");
  extern __shared__ uint32_t sh[];  // [passes][RADIX][SLOTS]
  __shared__ uint32_t s_tot[32];
  __shared__ int s_last;
  __shared__ uint32_t s_one;
  const int tid = threadIdx.x, lane = tid & 31;
  const uint32_t slot = uint32_t(lane & (SLOTS - 1));
  const int passes = a.passes;
  uint32_t shiftp[MAXP], maskp[MAXP];
#pragma unroll
  for (int p = 0; p < MAXP; ++p) {
    const int lo = a.begin_bit + p * RADIX_BITS;
    const int hi = min(lo + RADIX_BITS, a.end_bit);
    shiftp[p] = p < passes ? uint32_t(lo) : 0u;
    maskp[p] = p < passes ? ((1u << (hi - lo)) - 1u) : 0u;
  }
  auto count_key = [&](K k) {
#pragma unroll
    for (int p = 0; p < MAXP; ++p)
      if (p < passes)
        atomicAdd(&sh[(p * RADIX + int(digit_of(k, shiftp[p], maskp[p]))) * SLOTS + int(slot)],
                  1u);
  };
  pdl_wait();
  if (a.ctrl->error != 0u) return;  // bad offsets
  const uint32_t n_chunks = a.ctrl->tile_counter[kNChunks];
  const int words = passes * RADIX * SLOTS;
  for (uint32_t item = blockIdx.x; item < n_chunks; item += gridDim.x) {
    const uint32_t li = a.chunk_seg[item];
    const SegDesc d = a.descs[li];
    const uint32_t lc = item - d.chunk0;
    const uint32_t start = lc * uint32_t(CHUNK);
    const uint32_t len = min(uint32_t(CHUNK), d.len - start);
    const K* keys = k0 + d.off + start;
    for (int i = tid; i < words; i += THREADS) sh[i] = 0u;
    __syncthreads();
    // 16-byte aligned body, scalar head and tail
    const uintptr_t addr = reinterpret_cast<uintptr_t>(keys);
    uint32_t head = uint32_t(((16u - (addr & 15u)) & 15u) / sizeof(K));
    if (head > len) head = len;
    const uint32_t nvec = (len - head) / VEC;
    const uint32_t tail = head + nvec * VEC;
    if (uint32_t(tid) < head) count_key(keys[tid]);
    if (uint32_t(tid) < len - tail) count_key(keys[tail + tid]);
    const uint4* vp = reinterpret_cast<const uint4*>(keys + head);
    // two 16-byte loads in flight per thread before their keys are counted
    // (four need more than the 32 registers two CTAs of 1024 threads leave)
    constexpr int UNROLL = 2;
    for (uint32_t i0 = tid; i0 < nvec; i0 += THREADS * UNROLL) {
      uint4 buf[UNROLL];
#pragma unroll
      for (int u = 0; u < UNROLL; ++u) {
        const uint32_t i = i0 + uint32_t(u) * THREADS;
        if (i < nvec) buf[u] = vp[i];
      }
#pragma unroll
      for (int u = 0; u < UNROLL; ++u) {
        if (i0 + uint32_t(u) * THREADS < nvec) {
          const K* ks = reinterpret_cast<const K*>(&buf[u]);
#pragma unroll
          for (int e = 0; e < VEC; ++e) count_key(ks[e]);
        }
      }
    }
    __syncthreads();
    // the chunk's counts, one (pass, digit) per thread; a segment of several
    // chunks adds them up in memory
    constexpr int PER = THREADS / RADIX;  // passes at a time
    const int pq = tid / RADIX, dq = tid % RADIX;
    const uint32_t chunks = (d.len + CHUNK - 1) / CHUNK;
    uint32_t* cnt = a.counts + size_t(li) * passes * RADIX;
    uint32_t mine[(MAXP + PER - 1) / PER];
#pragma unroll
    for (int q = 0; q < (MAXP + PER - 1) / PER; ++q) {
      const int p = q * PER + pq;
      uint32_t c = 0u;
      if (p < passes) {
        const uint32_t* row = sh + (p * RADIX + dq) * SLOTS;
#pragma unroll
        for (int l = 0; l < SLOTS; ++l) c += row[(l + lane) & (SLOTS - 1)];  // rotated: no conflicts
        if (chunks > 1u && c != 0u &&
            dbg_ok((uint64_t(li) * passes + p) * RADIX + dq, a.nseg * passes * RADIX,
                   kSiteSegCounts))
          atomicAdd(&cnt[p * RADIX + dq], c);
      }
      mine[q] = c;
    }
    // clear the look-back words of this chunk's tiles [ta, tb), every pass.
    // In the [tile/4][digit][tile%4] layout one digit's words of four
    // consecutive tiles are 16 contiguous bytes: consecutive threads clear
    // consecutive 16-byte groups, a whole group when its four tiles are all
    // this chunk's, else word by word (the neighbouring segment owns the rest)
    const uint32_t t_first = lc * uint32_t(CHUNK_TILES);
    const uint32_t t_last = min(t_first + uint32_t(CHUNK_TILES), (d.len + TILE - 1) / TILE);
    const uint32_t ta = d.tile0 + t_first, tb = d.tile0 + t_last;
    const uint32_t g0 = ta / 4u, ng = (tb - 1u) / 4u - g0 + 1u;
    for (int p = 0; p < passes; ++p) {
      uint32_t* st = a.status + size_t(p) * a.tiles_max * RADIX;
      for (uint32_t i = tid; i < ng * RADIX; i += THREADS) {
        const uint32_t g = g0 + i / RADIX;
        const size_t q = size_t(g) * RADIX + i % RADIX;  // the 16-byte group
        if (!dbg_ok(q, a.tiles_max * RADIX / 4, kSiteSegClear)) continue;
        if (4u * g >= ta && 4u * g + 3u < tb) {
          reinterpret_cast<uint4*>(st)[q] = make_uint4(0u, 0u, 0u, 0u);
        } else {
#pragma unroll
          for (uint32_t c = 0; c < 4u; ++c)
            if (4u * g + c >= ta && 4u * g + c < tb) st[q * 4 + c] = 0u;
        }
      }
    }
    bool last = true;
    if (chunks > 1u) {
      __syncthreads();
      if (tid == 0) {
        // the CTA's counts and cleared words (ordered before by the barrier)
        // become visible before the ticket
        __threadfence();
        uint32_t* state = a.state + size_t(li) * kSegStateWords;
        s_last = dbg_ok(li, a.nseg, kSiteSegState) &&
                 atomicAdd(&state[kSegTicket], 1u) == chunks - 1u;
      }
      __syncthreads();
      last = s_last != 0;
      if (last) {
        __threadfence();
#pragma unroll
        for (int q = 0; q < (MAXP + PER - 1) / PER; ++q)
          mine[q] = q * PER + pq < passes ? ld_relaxed(&cnt[(q * PER + pq) * RADIX + dq]) : 0u;
      }
    }
    if (last) {
      // the segment's counts are complete: scan every pass's at once, and
      // find the passes that move data
      uint32_t* offs = a.offsets + size_t(li) * passes * RADIX;
      if (tid == 0) s_one = 0u;
#pragma unroll
      for (int q = 0; q < (MAXP + PER - 1) / PER; ++q) {
        const int p = q * PER + pq;
        const uint32_t inc = warp_inclusive_scan(mine[q], lane);
        const int warp = tid >> 5;
        __syncthreads();  // s_one is clear; the round before has read s_tot
        if (lane == 31) s_tot[warp] = inc;
        if (mine[q] == d.len) atomicOr(&s_one, 1u << p);  // one digit value holds every key
        __syncthreads();
        const int w0 = warp / (RADIX / 32) * (RADIX / 32);  // my pass's first warp
        const uint32_t start =
            __reduce_add_sync(kFull, lane >= w0 && lane < warp ? s_tot[lane] : 0u) + inc - mine[q];
        if (p < passes && dbg_ok((uint64_t(li) * passes + p) * RADIX + dq,
                                 a.nseg * passes * RADIX, kSiteSegCounts))
          offs[p * RADIX + dq] = start;
      }
      uint32_t exec = ~s_one & ((1u << passes) - 1u);
      if ((__popc(exec) & 1) != (passes & 1)) {  // every thread: the same exec
        const uint32_t skipped = ~exec & ((1u << passes) - 1u);
        exec |= skipped & (0u - skipped);
      }
      // every pass tile of the segment learns where it is and which passes
      // move data from one descriptor (read by the pass kernel, launched after)
      const uint32_t ntiles = (d.len + TILE - 1) / TILE;
      for (uint32_t t = tid; t < ntiles; t += THREADS) {
        if (!dbg_ok(uint64_t(d.tile0) + t, a.tiles_max, kSiteSegState)) continue;
        TileDesc td;
        td.off = d.off;
        td.len = d.len;
        td.li = li;
        td.tile0 = d.tile0;
        td.exec = exec;
        td.pad[0] = td.pad[1] = 0u;
        a.tdesc[d.tile0 + t] = td;
      }
    }
    __syncthreads();
  }
}

template <class K, int VB, int RADIX_BITS, int THREADS, int ITEMS, int CHUNK_TILES,
          int MINB, bool INDEX>
__global__ void __launch_bounds__(THREADS, MINB)
    k_seg_persistent(K* __restrict__ k0, ValT<VB>* __restrict__ v0, K* __restrict__ k1,
                     ValT<VB>* __restrict__ v1, SegArgs a) {
  using V = ValT<VB>;
  using C = SegKernelCfg<K, VB, RADIX_BITS, THREADS, ITEMS, CHUNK_TILES, ITEMS, INDEX>;
  constexpr int RADIX = C::RADIX, TILE = C::TILE;
  extern __shared__ __align__(16) unsigned char smem[];
  uint32_t* s_misc = reinterpret_cast<uint32_t*>(smem + C::MISC);
  const int tid = threadIdx.x;
  Ctrl* ctrl = a.ctrl;
  const int passes = a.passes;

  pdl_wait();
  const uint32_t n_tiles = ctrl->tile_counter[kNTiles];
  const uint32_t q_end = uint32_t(passes) * n_tiles;

  for (;;) {
    if (tid == 0) {
      s_misc[0] = atomicAdd(&ctrl->tile_counter[kQueue], 1u);
      s_misc[1] = ld_relaxed(&ctrl->error);
    }
    __syncthreads();
    const uint32_t item = s_misc[0];
    if (item >= q_end || s_misc[1] != 0u) break;  // CTA-uniform

    // ---- one tile of one pass of a long segment.  The histogram kernel
    // (launched before this one) has written the tile's descriptor and every
    // segment's scans; a tile of pass p > 0 waits (bounded) until every tile of
    // pass p - 1 of its segment is written, whether that pass moved data or not
    const int p = int(item / n_tiles);
    const uint32_t gt = item - uint32_t(p) * n_tiles;
    const TileDesc d = a.tdesc[gt];
    const uint32_t li = d.li;
    uint32_t* state = a.state + size_t(li) * kSegStateWords;
    const uint32_t ntiles = (d.len + TILE - 1) / TILE;
    const uint32_t exec = d.exec;
    bool ok = true;
    if (p > 0) {
      if (tid == 0) {
        bool w = ld_relaxed(&state[kSegDone0 + p - 1]) >= ntiles;
        if (w)
          __threadfence();  // acquire: the previous pass's output
        else
          w = wait_geq(&state[kSegDone0 + p - 1], ntiles, ctrl, a.knobs.timeout_ns, gt);
        s_misc[3] = w ? 1u : 0u;
      }
      __syncthreads();
      ok = s_misc[3] != 0u;
    }
    if (ok && ((exec >> p) & 1u)) {
      if (tid == 0) {
        const int lo = a.begin_bit + p * RADIX_BITS;
        auto* t = reinterpret_cast<TileArgs<K, VB>*>(smem + C::OS::ARGS);
        K *ka = k0 + d.off, *kb = k1 + d.off;
        V *va = nullptr, *vb = nullptr;
        if constexpr (VB > 0) {
          va = v0 + d.off;
          vb = v1 + d.off;
        }
        // segments are short: a flat walk over tiles, no groups
        pass_args<K, VB, RADIX>(t, ka, kb, va, vb, d.len, p, exec, uint32_t(lo),
                                (1u << (min(lo + RADIX_BITS, a.end_bit) - lo)) - 1u,
                                a.offsets + (size_t(li) * passes + p) * RADIX,
                                LookBackWords{a.status + size_t(p) * a.tiles_max * RADIX, nullptr,
                                              nullptr, nullptr},
                                ntiles, KeyXf<K>{}, a.knobs);
        t->tile0 = d.tile0;
        t->lb_words = a.tiles_max * RADIX;
        t->drop_tile = t->bad_tile = -1;
        t->trace = nullptr;
      }
      __syncthreads();
      onesweep_tile<K, VB, RADIX_BITS, THREADS, ITEMS, INDEX, true, false, true>(gt - d.tile0, ctrl,
                                                                    a.knobs.timeout_ns, smem);
    }
    __syncthreads();
    if (tid == 0) {
      __threadfence();  // the tile's output, ordered before by the barrier, then the count
      if (dbg_ok(li, a.nseg, kSiteSegState)) atomicAdd(&state[kSegDone0 + p], 1u);
    }
    __syncthreads();
  }
}

}  // namespace rs
