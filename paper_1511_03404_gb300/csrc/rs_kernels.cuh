// Device kernels of the LSD radix sort (arXiv 1511.03404, Sec. 2.6).
//
// One sort = one upsweep + one onesweep launch per digit pass:
//   k_upsweep   reads the keys once and builds the digit histogram of every
//               pass (the "count" step of each counting sort); its last CTA
//               takes the exclusive scan of each histogram (the "prefix"
//               step) and decides which passes move data.
//   k_onesweep  one digit pass: the tile's digit counts are published for the
//               following tiles, then its keys draw their places in the tile
//               (stable: warp-major, then item, then lane order, checked and
//               put right where the draws came in another order), the tile's
//               global digit offsets come from a look-back over the preceding
//               tiles, and the tile is scattered through shared memory so that
//               each digit run is written contiguously (the stable "scatter"
//               step).
//   k_small_sort  arrays that fit one tile: all passes in one CTA, in shared
//               memory, in a single launch.
// All arithmetic is on unsigned integers; results are exact.
#pragma once

#include <cuda_runtime.h>

#include <cstdint>
#include <type_traits>

#include "rs_common.h"
#include "rs_debug.cuh"

namespace rs {

constexpr unsigned kFull = 0xffffffffu;

template <int VB>
using ValT = typename std::conditional<VB == 8, uint64_t, uint32_t>::type;

// ---------------------------------------------------------------- helpers

__device__ __forceinline__ uint32_t ld_relaxed(const uint32_t* p) {
  uint32_t v;
  asm volatile("ld.relaxed.gpu.global.u32 %0, [%1];" : "=r"(v) : "l"(p) : "memory");
  return v;
}

__device__ __forceinline__ uint4 ld_relaxed_v4(const uint32_t* p) {
  uint4 v;
  asm volatile("ld.relaxed.gpu.global.v4.u32 {%0, %1, %2, %3}, [%4];"
               : "=r"(v.x), "=r"(v.y), "=r"(v.z), "=r"(v.w)
               : "l"(p)
               : "memory");
  return v;
}

__device__ __forceinline__ uint32_t ld_relaxed_u16(const uint16_t* p) {
  uint16_t v;
  asm volatile("ld.relaxed.gpu.global.u16 %0, [%1];" : "=h"(v) : "l"(p) : "memory");
  return v;
}

__device__ __forceinline__ void st_relaxed_u16(uint16_t* p, uint16_t v) {
  asm volatile("st.relaxed.gpu.global.u16 [%0], %1;" ::"l"(p), "h"(v) : "memory");
}

__device__ __forceinline__ void st_relaxed(uint32_t* p, uint32_t v) {
  asm volatile("st.relaxed.gpu.global.u32 [%0], %1;" ::"l"(p), "r"(v) : "memory");
}

__device__ __forceinline__ uint64_t global_ns() {
  uint64_t t;
  asm volatile("mov.u64 %0, %%globaltimer;" : "=l"(t));
  return t;
}

__device__ __forceinline__ uint32_t lanemask_lt() {
  uint32_t m;
  asm("mov.u32 %0, %%lanemask_lt;" : "=r"(m));
  return m;
}

template <class K>
__device__ __forceinline__ uint32_t digit_of(K key, uint32_t shift, uint32_t mask) {
  return static_cast<uint32_t>(key >> shift) & mask;
}

// Record the first device-side error of a call (later ones are dropped).
__device__ __forceinline__ void report_error(Ctrl* ctrl, uint32_t code, uint32_t info) {
  if (atomicCAS(&ctrl->error, 0u, code) == 0u) atomicExch(&ctrl->error_info, info);
}

// Per-call record read by rs_workspace_stats: the shape of the sort and the
// %globaltimer start of its first kernel (one thread), then times relative
// to that start, at least 1 so that 0 means "not reached".
__device__ __forceinline__ void stat_begin(Ctrl* ctrl, uint32_t n, uint32_t shape) {
  const uint64_t t = global_ns();
  ctrl->t0_lo = uint32_t(t);
  ctrl->t0_hi = uint32_t(t >> 32);
  ctrl->stat_n = n;
  ctrl->stat_shape = shape;
}

// The forms that do not start from a cleared control block clear the
// record's times themselves (one thread, before any other writes them).
__device__ __forceinline__ void stat_clear_times(Ctrl* ctrl) {
  ctrl->t_upsweep = 0u;
#pragma unroll
  for (int p = 0; p < kMaxPasses; ++p) ctrl->t_pass[p][0] = ctrl->t_pass[p][1] = 0u;
}

__device__ __forceinline__ uint32_t stat_now(const Ctrl* ctrl) {
  const uint64_t t0 = (uint64_t(ctrl->t0_hi) << 32) | ctrl->t0_lo;
  const uint64_t d = global_ns() - t0;
  return d >= 0xffffffffull ? 0xffffffffu : (d == 0 ? 1u : uint32_t(d));
}

// Programmatic dependent launch.  A kernel launched with programmatic stream
// serialization may start while the kernel before it on the stream is still
// running; pdl_wait() blocks (in hardware) until that kernel has completed and
// its memory operations are visible, and is a no-op for an ordinary launch.
// pdl_launch_dependents() lets the next such kernel be scheduled once every
// CTA of this grid has called it or exited.
__device__ __forceinline__ void pdl_wait() {
  asm volatile("griddepcontrol.wait;" ::: "memory");
}

__device__ __forceinline__ void pdl_launch_dependents() {
  asm volatile("griddepcontrol.launch_dependents;" ::: "memory");
}

__device__ __forceinline__ uint32_t ld_acquire(const uint32_t* p) {
  uint32_t v;
  asm volatile("ld.acquire.gpu.global.u32 %0, [%1];" : "=r"(v) : "l"(p) : "memory");
  return v;
}

// Bounded wait until *p >= target.  False when it ran out or another CTA
// already reported an error.
__device__ __noinline__ static bool wait_geq(const uint32_t* p, uint32_t target, Ctrl* ctrl,
                                             uint64_t timeout_ns, uint32_t info) {
  if (ld_acquire(p) >= target) return true;
  const uint64_t t0 = global_ns();
  for (uint32_t it = 1;; ++it) {
    if (ld_acquire(p) >= target) return true;
    if ((it & 63u) == 0u) {
      if (ld_relaxed(&ctrl->error) != 0u) return false;
      if (global_ns() - t0 > timeout_ns) {
        report_error(ctrl, kDevTimeout, info);
        return false;
      }
    }
  }
}


__device__ __forceinline__ uint32_t warp_inclusive_scan(uint32_t x, int lane) {
#pragma unroll
  for (int off = 1; off < 32; off <<= 1) {
    uint32_t y = __shfl_up_sync(kFull, x, off);
    if (lane >= off) x += y;
  }
  return x;
}

// Exclusive scan of one value per thread across the CTA.  s_tot holds 32
// words.  Every thread must call it; the caller separates two calls with a
// barrier.
template <int THREADS>
__device__ __forceinline__ uint32_t block_exclusive_scan(uint32_t x, uint32_t* s_tot) {
  constexpr int WARPS = THREADS / 32;
  const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
  const uint32_t inc = warp_inclusive_scan(x, lane);
  if (lane == 31) s_tot[warp] = inc;
  __syncthreads();
  if (warp == 0) {
    const uint32_t t = lane < WARPS ? s_tot[lane] : 0u;
    const uint32_t ti = warp_inclusive_scan(t, lane);
    s_tot[lane] = ti - t;
  }
  __syncthreads();
  return inc - x + s_tot[warp];
}

// --------------------------------------------------------------- upsweep

// Digit histograms of every pass in one read of the keys, then (last CTA)
// the exclusive scan of each and the set of passes that move data.
//
// Shared counters are laid out [pass][digit][slot] with slot = lane mod
// SLOTS: with 32 slots (32-bit keys) lane l only ever touches bank l, so a
// warp's 32 increments never meet on a bank whatever the digits are (the zero
// and sorted distributions included).  64-bit keys have twice the passes and
// use 16 slots to stay within shared memory.  FULL: the bit range is the whole
// key and r = 8, so every digit is one byte, taken with a byte permute.
//
// COPY: keys_to (and vals_to, if given) receive a copy of the keys (and values):
// a sort of an odd number of passes whose result has to end where its input
// was starts from the copy.  The counting is bound by its shared-memory
// atomics and leaves the memory idle, and the first pass finds much of the
// copy in the L2: 10,000,019 pairs of 32 bits over 20 bits take 152 us where
// the result may end anywhere, 168 with the copy, 188 when copied back after
// the passes.  A switch of its own, since a run-time test of it in the loop
// cost the sorts that copy nothing 4 to 6 us at that size.
template <class K, int RADIX_BITS, int THREADS, int MAXP, bool FULL, bool COPY>
__global__ void __launch_bounds__(THREADS, 1)
    k_upsweep(const K* __restrict__ keys, uint32_t n, int begin_bit, int end_bit, int passes,
              uint32_t* __restrict__ counts, uint32_t* __restrict__ offsets,
              Ctrl* __restrict__ ctrl, uint4* __restrict__ zero_base, uint64_t zero_vec4,
              KeyXf<K> xf, bool early_dependents, uint32_t shape, K* __restrict__ keys_to,
              const K* __restrict__ vals, K* __restrict__ vals_to) {
  constexpr int RADIX = 1 << RADIX_BITS;
  constexpr int SLOTS = sizeof(K) == 4 ? 32 : 16;
  constexpr int VEC = 16 / int(sizeof(K));
  constexpr int UNROLL = 4;
  static_assert(THREADS == 1024 && RADIX % 32 == 0, "32 warps' sums, whole warps per pass");
  static_assert(!FULL || RADIX_BITS == 8, "byte digits");

  extern __shared__ uint32_t sh[];  // [passes][RADIX][SLOTS]
  __shared__ uint32_t s_tot[32];
  __shared__ uint32_t s_one;
  __shared__ int s_last;
  // a first pass that fills the GPU may be scheduled beside this grid (one
  // that does not is scheduled as this grid's CTAs exit)
  if (early_dependents) pdl_launch_dependents();

  const int tid = threadIdx.x, lane = tid & 31;
  if (shape != 0u && blockIdx.x == 0 && tid == 0) stat_begin(ctrl, n, shape);
  const uint32_t slot = uint32_t(lane & (SLOTS - 1));
  uint32_t shiftp[MAXP], maskp[MAXP];
#pragma unroll
  for (int p = 0; p < MAXP; ++p) {
    const int lo = begin_bit + p * RADIX_BITS;
    const int hi = min(lo + RADIX_BITS, end_bit);
    shiftp[p] = p < passes ? uint32_t(lo) : 0u;
    maskp[p] = p < passes ? ((1u << (hi - lo)) - 1u) : 0u;
  }
  const int words = passes * RADIX * SLOTS;
  for (int i = tid; i < words; i += THREADS) sh[i] = 0u;
  __syncthreads();

  // XF: the digits are those of the transformed key (a compile-time switch,
  // so that plain unsigned sorts pay nothing for it)
  auto count_key = [&](K k, auto XF) {
    if constexpr (decltype(XF)::value) k = xf_fwd(k, xf);
#pragma unroll
    for (int p = 0; p < MAXP; ++p) {
      if (FULL || p < passes) {
        uint32_t d;
        if constexpr (FULL) {
          const uint32_t half = (sizeof(K) == 8 && p >= 4) ? uint32_t(uint64_t(k) >> 32)
                                                           : uint32_t(k);
          d = __byte_perm(half, 0u, 0x4440u | uint32_t(p & 3));
        } else {
          d = digit_of(k, shiftp[p], maskp[p]);
        }
        atomicAdd(&sh[(p * RADIX + int(d)) * SLOTS + int(slot)], 1u);
      }
    }
  };

  // 16-byte aligned body, scalar head and tail
  const uintptr_t addr = reinterpret_cast<uintptr_t>(keys);
  uint32_t head = uint32_t(((16u - (addr & 15u)) & 15u) / sizeof(K));
  if (head > n) head = n;
  const uint32_t nvec = (n - head) / VEC;
  const uint32_t tail = head + nvec * VEC;
  const uint4* vp = reinterpret_cast<const uint4*>(keys + head);
  const uint32_t stride = gridDim.x * THREADS;
  // copying whole vectors takes the two buffers equally aligned
  const bool kvec = COPY && ((addr ^ reinterpret_cast<uintptr_t>(keys_to)) & 15u) == 0u;
  if constexpr (COPY) {
    if (vals_to != nullptr) {
      const uintptr_t va = reinterpret_cast<uintptr_t>(vals);
      uint32_t done = 0u;  // elements before the scalar rest
      if (((va ^ reinterpret_cast<uintptr_t>(vals_to)) & 15u) == 0u) {
        const uint32_t vhead = min(uint32_t(((16u - (va & 15u)) & 15u) / sizeof(K)), n);
        const uint32_t nv = (n - vhead) / VEC;
        if (blockIdx.x == 0 && uint32_t(tid) < vhead && dbg_ok(tid, n, kSiteCopyVals))
          vals_to[tid] = vals[tid];
        const uint4* src = reinterpret_cast<const uint4*>(vals + vhead);
        uint4* dst = reinterpret_cast<uint4*>(vals_to + vhead);
        for (uint32_t base = blockIdx.x * THREADS + tid; base < nv; base += stride * UNROLL) {
          uint4 buf[UNROLL];
#pragma unroll
          for (int u = 0; u < UNROLL; ++u)
            if (base + uint32_t(u) * stride < nv) buf[u] = src[base + uint32_t(u) * stride];
#pragma unroll
          for (int u = 0; u < UNROLL; ++u)
            if (base + uint32_t(u) * stride < nv &&
                dbg_ok(vhead + uint64_t(base + uint32_t(u) * stride) * VEC + (VEC - 1), n,
                       kSiteCopyVals))
              dst[base + uint32_t(u) * stride] = buf[u];
        }
        done = vhead + nv * VEC;
      }
      for (uint32_t i = done + blockIdx.x * THREADS + tid; i < n; i += stride)
        if (dbg_ok(i, n, kSiteCopyVals)) vals_to[i] = vals[i];
    }
  }
  auto count_all = [&](auto XF) {
    if (blockIdx.x == 0) {
      if (uint32_t(tid) < head) {
        count_key(keys[tid], XF);
        if constexpr (COPY)
          if (dbg_ok(tid, n, kSiteCopyKeys)) keys_to[tid] = keys[tid];
      }
      if (uint32_t(tid) < n - tail) {
        count_key(keys[tail + tid], XF);
        if constexpr (COPY)
          if (dbg_ok(tail + tid, n, kSiteCopyKeys)) keys_to[tail + tid] = keys[tail + tid];
      }
    }
    for (uint32_t base = blockIdx.x * THREADS + tid; base < nvec; base += stride * UNROLL) {
      uint4 buf[UNROLL];
#pragma unroll
      for (int u = 0; u < UNROLL; ++u) {
        const uint32_t i = base + uint32_t(u) * stride;
        if (i < nvec) buf[u] = vp[i];
      }
#pragma unroll
      for (int u = 0; u < UNROLL; ++u) {
        const uint32_t i = base + uint32_t(u) * stride;
        if (i < nvec) {
          const K* ks = reinterpret_cast<const K*>(&buf[u]);
          if constexpr (COPY) {
            const bool in = dbg_ok(head + uint64_t(i) * VEC + (VEC - 1), n, kSiteCopyKeys);
            if (in && kvec) {
              reinterpret_cast<uint4*>(keys_to + head)[i] = buf[u];
            } else if (in) {
#pragma unroll
              for (int e = 0; e < VEC; ++e) keys_to[head + i * VEC + e] = ks[e];
            }
          }
#pragma unroll
          for (int e = 0; e < VEC; ++e) count_key(ks[e], XF);
        }
      }
    }
  };
  if (xf.on)
    count_all(std::true_type{});
  else
    count_all(std::false_type{});
  __syncthreads();
  // drain: one (pass, digit) per thread, summed over its slots
  for (int w = tid; w < passes * RADIX; w += THREADS) {
    const uint32_t* row = sh + w * SLOTS;
    uint32_t c = 0u;
#pragma unroll 8
    for (int l = 0; l < SLOTS; ++l) c += row[(l + lane) & (SLOTS - 1)];  // rotated: no bank conflicts
    if (c && dbg_ok(w, uint64_t(passes) * RADIX, kSiteUpCounts)) atomicAdd(&counts[w], c);
  }

  // clear the look-back status words of every pass of this call
  for (uint64_t i = uint64_t(blockIdx.x) * THREADS + tid; i < zero_vec4; i += stride)
    if (dbg_ok(i, zero_vec4, kSiteUpClear)) zero_base[i] = make_uint4(0u, 0u, 0u, 0u);

  // last CTA: scan each histogram, choose the passes that move data
  __threadfence();
  __syncthreads();
  if (tid == 0) s_last = (atomicAdd(&ctrl->hist_ticket, 1u) == gridDim.x - 1u);
  __syncthreads();
  if (!s_last) return;
  __threadfence();
  // THREADS / RADIX passes at a time, one digit a thread (one pass after
  // another, each with its own round trip to the L2 and its own barriers, this
  // took 4.5 of 12 us for 2^20 32-bit keys, twice that for 64-bit ones)
  constexpr int PER = THREADS / RADIX, ROUNDS = (MAXP + PER - 1) / PER;
  const int warp = tid >> 5, pq = tid / RADIX, dq = tid % RADIX;
  const int w0 = warp / (RADIX / 32) * (RADIX / 32);  // my pass's first warp
  uint32_t c[ROUNDS];
#pragma unroll
  for (int q = 0; q < ROUNDS; ++q)
    c[q] = q * PER + pq < passes ? ld_relaxed(&counts[(q * PER + pq) * RADIX + dq]) : 0u;
  if (tid == 0) s_one = 0u;
#pragma unroll
  for (int q = 0; q < ROUNDS; ++q) {
    const int p = q * PER + pq;
    const uint32_t inc = warp_inclusive_scan(c[q], lane);
    __syncthreads();  // s_one is clear; the round before has read s_tot
    if (lane == 31) s_tot[warp] = inc;
    // a pass in which one digit value holds every key leaves the order as it is
    if (p < passes && c[q] == n) atomicOr(&s_one, 1u << p);
    __syncthreads();
    const uint32_t start =
        __reduce_add_sync(kFull, lane >= w0 && lane < warp ? s_tot[lane] : 0u) + inc - c[q];
    if (p < passes && dbg_ok(uint64_t(p) * RADIX + dq, uint64_t(passes) * RADIX, kSiteUpOffsets))
      offsets[p * RADIX + dq] = start;
  }
  uint32_t exec = ~s_one & ((1u << passes) - 1u);
  if (tid == 0) {
    // the sorted data must end in the buffer the host named (pass count
    // parity): if skipping changed the parity, the lowest skipped pass runs
    if ((__popc(exec) & 1) != (passes & 1)) {
      const uint32_t skipped = ~exec & ((1u << passes) - 1u);
      exec |= skipped & (0u - skipped);
    }
    ctrl->exec_mask = exec;
    if (shape != 0u) ctrl->t_upsweep = stat_now(ctrl);
  }
}

// -------------------------------------------------------------- onesweep

// Words of the zero source of the counter-clearing bulk copies: the counters
// of up to 16 warps x 256 digits.
constexpr int kZeroWords = 4096;

// INDEX: the stage holds 16-bit tile slots, and keys and values stay in the
// buffers they were loaded into until the scatter gathers them (10 bytes of
// shared memory for a 32-bit pair).  Otherwise (keys only) it holds the keys,
// and the next tile's keys can land in the key buffer from then on.
template <class K, int VB, int RADIX_BITS, int THREADS, int ITEMS, bool INDEX>
struct OnesweepSmem {
  static constexpr int RADIX = 1 << RADIX_BITS;
  static constexpr int WARPS = THREADS / 32;
  static constexpr int TILE = THREADS * ITEMS;
  static constexpr int WH = 0;                             // u32 [WARPS][RADIX] warp counters
  // the counters are cleared by a bulk copy with each tile's keys
  static constexpr uint32_t ZERO_BYTES = uint32_t(WARPS * RADIX * 4);
  static_assert(ZERO_BYTES <= kZeroWords * 4 && ZERO_BYTES % 16 == 0, "one bulk copy of zeros");
  static constexpr int GBASE = WH + WARPS * RADIX * 4;     // u32 [RADIX] global base
  static constexpr int TOT = GBASE + RADIX * 4;            // u32 [32]
  static constexpr int MISC = TOT + 32 * 4;                // u32 [8]: [0] tile, [2] error,
                                                           // [3] next tile, [5..6] check sums
  static constexpr int MBAR = MISC + 32;                   // u64 [2] mbarriers: keys, values
  static constexpr int ARGS = MBAR + 16;                   // TileArgs
  static constexpr int KIN = ARGS + 208;   // the tile's keys as loaded (+16 B skew)
  static constexpr int VIN = KIN + TILE * int(sizeof(K)) + 16;    // the tile's values as loaded
  static constexpr int OUT = VIN + (VB > 0 ? TILE * VB + 16 : 0); // the stage and an end mark
  static constexpr int BYTES = OUT + (INDEX ? (TILE + 8) * 2 : (TILE + 2) * int(sizeof(K)));
};

// Operands of the tiles of one digit pass over one array (or one segment).
// They lie in shared memory (written by one thread before a barrier): held in
// registers over the resident CTAs' loop, they and what the compiler derives
// from them cost up to 60 registers a thread, most of them spilled.
template <class K, int VB>
struct TileArgs {
  const K* ksrc;
  K* kdst;
  const ValT<VB>* vsrc;
  ValT<VB>* vdst;
  const uint32_t* pass_offsets; // [RADIX] global digit offsets of this pass
  // look-back words of this pass.  Whole arrays: status u16 [tiles][RADIX],
  // gagg [groups][RADIX], sagg and sinc [supers][RADIX].  Segments: status u32
  // [tiles/4][RADIX][4] alone.
  uint32_t *status, *gagg, *sagg, *sinc;
  uint64_t lb_words;            // words in status (debug bounds checks only)
  uint64_t g_words, s_words;    // words in gagg; in sagg and in sinc (the same)
  uint64_t* trace;              // test-only: [tiles][16] phase stamps and counters, or null
  KeyXf<K> xf;                  // order-preserving key transform of the sort
  uint32_t n;                   // elements of the array / segment
  uint32_t shift, mask;         // digit of this pass: (key >> shift) & mask
  uint32_t tile0;               // index of this array's tile 0 in status (a segment's first tile)
  uint32_t trace_tiles;         // test-only: tiles the trace holds
  int32_t drop_tile;            // test-only: this tile publishes nothing (-1: none)
  int32_t bad_tile;             // debug builds, test-only: this tile's scatter indices are
                                // pushed past n (-1: none)
  OrderTest order;              // test-only
  bool xin;                     // the source holds untransformed keys: apply xf on load
  bool xout;                    // write untransformed keys (apply xf's inverse)
};

// debug builds, one thread (in release builds the count cost the 1024-thread
// CTA sorts 4-12 bytes of spills and up to 5 %)
__device__ __forceinline__ void count_repair(const OrderTest& order) {
  if constexpr (kDebugChecks) {
    if (order.repairs != nullptr) atomicAdd(order.repairs, 1u);
  }
}

__device__ __forceinline__ uint32_t sm_id() {
  uint32_t r;
  asm volatile("mov.u32 %0, %%smid;" : "=r"(r));
  return r;
}

// test-only phase stamp (thread 0)
__device__ __forceinline__ void stamp(uint64_t* tr, int k) {
  if (tr != nullptr && threadIdx.x == 0) tr[k] = global_ns();
}

// test-only counters of digit 0's look-back (thread 0)
__device__ __forceinline__ void trace_add(uint64_t* tr, int k, uint64_t v) {
  if (tr != nullptr && threadIdx.x == 0) tr[k] += v;
}

// The look-back of one digit (one thread): the sum of the counts of the
// earlier tiles, in steps that a caller can put between other work.  issue()
// starts the L2 loads, consume() adds what has arrived; finish() does both
// until nothing is missing, every wait without progress bounded.
//
// Whole arrays: every tile adds its counts to its group's (8 tiles) and its
// super's (64 tiles) when it publishes them, so the sum is at most 7 tiles, 7
// groups and the earlier supers, nearest first: complete counts (go on) or an
// inclusive prefix (stop; the last tile of each super publishes it).  All
// levels are fetched at once, 18 words a thread at most, a warp's 32 digits
// side by side.  Under load such a round trip takes 1-2 us, and how many
// follow one another is what a look-back costs: a walk over groups of 32
// tiles, 8 tiles at a time, took 3.8 of them a tile (5.9 of its 10.5 us, keys
// alone at 2^26); this one takes 1.4 to 1.7, the first under the stage, and
// leaves 2.5 of 9.5 us.  What is left waits for tiles in flight: windows of 4
// and 6 supers (1.04 round trips) took u32 pairs from 1.012 to 1.057 and
// 1.088 ms, for their words.
template <class K, int VB, int RADIX>
struct TreeLookBack {
  uint32_t excl = 0u;
  uint32_t missing = 0u;        // bit l: level l (tiles, groups, supers) is not summed yet
  uint32_t at_tile = 0u;
  int32_t super = -1;           // the next super to add
  uint32_t w[kGroupTiles - 1], g[kSuperGroups - 1], agg[2], inc[2];

  __device__ __forceinline__ void start(const TileArgs<K, VB>&, uint32_t tile) {
    at_tile = tile;
    super = int32_t(tile / kSuperTiles) - 1;
    missing = (tile % kGroupTiles ? 1u : 0u) | (tile / kGroupTiles % kSuperGroups ? 2u : 0u) |
              (super >= 0 ? 4u : 0u);
  }

  __device__ __forceinline__ bool done() const { return missing == 0u; }

  __device__ __forceinline__ void issue(const TileArgs<K, VB>& t, uint32_t d) {
    if (missing & 1u) {
      const uint16_t* p = reinterpret_cast<const uint16_t*>(t.status) +
                          size_t(at_tile / kGroupTiles * kGroupTiles) * RADIX + d;
#pragma unroll
      for (uint32_t c = 0; c < kGroupTiles - 1; ++c)
        if (c < at_tile % kGroupTiles) w[c] = ld_relaxed_u16(p + c * RADIX);
    }
    if (missing & 2u) {
      const uint32_t* p = t.gagg + size_t(at_tile / kSuperTiles * kSuperGroups) * RADIX + d;
#pragma unroll
      for (uint32_t c = 0; c < kSuperGroups - 1; ++c)
        if (c < at_tile / kGroupTiles % kSuperGroups) g[c] = ld_relaxed(p + c * RADIX);
    }
    if (missing & 4u) {
#pragma unroll
      for (int c = 0; c < 2; ++c)
        if (super >= c) {
          agg[c] = ld_relaxed(t.sagg + size_t(super - c) * RADIX + d);
          inc[c] = ld_relaxed(t.sinc + size_t(super - c) * RADIX + d);
        }
    }
  }

  __device__ __forceinline__ void consume(uint64_t* tr) {
    if (missing != 0u) trace_add(tr, 10, 1);
    if (missing & 1u) {
      uint32_t sum = 0u, all = kTilePublished;
#pragma unroll
      for (uint32_t c = 0; c < kGroupTiles - 1; ++c)
        if (c < at_tile % kGroupTiles) {
          sum += w[c] & ~kTilePublished;
          all &= w[c];
        }
      if (all) {
        excl += sum;
        missing &= ~1u;
      }
    }
    if (missing & 2u) {
      uint32_t sum = 0u;
      bool whole = true;
#pragma unroll
      for (uint32_t c = 0; c < kSuperGroups - 1; ++c)
        if (c < at_tile / kGroupTiles % kSuperGroups) {
          sum += g[c] & kGroupCountMask;
          whole = whole && (g[c] >> 24) == uint32_t(kGroupTiles);
        }
      if (whole) {
        excl += sum;
        missing &= ~2u;
      }
    }
    if (missing & 4u) {
      const int32_t s0 = super;
#pragma unroll
      for (int c = 0; c < 2; ++c) {
        if (super != s0 - c || super < 0 || !(missing & 4u)) continue;
        if (inc[c] & kFlagMask) {
          excl += inc[c] & kValueMask;
          missing &= ~4u;
        } else if ((agg[c] >> 24) == uint32_t(kSuperTiles)) {
          excl += agg[c] & kGroupCountMask;
          --super;
        }
      }
      if (super < 0) missing &= ~4u;  // every super summed
    }
  }

  __device__ __forceinline__ bool finish(const TileArgs<K, VB>& t, uint32_t d, Ctrl* ctrl,
                                         uint64_t timeout_ns, uint32_t tile, uint64_t* tr) {
    uint64_t t0 = 0;
    for (uint32_t idle = 0; missing != 0u;) {
      const uint32_t m0 = missing;
      const int32_t s0 = super;
      issue(t, d);
      consume(tr);
      if (missing != m0 || super != s0) {
        idle = 0;
        continue;
      }
      trace_add(tr, 12, 1);
      if (idle == 0) t0 = global_ns();
      if ((++idle & 63u) == 0u) {
        if (ld_relaxed(&ctrl->error) != 0u) return false;
        if (global_ns() - t0 > timeout_ns) {
          report_error(ctrl, kDevTimeout, tile);
          return false;
        }
      }
    }
    return true;
  }
};

// Segments: a walk over the segment's tiles, nearest first, 8 at a time, down
// to an inclusive prefix (every tile publishes its own once it has it).
template <class K, int VB, int RADIX>
struct FlatLookBack {
  uint32_t excl = 0u;
  int32_t at = -1, lo = 0;  // next tile to add; the segment's first
  uint4 w[2];

  __device__ __forceinline__ void start(const TileArgs<K, VB>& t, uint32_t tile) {
    lo = int32_t(t.tile0);
    at = tile ? lo + int32_t(tile) - 1 : lo - 1;
  }

  __device__ __forceinline__ bool done() const { return at < lo; }

  __device__ __forceinline__ void issue(const TileArgs<K, VB>& t, uint32_t d) {
    if (done()) return;
#pragma unroll
    for (int k = 0; k < 2; ++k) {
      const int32_t b = (at >> 2) - k;
      w[k] = 4 * b + 3 >= lo ? ld_relaxed_v4(t.status + (size_t(b) * RADIX + d) * 4)
                             : make_uint4(0u, 0u, 0u, 0u);
    }
  }

  __device__ __forceinline__ void consume(uint64_t* tr) {
    if (done()) return;
    trace_add(tr, 10, 1);
    const int32_t b0 = at >> 2;
    bool go = true;
#pragma unroll
    for (int k = 0; k < 2; ++k) {
#pragma unroll
      for (int c = 3; c >= 0; --c) {
        if (!go || 4 * (b0 - k) + c != at || at < lo) continue;
        const uint32_t sw = c == 0 ? w[k].x : c == 1 ? w[k].y : c == 2 ? w[k].z : w[k].w;
        const uint32_t f = sw & kFlagMask;
        if (f == 0u) {
          go = false;
        } else {
          excl += sw & kValueMask;
          at = f == kFlagInc ? lo - 1 : at - 1;
          go = f != kFlagInc;
        }
      }
    }
  }

  __device__ __forceinline__ bool finish(const TileArgs<K, VB>& t, uint32_t d, Ctrl* ctrl,
                                         uint64_t timeout_ns, uint32_t tile, uint64_t* tr) {
    uint64_t t0 = 0;
    for (uint32_t idle = 0; !done();) {
      const int32_t at0 = at;
      issue(t, d);
      consume(tr);
      if (at != at0) {
        idle = 0;
        continue;
      }
      trace_add(tr, 12, 1);
      if (idle == 0) t0 = global_ns();
      if ((++idle & 63u) == 0u) {
        if (ld_relaxed(&ctrl->error) != 0u) return false;
        if (global_ns() - t0 > timeout_ns) {
          report_error(ctrl, kDevTimeout, tile);
          return false;
        }
      }
    }
    return true;
  }
};

// ---- bulk (TMA engine) copies global -> shared, completed on an mbarrier

__device__ __forceinline__ uint32_t smem_u32(const void* p) {
  return static_cast<uint32_t>(__cvta_generic_to_shared(p));
}

__device__ __forceinline__ void mbar_init(uint64_t* bar) {
  asm volatile("mbarrier.init.shared::cta.b64 [%0], 1;" ::"r"(smem_u32(bar)) : "memory");
  asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
}

// Before the barrier's shared memory is used for anything else.
__device__ __forceinline__ void mbar_inval(uint64_t* bar) {
  asm volatile("mbarrier.inval.shared::cta.b64 [%0];" ::"r"(smem_u32(bar)) : "memory");
}

__device__ __forceinline__ void mbar_arrive_expect_tx(uint64_t* bar, uint32_t bytes) {
  asm volatile("mbarrier.arrive.expect_tx.shared::cta.b64 _, [%0], %1;" ::"r"(smem_u32(bar)),
               "r"(bytes)
               : "memory");
}

__device__ __forceinline__ bool mbar_try_wait(uint64_t* bar, uint32_t parity) {
  uint32_t ok;
  asm volatile(
      "{\n\t.reg .pred p;\n\t"
      "mbarrier.try_wait.parity.shared::cta.b64 p, [%1], %2;\n\t"
      "selp.u32 %0, 1, 0, p;\n\t}"
      : "=r"(ok)
      : "r"(smem_u32(bar)), "r"(parity)
      : "memory");
  return ok != 0u;
}

// dst and src 16-byte aligned, bytes a multiple of 16
__device__ __forceinline__ void bulk_load(void* dst, const void* src, uint32_t bytes,
                                          uint64_t* bar) {
  asm volatile(
      "cp.async.bulk.shared::cluster.global.mbarrier::complete_tx::bytes [%0], [%1], %2, [%3];"
      ::"r"(smem_u32(dst)), "l"(src), "r"(bytes), "r"(smem_u32(bar))
      : "memory");
}

// Bounded wait for phase `parity` of the tile-load barrier.  False when the
// limit ran out (the error is recorded); in that case the caller waits once
// more, again bounded, so that no copy is still landing when it leaves.
__device__ __noinline__ static bool mbar_wait_bounded(uint64_t* bar, uint32_t parity,
                                                      Ctrl* ctrl, uint64_t timeout_ns,
                                                      uint32_t info) {
  if (mbar_try_wait(bar, parity)) return true;
  const uint64_t t0 = global_ns();
  for (;;) {
    if (mbar_try_wait(bar, parity)) return true;
    if (global_ns() - t0 > timeout_ns) {
      report_error(ctrl, kDevTimeout, info);
      return false;
    }
  }
}

// The same with the first try in line: a call's saved registers then cost
// only the waits that need it.
__device__ __forceinline__ bool mbar_wait(uint64_t* bar, uint32_t parity, Ctrl* ctrl,
                                          uint64_t timeout_ns, uint32_t info) {
  return mbar_try_wait(bar, parity) || mbar_wait_bounded(bar, parity, ctrl, timeout_ns, info) ||
         mbar_wait_bounded(bar, parity, ctrl, timeout_ns, info);
}

// Shared-memory staging of elements [0, len) of src: element i lands at byte
// (skew + i * sizeof(T)) of `buf`, skew = src address mod 16, so that the
// 16-byte aligned middle ("body") goes by one bulk copy while the few head
// and tail elements are loaded by threads.
template <class T>
struct Stage {
  uint32_t skew, head, body, head_n, tail0;
  __device__ __forceinline__ Stage(const T* src, uint32_t len) {
    skew = uint32_t(reinterpret_cast<uintptr_t>(src) & 15u);
    const uint32_t bytes = len * uint32_t(sizeof(T));
    head = (16u - skew) & 15u;
    if (head > bytes) head = bytes;
    body = (bytes - head) & ~15u;
    head_n = head / uint32_t(sizeof(T));
    tail0 = (head + body) / uint32_t(sizeof(T));
  }
  __device__ __forceinline__ T* at(unsigned char* buf) const {
    return reinterpret_cast<T*>(buf + skew);
  }
  // thread 0 only
  __device__ __forceinline__ void issue(unsigned char* buf, const T* src, uint64_t* bar) const {
    if (body)
      bulk_load(buf + skew + head, reinterpret_cast<const unsigned char*>(src) + head, body, bar);
  }
  // every thread; L2 loads, since other CTAs of the same kernel may have
  // written the source
  __device__ __forceinline__ void edges(unsigned char* buf, const T* src, uint32_t len) const {
    T* s = at(buf);
    const uint32_t tid = threadIdx.x;
    if (tid < head_n) s[tid] = __ldcg(src + tid);
    if (tid < len - tail0) s[tail0 + tid] = __ldcg(src + tail0 + tid);
  }
};

// Zeros in global memory, the source of the bulk copies that clear the rank
// counters of a tile (one copy per TU; never written).
namespace {
__device__ __align__(128) uint32_t g_zero_words[kZeroWords];
}

// Start staging the keys of tile `tile` of an array of n keys into the key
// buffer: one bulk copy issued by thread 0 on `bar`, head and tail elements
// loaded by the other threads.  zero_dst (optional):
// zero_bytes (a multiple of 16, at most kZeroWords words) of shared memory cleared by a
// second bulk copy on the same barrier, so that the tile's counters are zero
// once its keys have landed, without a store loop on the shared-memory pipe.
template <class K, int THREADS, int TILE, bool CG>
__device__ __forceinline__ void stage_keys(unsigned char* kin, const K* ksrc, uint32_t n,
                                           uint32_t tile, uint64_t* bar,
                                           void* zero_dst = nullptr, uint32_t zero_bytes = 0u) {
  const uint32_t tile_base = tile * uint32_t(TILE);
  const uint32_t tile_len = min(uint32_t(TILE), n - tile_base);
  const K* gk = ksrc + tile_base;
  const Stage<K> sk(gk, tile_len);
  if (threadIdx.x == 0) {
    // shared memory this CTA used through ordinary loads and stores before is
    // about to be written by the copy engine; and, when the source was written
    // by other CTAs of this kernel, those stores must be ordered before the
    // copy engine reads them
    asm volatile("fence.proxy.async.shared::cta;" ::: "memory");
    if constexpr (CG) asm volatile("fence.proxy.async.global;" ::: "memory");
    mbar_arrive_expect_tx(bar, sk.body + zero_bytes);
    sk.issue(kin, gk, bar);
    if (zero_bytes) bulk_load(zero_dst, g_zero_words, zero_bytes, bar);
  }
  sk.edges(kin, gk, tile_len);
}

// Start loading tile `tile`'s keys and the cleared counters, on the keys'
// barrier.  Every thread of the CTA calls it.
template <class S, class K, int VB, int THREADS, bool CG>
__device__ __forceinline__ void stage_tile(unsigned char* smem, uint32_t tile) {
  const TileArgs<K, VB>& t = *reinterpret_cast<const TileArgs<K, VB>*>(smem + S::ARGS);
  stage_keys<K, THREADS, S::TILE, CG>(smem + S::KIN, t.ksrc, t.n, tile,
                                      reinterpret_cast<uint64_t*>(smem + S::MBAR), smem + S::WH,
                                      S::ZERO_BYTES);
}

// The same for its values, on theirs.
template <class S, class K, int VB, bool CG>
__device__ __forceinline__ void stage_values(unsigned char* smem, uint32_t tile) {
  const TileArgs<K, VB>& t = *reinterpret_cast<const TileArgs<K, VB>*>(smem + S::ARGS);
  uint64_t* s_bar = reinterpret_cast<uint64_t*>(smem + S::MBAR);
  const uint32_t base = tile * uint32_t(S::TILE);
  const uint32_t len = min(uint32_t(S::TILE), t.n - base);
  const ValT<VB>* gv = t.vsrc + base;
  const Stage<ValT<VB>> sv(gv, len);
  if (threadIdx.x == 0) {
    asm volatile("fence.proxy.async.shared::cta;" ::: "memory");
    if constexpr (CG) asm volatile("fence.proxy.async.global;" ::: "memory");
    mbar_arrive_expect_tx(&s_bar[1], sv.body);
    sv.issue(smem + S::VIN, gv, &s_bar[1]);
  }
  sv.edges(smem + S::VIN, gv, len);
}

// Persistent CTAs: where the next tile id comes from.
struct Prefetch {
  uint32_t* counter;  // the pass's tile counter
  uint32_t tiles;
};

// One tile of one counting-sort pass (Sec. 2.6), its operands at S::ARGS in
// shared memory.  Every thread of the CTA calls it.  Returns false
// (CTA-uniform) when a bounded wait gave up, in which case no copy into shared
// memory is pending.
//
//   1. count: every warp counts its keys' digits (shared atomics);
//   2. per digit, the sum over the warps is the tile's count, published at
//      once, before anything is ranked; the counters become the warps' first
//      slots in the tile;
//   3. stage, in (digit, input) order: each warp takes its keys item by item
//      and draws a slot from its counter of the key's digit (one returning
//      atomicAdd); into the slot goes the key itself, or (INDEX) its 16-bit
//      place in the tile.  The look-back's first round trip runs meanwhile;
//   4. the rest of the look-back, then the scatter in stage order: contiguous
//      stores inside each digit run.  With INDEX the keys are gathered from
//      the buffer they were loaded into, then the values from theirs.
//
// The order of equal digits inside one warp's atomicAdd is the hardware's: on
// sm_103a it went by lane in every pair measured (0.9e9), which is the input
// order, but nothing promises it.  So the scatter checks what it reads:
//   - INDEX: places ascend inside every digit run, i.e. the stage has no
//     descents but those at the starts of runs;
//   - keys (only sorts of whole keys, where no pass looks below or above the
//     key's bits): the bits up to this digit ascend over the whole stage.
//     Keys that agree in all of them need no order: later passes tell them
//     apart, or they are equal.
// A tile that fails is put in order, whatever order its draws took, and
// scattered again to the same destinations.
//
// What bounds it: the shared-memory pipe.  Each of the accesses by a random
// digit or slot costs 3.1-3.6 wavefronts a warp: the count, the draw, the
// stage store and (INDEX) the gathers.  A rank by peer masks (atomicOr, its
// load, the leader's store, then the offset's load) took two more and, item
// after item, a chain of three of them; the returning atomic ranks 2.58e12
// digits a second on the whole GPU, the masks 0.91e12 (random digits in
// registers; all 32 lanes on one digit: 0.297e12 and 0.267e12).  Measured at
// 2^26, a whole sort, before -> now, ms: u32 keys 1.09 -> 0.726, u32 pairs
// 1.31 -> 1.012, u64 keys 3.04 -> 2.285, u64 pairs 4.08 -> 3.51; pipe busy
// 68 % -> 76 % (u32 keys) and 80 % (u32 pairs) at 25.5 -> 16.8 and 29.6 ->
// 25.5 wavefronts per 32 elements.
//
// PERSIST: the calling kernel keeps the CTA resident over many tiles.  The
// barriers are initialised once by the kernel, this tile's keys were staged
// by the previous call (or the kernel's prologue) on barrier phase `parity`,
// and as soon as the key buffer is free (the keys staged, or with INDEX
// scattered: under the values' scatter) this call takes the next tile id
// (*next, at least pf->tiles when there is none) and starts loading it.
template <class K, int VB, int RADIX_BITS, int THREADS, int ITEMS, bool INDEX, bool CG,
          bool PERSIST = false, bool FLAT = false>
__device__ __forceinline__ bool onesweep_tile(uint32_t tile, Ctrl* ctrl, uint64_t timeout_ns,
                                              unsigned char* smem, uint32_t parity = 0u,
                                              const Prefetch* pf = nullptr,
                                              uint32_t* next = nullptr) {
  using V = ValT<VB>;
  using S = OnesweepSmem<K, VB, RADIX_BITS, THREADS, ITEMS, INDEX>;
  constexpr int RADIX = S::RADIX, WARPS = S::WARPS, TILE = S::TILE;
  static_assert(RADIX <= THREADS, "one thread per digit");
  static_assert(TILE < 1 << 15, "a tile's counts fit 15 bits, its slots 16");
  static_assert(INDEX || VB == 0, "values follow their keys' slots");
  uint32_t* s_wh = reinterpret_cast<uint32_t*>(smem + S::WH);
  uint32_t* s_gbase = reinterpret_cast<uint32_t*>(smem + S::GBASE);
  uint32_t* s_tot = reinterpret_cast<uint32_t*>(smem + S::TOT);
  uint32_t* s_misc = reinterpret_cast<uint32_t*>(smem + S::MISC);
  uint64_t* s_bar = reinterpret_cast<uint64_t*>(smem + S::MBAR);  // [0] keys, [1] values
  static_assert(sizeof(TileArgs<K, VB>) <= S::KIN - S::ARGS, "the operands' place");
  const TileArgs<K, VB>& t = *reinterpret_cast<const TileArgs<K, VB>*>(smem + S::ARGS);
  const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;

  const uint32_t tile_base = tile * uint32_t(TILE);
  const uint32_t tile_len = min(uint32_t(TILE), t.n - tile_base);
  const bool silent = int(tile) == t.drop_tile;
  auto trace = [&]() { return t.trace && tile < t.trace_tiles ? t.trace + size_t(tile) * 16 : nullptr; };
  stamp(trace(), 0);
  if (tid == 0 && trace()) trace()[7] = sm_id();

  if constexpr (!PERSIST) {
    if (tid == 0) {
      mbar_init(&s_bar[0]);
      if constexpr (VB > 0) mbar_init(&s_bar[1]);
    }
    __syncthreads();
    stage_tile<S, K, VB, THREADS, CG>(smem, tile);
    if constexpr (VB > 0) stage_values<S, K, VB, CG>(smem, tile);
  }
  const bool landed = mbar_wait(&s_bar[0], parity, ctrl, timeout_ns, tile);
  auto leave = [&](bool ok, bool values) {
    if constexpr (VB > 0) {  // the value copy must not land after this call
      if (!ok && values) {
        mbar_wait(&s_bar[1], parity, ctrl, timeout_ns, tile);
        __syncthreads();
      }
    }
    if constexpr (!PERSIST) {
      if (tid == 0) {
        mbar_inval(&s_bar[0]);
        if constexpr (VB > 0) mbar_inval(&s_bar[1]);
      }
    }
    return ok;
  };
  if (__syncthreads_or(!landed)) return leave(false, !PERSIST);  // CTA-uniform
  if constexpr (PERSIST && VB > 0) stage_values<S, K, VB, CG>(smem, tile);
  stamp(trace(), 1);

  // ---- 1. count.  Warp w owns tile slots [w*ITEMS*32, (w+1)*ITEMS*32); item j
  // of lane l is slot w*ITEMS*32 + j*32 + l.  mirror 1 (test-only): the lanes
  // are taken in reverse, so that every repeated digit draws out of turn.
  K* s_kin = Stage<K>(t.ksrc + tile_base, tile_len).at(smem + S::KIN);
  const uint32_t slot0 = uint32_t(warp * ITEMS * 32 + (t.order.mirror == 1 ? 31 - lane : lane));
  uint32_t* wh = s_wh + warp * RADIX;
  // a tile's keys are its first tile_len slots; the rest draw nothing
  const uint32_t lim = tile_len - min(slot0, tile_len);  // item j is a key if j * 32 < lim
  const bool full = tile_len == uint32_t(TILE);
  // until they are staged: the keys, or (INDEX) their digits, four a word
  K key[INDEX ? 1 : ITEMS];
  uint32_t dig[INDEX ? (ITEMS + 3) / 4 : 1];
  // in batches, so that a batch's loads, atomics and stores each go back to
  // back: one after another per item they would wait on one another.  Three
  // at a time where many tiles compete for the pipe (nine: u32 pairs at 2^26
  // 1.088 ms instead of 1.010, u64 pairs 3.68 instead of 3.46; one: 1.110 and
  // 3.45), nine to count and stage where a tile is alone on its SM (2^18 u32
  // keys 41.4 -> 39.6 us).
  constexpr int MOST = PERSIST ? 3 : 9;
  constexpr int BATCH = ITEMS < MOST ? ITEMS : MOST;
  constexpr int OUT_BATCH = ITEMS < 3 ? ITEMS : 3;
  auto count = [&](auto FULL) __attribute__((always_inline)) {
    const uint32_t shift = t.shift, mask = t.mask;
    const bool xin = t.xin;
    const KeyXf<K> xf = t.xf;
#pragma unroll
    for (int j0 = 0; j0 < ITEMS; j0 += BATCH) {
      K k[BATCH];
#pragma unroll
      for (int j = j0; j < ITEMS && j < j0 + BATCH; ++j) k[j - j0] = s_kin[slot0 + j * 32];
      if (xin) {  // the first pass that moves data: from here on the keys are transformed
#pragma unroll
        for (int j = j0; j < ITEMS && j < j0 + BATCH; ++j) {
          k[j - j0] = xf_fwd(k[j - j0], xf);
          if constexpr (INDEX) s_kin[slot0 + j * 32] = k[j - j0];
        }
      }
#pragma unroll
      for (int j = j0; j < ITEMS && j < j0 + BATCH; ++j) {
        const uint32_t d = digit_of(k[j - j0], shift, mask);
        if (decltype(FULL)::value || uint32_t(j * 32) < lim) atomicAdd(&wh[d], 1u);
        if constexpr (INDEX) dig[j / 4] = j % 4 ? dig[j / 4] | d << (8 * (j % 4)) : d;
        else key[j] = k[j - j0];
      }
    }
  };
  if (full)
    count(std::true_type{});
  else
    count(std::false_type{});
  if (INDEX && tid == 0) s_misc[5] = s_misc[6] = 0u;  // the check's sums, one a round
  __syncthreads();
  stamp(trace(), 2);

  // ---- 2. per digit: the tile's count, published; then the exclusive prefix
  // over the warps from the digit's first slot in the tile
  typename std::conditional<FLAT, FlatLookBack<K, VB, RADIX>, TreeLookBack<K, VB, RADIX>>::type lb;
  uint32_t my_cnt = 0u, off0 = 0u;
  uint32_t c[WARPS];
  if (tid < RADIX) {
#pragma unroll
    for (int w = 0; w < WARPS; ++w) {
      c[w] = s_wh[w * RADIX + tid];
      my_cnt += c[w];
    }
    if (!silent) {
      if constexpr (FLAT) {
        if (dbg_ok(lb_index<RADIX>(t.tile0 + tile, tid), t.lb_words, kSiteTileStatus))
          st_relaxed(&t.status[lb_index<RADIX>(t.tile0 + tile, tid)],
                     (tile == 0u ? kFlagInc : kFlagAgg) | my_cnt);
      } else {
        const size_t at = size_t(tile) * RADIX + tid;
        if (dbg_ok(at, t.lb_words, kSiteTileStatus))
          st_relaxed_u16(reinterpret_cast<uint16_t*>(t.status) + at,
                         uint16_t(kTilePublished | my_cnt));
        const size_t g = size_t(tile / kGroupTiles) * RADIX + tid;
        if (dbg_ok(g, t.g_words, kSiteGroupAgg)) atomicAdd(&t.gagg[g], my_cnt | kGroupOne);
        const size_t s = size_t(tile / kSuperTiles) * RADIX + tid;
        if (dbg_ok(s, t.s_words, kSiteGroupAgg)) atomicAdd(&t.sagg[s], my_cnt | kGroupOne);
      }
    }
    off0 = t.pass_offsets[tid];
  }
  const uint32_t inc = warp_inclusive_scan(my_cnt, lane);
  if (lane == 31) s_tot[warp] = inc;
  __syncthreads();
  const uint32_t my_start =
      __reduce_add_sync(kFull, lane < WARPS && lane < warp ? s_tot[lane] : 0u) + inc - my_cnt;
  if (tid < RADIX) {
    uint32_t run = my_start;
#pragma unroll
    for (int w = 0; w < WARPS; ++w) {
      s_wh[w * RADIX + tid] = run;
      run += c[w];
    }
    lb.start(t, tile);
  }
  __syncthreads();
  stamp(trace(), 3);

  // ---- 3. stage, the look-back in between
  K* s_out = reinterpret_cast<K*>(smem + S::OUT);
  uint16_t* s_idx = reinterpret_cast<uint16_t*>(smem + S::OUT);
  constexpr int LB_AT = ((ITEMS + BATCH - 1) / BATCH - 1) / 2;
  auto stage = [&](auto FULL) __attribute__((always_inline)) {
    [[maybe_unused]] const uint32_t shift = t.shift, mask = t.mask;
#pragma unroll
    for (int j0 = 0; j0 < ITEMS; j0 += BATCH) {
      uint32_t p[BATCH];
#pragma unroll
      for (int j = j0; j < ITEMS && j < j0 + BATCH; ++j) {
        uint32_t d;
        if constexpr (INDEX) d = dig[j / 4] >> (8 * (j % 4)) & 0xffu;
        else d = digit_of(key[j], shift, mask);
        p[j - j0] = 0u;
        if (decltype(FULL)::value || uint32_t(j * 32) < lim) p[j - j0] = atomicAdd(&wh[d], 1u);
      }
#pragma unroll
      for (int j = j0; j < ITEMS && j < j0 + BATCH; ++j) {
        if (decltype(FULL)::value || uint32_t(j * 32) < lim) {
          if constexpr (INDEX) s_idx[p[j - j0]] = uint16_t(slot0 + j * 32);
          else s_out[p[j - j0]] = key[j];
        }
      }
      // half-way, so that the tiles just before this one, which publish at
      // about the same time, mostly have
      if (j0 / BATCH == LB_AT && tid < RADIX) lb.issue(t, tid);
    }
  };
  if (full)
    stage(std::true_type{});
  else
    stage(std::false_type{});
  if constexpr (kDebugChecks) {
    if (t.order.mirror == 2) {  // test-only: as if each warp's draws had come last item first
      __syncthreads();
      if (tid < RADIX) {
        uint32_t at = my_start;
        for (int w = 0; w < WARPS; ++w) {
          const uint32_t end = s_wh[w * RADIX + tid];  // one past the slots drawn
          for (uint32_t a = at, b = end; a + 1u < b; ++a) {
            --b;
            if constexpr (INDEX) {
              const uint16_t x = s_idx[a];
              s_idx[a] = s_idx[b];
              s_idx[b] = x;
            } else {
              const K x = s_out[a];
              s_out[a] = s_out[b];
              s_out[b] = x;
            }
          }
          at = end;
        }
      }
    }
  }
  // past the end, and one more: what the scatter may read, and ascends to
  for (uint32_t i = tile_len + tid; i <= uint32_t(TILE); i += THREADS) {
    if constexpr (INDEX) s_idx[i] = uint16_t(tile_len - 1u);
    else s_out[i] = ~K(0);
  }
  stamp(trace(), 8);
  if constexpr (PERSIST) {
    if (tid == 0) s_misc[3] = atomicAdd(pf->counter, 1u);
  }

  // ---- 4. the rest of the look-back
  bool gave_up = false;
  if (tid < RADIX) {
    lb.consume(trace());
    gave_up = !lb.finish(t, tid, ctrl, timeout_ns, tile, trace());
    const uint32_t excl = lb.excl;
    if (!gave_up && !silent) {
      const uint32_t pub = kFlagInc | ((excl + my_cnt) & kValueMask);
      if constexpr (FLAT) {
        if (tile > 0u && dbg_ok(lb_index<RADIX>(t.tile0 + tile, tid), t.lb_words, kSiteTileStatus))
          st_relaxed(&t.status[lb_index<RADIX>(t.tile0 + tile, tid)], pub);
      } else {
        const size_t s = size_t(tile / kSuperTiles) * RADIX + tid;
        if ((tile + 1) % kSuperTiles == 0 && dbg_ok(s, t.s_words, kSiteGroupInc))
          st_relaxed(&t.sinc[s], pub);
      }
    }
    // every key of digit tid goes to [pass offset + excl, ... + its count):
    // checked here once, so that the scatters below need no per-element
    // bound.
    const uint32_t base = off0 + excl;
    if (!gave_up && (base > t.n || my_cnt > t.n - base)) {
      report_error(ctrl, kDevIndex, tile);
      gave_up = true;
    }
    stamp(trace(), 9);
    s_gbase[tid] = base - my_start;
  }
  if constexpr (VB > 0) {
    if (!mbar_wait(&s_bar[1], parity, ctrl, timeout_ns, tile)) gave_up = true;
  }
  // the output of a call that gave up is void (ctrl->error says why)
  if (__syncthreads_or(gave_up)) return leave(false, true);
  stamp(trace(), 4);
  if constexpr (PERSIST) {
    *next = s_misc[3];
    if (*next < pf->tiles) {
      // staged keys: their buffer and the counters are free -- start the next tile
      if constexpr (!INDEX) stage_tile<S, K, VB, THREADS, CG>(smem, *next);
    }
  }

  // consecutive threads take consecutive stage slots, which map to
  // consecutive output addresses inside each digit run; first the keys
  const V* s_vin = nullptr;
  if constexpr (VB > 0) s_vin = Stage<V>(t.vsrc + tile_base, tile_len).at(smem + S::VIN);
  // the bits that ascend over a stage of keys
  auto upto_bits = [&]() { return K((K(t.mask) << t.shift) | ((K(1) << t.shift) - K(1))); };
  // one instance for full and partial tiles, with or without the last pass's
  // inverse transform: of four, the compiler kept the common loads in
  // registers across the branch and spilled
  uint32_t bad = 0u;
  uint32_t dst[VB > 0 ? ITEMS : 1];  // the values' destinations
  uint32_t places[VB > 0 ? (ITEMS + 1) / 2 : 1];  // and places in the tile, two a word
  {
    const uint32_t shift = t.shift, mask = t.mask;
    const bool xout = t.xout;
    [[maybe_unused]] const uint32_t n = t.n;
    [[maybe_unused]] const K upto = upto_bits();
    K* kdst = t.kdst;
    // debug builds, test-only: every destination of this tile past the array,
    // so that the bounds checks must drop the stores (0 otherwise)
    const uint32_t dbg_push = (kDebugChecks && int(tile) == t.bad_tile) ? n : 0u;
#pragma unroll
    for (int s0 = 0; s0 < ITEMS; s0 += OUT_BATCH) {
      K k[OUT_BATCH];
      uint32_t g[OUT_BATCH];
      [[maybe_unused]] uint32_t at[OUT_BATCH];
#pragma unroll
      for (int s = s0; s < ITEMS && s < s0 + OUT_BATCH; ++s) {
        const uint32_t i = uint32_t(s * THREADS + tid);
        if constexpr (INDEX) {
          at[s - s0] = s_idx[i];
          bad += at[s - s0] > uint32_t(s_idx[i + 1]) ? 1u : 0u;
          if constexpr (VB > 0)
            places[s / 2] = s & 1 ? places[s / 2] | at[s - s0] << 16 : at[s - s0];
        } else {
          k[s - s0] = s_out[i];
          bad |= (k[s - s0] & upto) > (s_out[i + 1] & upto) ? 1u : 0u;
        }
      }
#pragma unroll
      for (int s = s0; s < ITEMS && s < s0 + OUT_BATCH; ++s) {
        if constexpr (INDEX) k[s - s0] = s_kin[at[s - s0]];
        g[s - s0] = s_gbase[digit_of(k[s - s0], shift, mask)] + uint32_t(s * THREADS + tid) +
                    dbg_push;
      }
      if (xout) {  // the last pass that moves data writes the keys back untransformed
        const KeyXf<K> xf = t.xf;
#pragma unroll
        for (int s = s0; s < ITEMS && s < s0 + OUT_BATCH; ++s) k[s - s0] = xf_inv(k[s - s0], xf);
      }
#pragma unroll
      for (int s = s0; s < ITEMS && s < s0 + OUT_BATCH; ++s) {
        const bool in = uint32_t(s * THREADS + tid) < tile_len;
        if (in && dbg_ok(g[s - s0], n, kSiteKeyScatter)) kdst[g[s - s0]] = k[s - s0];
        if constexpr (VB > 0) dst[s] = g[s - s0];
      }
    }
  }
  // the sum of a check over the CTA (a barrier): 0 when the stage is in order
  auto check = [&](uint32_t bad, int which) {
    if constexpr (INDEX) {
      // descents at the starts of digit runs are due: take them off the count
      if (tid < RADIX && my_cnt > 0u && my_start > 0u &&
          s_idx[my_start - 1] > s_idx[my_start])
        bad -= 1u;
      bad = __reduce_add_sync(kFull, bad);
      if (lane == 0 && bad != 0u) atomicAdd(&s_misc[which], bad);
      __syncthreads();
      return s_misc[which];
    } else {
      return uint32_t(__syncthreads_or(bad != 0u));
    }
  };
  bool ok = check(bad, 5) == 0u;
  const bool repaired = !ok;
  if (!ok) {
    if (tid == 0) count_repair(t.order);
    // out of turn.  A warp draws a digit's slots from a range that no other
    // warp draws from, and the ranges are in order, so that no element is further
    // from its place than such a range is long (at most ITEMS * 32): that many
    // rounds of odd-even transposition, and one for the first parity, put
    // every digit run in order.  Two rounds without an exchange end them
    // early (draws out of turn within one item take up to 32).
    auto wrong = [&](uint32_t i) {  // stage slots i and i + 1 are out of order
      if constexpr (INDEX) {
        const uint32_t a = s_idx[i], b = s_idx[i + 1];
        return a > b && digit_of(s_kin[a], t.shift, t.mask) == digit_of(s_kin[b], t.shift, t.mask);
      } else {
        return (s_out[i] & upto_bits()) > (s_out[i + 1] & upto_bits());
      }
    };
    for (int r = 0, go = 2; r <= ITEMS * 32 && go > 0; ++r) {
      bool moved = false;
      for (uint32_t i = uint32_t(2 * tid + (r & 1)); i + 1u < tile_len; i += 2 * THREADS) {
        if (!wrong(i)) continue;
        moved = true;
        if constexpr (INDEX) {
          const uint16_t a = s_idx[i];
          s_idx[i] = s_idx[i + 1];
          s_idx[i + 1] = a;
        } else {
          const K a = s_out[i];
          s_out[i] = s_out[i + 1];
          s_out[i + 1] = a;
        }
      }
      go = __syncthreads_or(moved) ? 2 : go - 1;
    }
    bad = 0u;
    for (uint32_t i = tid; i < tile_len; i += THREADS) {
      K k;
      uint32_t at = 0u;
      if constexpr (INDEX) {
        at = s_idx[i];
        bad += at > uint32_t(s_idx[i + 1]) ? 1u : 0u;
        k = s_kin[at];
      } else {
        k = s_out[i];
        bad |= wrong(i) && i + 1u < tile_len ? 1u : 0u;
      }
      const uint32_t g = s_gbase[digit_of(k, t.shift, t.mask)] + i;
      if (dbg_ok(g, t.n, kSiteKeyScatter)) t.kdst[g] = t.xout ? xf_inv(k, t.xf) : k;
      if constexpr (VB > 0)
        if (dbg_ok(g, t.n, kSiteValScatter)) t.vdst[g] = s_vin[at];
    }
    ok = check(bad, 6) == 0u;
  }
  if (!ok && tid == 0) report_error(ctrl, kDevIndex, tile);
  // INDEX: every key has left the buffer -- start the next tile, under the
  // scatter of the values
  if constexpr (PERSIST && INDEX) {
    if (ok && *next < pf->tiles) stage_tile<S, K, VB, THREADS, CG>(smem, *next);
  }
  if constexpr (VB > 0) {
    if (!repaired) {  // (a repaired tile's values went with its keys)
      V* vdst = t.vdst;
      [[maybe_unused]] const uint32_t n = t.n;
#pragma unroll
      for (int s = 0; s < ITEMS; ++s) {
        const uint32_t i = uint32_t(s * THREADS + tid);
        const V v = s_vin[s & 1 ? places[s / 2] >> 16 : places[s / 2] & 0xffffu];
        if (i < tile_len && dbg_ok(dst[s], n, kSiteValScatter)) vdst[dst[s]] = v;
      }
    }
  }
  stamp(trace(), 6);
  if (!ok) {
    // (keys, resident: the next tile's copy is in flight and must land first)
    if constexpr (PERSIST && !INDEX) {
      if (*next < pf->tiles) mbar_wait(&s_bar[0], parity ^ 1u, ctrl, timeout_ns, tile);
      __syncthreads();
    }
  }
  return leave(ok, true);
}

// The operands of a whole-array pass (one thread; a barrier follows).
template <class K, int VB, int RADIX>
__device__ __forceinline__ void pass_args(
    TileArgs<K, VB>* t, K* k0, K* k1, ValT<VB>* v0, ValT<VB>* v1, uint32_t n, int pass,
    uint32_t exec, uint32_t shift, uint32_t mask, const uint32_t* pass_offsets,
    const LookBackWords& lbw, uint32_t tiles, const KeyXf<K>& xf, const Knobs& knobs) {
  const bool from_alt = (__popc(exec & ((1u << pass) - 1u)) & 1) != 0;
  t->ksrc = from_alt ? k1 : k0;
  t->kdst = from_alt ? k0 : k1;
  t->vsrc = from_alt ? v1 : v0;
  t->vdst = from_alt ? v0 : v1;
  t->pass_offsets = pass_offsets;
  t->status = lbw.status;
  t->gagg = lbw.gagg;
  t->sagg = lbw.sagg;
  t->sinc = lbw.sinc;
  t->lb_words = uint64_t(tiles) * RADIX;
  t->g_words = uint64_t((tiles + kGroupTiles - 1) / kGroupTiles) * RADIX;
  t->s_words = uint64_t((tiles + kSuperTiles - 1) / kSuperTiles) * RADIX;
  t->xf = xf;
  t->n = n;
  t->shift = shift;
  t->mask = mask;
  t->tile0 = 0u;
  t->xin = xf.on && pass == __ffs(int(exec)) - 1;  // first and last pass that move data
  t->xout = xf.on && pass == 31 - __clz(exec);
  t->order = knobs.order;
  t->drop_tile = pass == knobs.drop_pass ? knobs.drop_tile : -1;
  t->bad_tile = kDebugChecks && pass == 0 ? knobs.dbg_bad_tile : -1;
  t->trace = pass == knobs.trace_pass ? knobs.trace : nullptr;
  t->trace_tiles = knobs.trace_tiles;
}

// One digit pass, one tile per CTA.  The grid has one CTA per tile; tile ids
// come from an atomic counter so that a tile's predecessors have always
// started before it (forward progress of the look-back).
template <class K, int VB, int RADIX_BITS, int THREADS, int ITEMS, int MINB, bool INDEX>
__global__ void __launch_bounds__(THREADS, MINB)
    k_onesweep(K* __restrict__ k0, K* __restrict__ k1, ValT<VB>* __restrict__ v0,
               ValT<VB>* __restrict__ v1, uint32_t n, int pass, uint32_t shift, uint32_t mask,
               const uint32_t* __restrict__ pass_offsets, LookBackWords lbw, uint32_t tiles,
               Ctrl* __restrict__ ctrl, Knobs knobs, KeyXf<K> xf, bool early_dependents) {
  using S = OnesweepSmem<K, VB, RADIX_BITS, THREADS, ITEMS, INDEX>;
  extern __shared__ __align__(16) unsigned char smem[];
  uint32_t* s_misc = reinterpret_cast<uint32_t*>(smem + S::MISC);
  pdl_wait();  // the kernel before (upsweep or previous pass) is complete
  // a grid of more tiles than CTA slots lets the next pass be scheduled
  // during its last wave; a one-wave grid lets it in as its CTAs exit, so
  // that the next pass's CTAs spread over the SMs
  if (early_dependents) pdl_launch_dependents();

  const uint32_t exec = ctrl->exec_mask;
  if (!((exec >> pass) & 1u)) return;  // every key has the same digit: nothing moves
  if (threadIdx.x == 0) {
    s_misc[0] = atomicAdd(&ctrl->tile_counter[pass], 1u);
    s_misc[2] = ld_relaxed(&ctrl->error);  // an earlier pass of this call gave up
    if (s_misc[0] == 0u) ctrl->t_pass[pass][0] = stat_now(ctrl);
    pass_args<K, VB, S::RADIX>(reinterpret_cast<TileArgs<K, VB>*>(smem + S::ARGS), k0, k1, v0, v1,
                               n, pass, exec, shift, mask, pass_offsets, lbw, tiles, xf, knobs);
  }
  __syncthreads();
  if (s_misc[2] != 0u) return;  // CTA-uniform
  onesweep_tile<K, VB, RADIX_BITS, THREADS, ITEMS, INDEX, false>(s_misc[0], ctrl, knobs.timeout_ns,
                                                                smem);
  __syncthreads();
  if (threadIdx.x == 0) atomicMax(&ctrl->t_pass[pass][1], stat_now(ctrl));
}

// One digit pass with resident CTAs (a grid of SMs x resident CTAs): each CTA
// takes tiles from the pass's atomic counter one after another and starts
// loading its next tile while it finishes the current one.  Tile ids are
// still taken in order by running CTAs, so the look-back keeps making
// progress: the lowest unfinished tile is always being worked on.
template <class K, int VB, int RADIX_BITS, int THREADS, int ITEMS, int MINB, bool INDEX>
__global__ void __launch_bounds__(THREADS, MINB)
    k_onesweep_persist(K* __restrict__ k0, K* __restrict__ k1, ValT<VB>* __restrict__ v0,
                       ValT<VB>* __restrict__ v1, uint32_t n, int pass, uint32_t shift,
                       uint32_t mask, const uint32_t* __restrict__ pass_offsets,
                       LookBackWords lbw, uint32_t tiles, Ctrl* __restrict__ ctrl,
                       Knobs knobs, KeyXf<K> xf, bool early_dependents) {
  using S = OnesweepSmem<K, VB, RADIX_BITS, THREADS, ITEMS, INDEX>;
  extern __shared__ __align__(16) unsigned char smem[];
  uint32_t* s_misc = reinterpret_cast<uint32_t*>(smem + S::MISC);
  uint64_t* s_bar = reinterpret_cast<uint64_t*>(smem + S::MBAR);
  pdl_wait();  // the kernel before (upsweep or previous pass) is complete
  if (early_dependents) pdl_launch_dependents();

  const uint32_t exec = ctrl->exec_mask;
  if (!((exec >> pass) & 1u)) return;  // every key has the same digit: nothing moves
  Prefetch pf{&ctrl->tile_counter[pass], tiles};
  if (threadIdx.x == 0) {
    mbar_init(&s_bar[0]);
    if constexpr (VB > 0) mbar_init(&s_bar[1]);
    s_misc[3] = atomicAdd(pf.counter, 1u);
    s_misc[2] = ld_relaxed(&ctrl->error);  // an earlier pass of this call gave up
    if (s_misc[3] == 0u) ctrl->t_pass[pass][0] = stat_now(ctrl);
    pass_args<K, VB, S::RADIX>(reinterpret_cast<TileArgs<K, VB>*>(smem + S::ARGS), k0, k1, v0, v1,
                               n, pass, exec, shift, mask, pass_offsets, lbw, tiles, xf, knobs);
  }
  __syncthreads();
  uint32_t tile = s_misc[2] == 0u ? s_misc[3] : tiles;
  if (tile < tiles) stage_tile<S, K, VB, THREADS, false>(smem, tile);
  for (uint32_t it = 0; tile < tiles; ++it) {
    uint32_t next = tiles;
    // a tile that gives up has taken no next one, or not started to load it
    if (!onesweep_tile<K, VB, RADIX_BITS, THREADS, ITEMS, INDEX, false, true>(
            tile, ctrl, knobs.timeout_ns, smem, it & 1u, &pf, &next))
      break;
    tile = next;
  }
  __syncthreads();
  if (threadIdx.x == 0) {
    mbar_inval(&s_bar[0]);
    if constexpr (VB > 0) mbar_inval(&s_bar[1]);
    atomicMax(&ctrl->t_pass[pass][1], stat_now(ctrl));
  }
}

// ------------------------------------------------------------ small sort

// The rank of one key among its warp's keys of digit d so far, from the warp's
// counters wh.  Fast: one returning atomic, whose order among the lanes is the
// hardware's (see onesweep_tile), so the caller checks the sorted result.
// careful: the lanes holding the same digit are found with match.any and take
// consecutive ranks in lane order; the whole warp calls it, in: lanes that
// hold a key.
__device__ __forceinline__ uint32_t draw_rank(uint32_t* wh, uint32_t d, bool in, bool careful,
                                              int lane) {
  uint32_t r = 0u;
  if (!careful) {
    if (in) r = atomicAdd(&wh[d], 1u);
    return r;
  }
  const uint32_t peers = __match_any_sync(kFull, in ? d : ~0u);
  const int leader = 31 - __clz(peers);
  if (in && lane == leader) {
    r = wh[d];
    wh[d] = r + uint32_t(__popc(peers));
  }
  __syncwarp();
  return __shfl_sync(kFull, r, leader) + uint32_t(__popc(peers & lanemask_lt()));
}

// Shared memory of a sort inside one CTA.  INDEX: the keys' 16-bit input
// positions travel with them, which orders the values at the end and lets the
// result be checked for stability; whole keys without values need neither.
template <class K, int VB, int RADIX_BITS, int THREADS, int ITEMS, bool INDEX>
struct SmallSmem {
  static constexpr int RADIX = 1 << RADIX_BITS;
  static constexpr int WARPS = THREADS / 32;
  static constexpr int TILE = THREADS * ITEMS;
  static constexpr int WH = 0;                            // u32 [2][WARPS][RADIX], by pass parity
  static constexpr int TOT = WH + 2 * WARPS * RADIX * 4;  // u32 [32]
  static constexpr int KEYS = TOT + 32 * 4;                              // K [TILE]
  static constexpr int IDX = KEYS + TILE * int(sizeof(K));               // u16 [TILE]
  static constexpr int END = (IDX + (INDEX ? TILE * 2 : 0) + 15) / 16 * 16;
  static constexpr int BYTES = END;
  // the values, in the end, go where the counters were if they fit, else
  // where the keys were
  static constexpr bool VALS_FIT = TILE * VB <= TOT;
  static_assert(VB == 0 || VB == int(sizeof(K)), "the values fit the keys' place");
};

// All digit passes of one array of len <= TILE elements inside one CTA.  The
// input and output may be the same buffers: everything is read before the
// first write.
//
// Bound by latency: a pass is a chain of five barriers, the draws, the sums
// over the warps and the stage.  Work follows the length (items per thread =
// len / THREADS, rounded up), and a pass's loads, draws and stores go in
// batches.  A sort whose result is out of order is done again with careful
// ranks.  Peer-mask ranks and a full tile whatever the length took 15.2 us for
// 3,000 32-bit keys and 643 us for 10,000 rows of 1,500 keys on average.
template <class K, int VB, int RADIX_BITS, int THREADS, int ITEMS, bool INDEX>
__device__ __forceinline__ void cta_sort(const K* kin, const ValT<VB>* vin, K* kout,
                                         ValT<VB>* vout, uint32_t len, int begin_bit,
                                         int end_bit, unsigned char* smem, const KeyXf<K>& xf,
                                         const OrderTest& order) {
  using V = ValT<VB>;
  using S = SmallSmem<K, VB, RADIX_BITS, THREADS, ITEMS, INDEX>;
  constexpr int RADIX = S::RADIX, WARPS = S::WARPS;
  static_assert(INDEX || VB == 0, "values follow their keys' positions");
  static_assert(S::TILE <= 65536, "positions fit 16 bits");
  uint32_t* s_tot = reinterpret_cast<uint32_t*>(smem + S::TOT);
  K* s_k = reinterpret_cast<K*>(smem + S::KEYS);
  uint16_t* s_i = reinterpret_cast<uint16_t*>(smem + S::IDX);
  const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
  const int items = int((len + THREADS - 1) / THREADS);
  constexpr int BATCH = ITEMS < 4 ? ITEMS : 4;
  // the bits the sort looks at
  const K looked = (end_bit - begin_bit == 8 * int(sizeof(K)))
                       ? ~K(0)
                       : K(((K(1) << (end_bit - begin_bit)) - K(1)) << begin_bit);

  if constexpr (VB > 0) {  // needed in the end only: into the L2 meanwhile
    for (uint32_t i = tid * (32 / VB); i < len; i += THREADS * (32 / VB))
      asm volatile("prefetch.global.L2 [%0];" ::"l"(vin + i));
  }
  for (int attempt = 0; attempt < 2; ++attempt) {
    const bool careful = attempt != 0;
    // item j of lane l of warp w is element (w * items + j) * 32 + l
    const uint32_t slot0 =
        uint32_t(warp * items * 32 + (order.mirror && !careful ? 31 - lane : lane));
    for (uint32_t i = tid; i < len; i += THREADS) {
      const K k = kin[i];
      s_k[i] = xf.on ? xf_fwd(k, xf) : k;
      if constexpr (INDEX) s_i[i] = uint16_t(i);
    }
    for (int i = tid; i < WARPS * RADIX / 4; i += THREADS)
      reinterpret_cast<uint4*>(smem + S::WH)[i] = make_uint4(0u, 0u, 0u, 0u);
    __syncthreads();
    int parity = 0;
    for (int lo = begin_bit; lo < end_bit; lo += RADIX_BITS, parity ^= 1) {
      const uint32_t shift = uint32_t(lo);
      const uint32_t mask = (1u << (min(lo + RADIX_BITS, end_bit) - lo)) - 1u;
      uint32_t* s_wh = reinterpret_cast<uint32_t*>(smem + S::WH) + parity * WARPS * RADIX;
      uint32_t* wh = s_wh + warp * RADIX;
      K key[ITEMS];
      uint32_t meta[ITEMS];  // rank << 16 | input position
#pragma unroll
      for (int j0 = 0; j0 < ITEMS; j0 += BATCH) {
        if (j0 >= items) break;
#pragma unroll
        for (int j = j0; j < ITEMS && j < j0 + BATCH; ++j) {
          const uint32_t at = slot0 + j * 32;
          const bool in = j < items && at < len;
          key[j] = in ? s_k[at] : K(0);
          meta[j] = 0u;
          if constexpr (INDEX) meta[j] = in ? s_i[at] : 0u;
        }
#pragma unroll
        for (int j = j0; j < ITEMS && j < j0 + BATCH; ++j) {
          const bool in = j < items && slot0 + j * 32 < len;
          meta[j] |= draw_rank(wh, digit_of(key[j], shift, mask), in, careful, lane) << 16;
        }
      }
      __syncthreads();
      // per digit: the count, its start, and from there the warps' starts
      // (32 warps' counts are read twice: in registers they would spill)
      constexpr bool KEEP = WARPS <= 16;
      uint32_t c[KEEP ? WARPS : 1], cnt = 0u;
      if (tid < RADIX) {
#pragma unroll
        for (int w = 0; w < WARPS; ++w) {
          const uint32_t x = s_wh[w * RADIX + tid];
          if constexpr (KEEP) c[w] = x;
          cnt += x;
        }
      }
      const uint32_t inc = warp_inclusive_scan(cnt, lane);
      if (lane == 31) s_tot[warp] = inc;
      __syncthreads();
      if (tid < RADIX) {
        uint32_t run =
            __reduce_add_sync(kFull, lane < RADIX / 32 && lane < warp ? s_tot[lane] : 0u) + inc -
            cnt;
#pragma unroll(KEEP ? WARPS : 8)
        for (int w = 0; w < WARPS; ++w) {
          uint32_t x;
          if constexpr (KEEP) x = c[w];
          else x = s_wh[w * RADIX + tid];
          s_wh[w * RADIX + tid] = run;
          run += x;
        }
      }
      __syncthreads();
#pragma unroll
      for (int j0 = 0; j0 < ITEMS; j0 += BATCH) {
        if (j0 >= items) break;
        uint32_t p[BATCH];
#pragma unroll
        for (int j = j0; j < ITEMS && j < j0 + BATCH; ++j)
          p[j - j0] = wh[digit_of(key[j], shift, mask)] + (meta[j] >> 16);
#pragma unroll
        for (int j = j0; j < ITEMS && j < j0 + BATCH; ++j) {
          if (j < items && slot0 + j * 32 < len) {
            s_k[p[j - j0]] = key[j];
            if constexpr (INDEX) s_i[p[j - j0]] = uint16_t(meta[j]);
          }
        }
      }
      // the next pass's counters (nothing reads them until then)
      uint4* zero = reinterpret_cast<uint4*>(smem + S::WH) + (parity ^ 1) * WARPS * RADIX / 4;
      for (int i = tid; i < WARPS * RADIX / 4; i += THREADS) zero[i] = make_uint4(0u, 0u, 0u, 0u);
      __syncthreads();
    }
    bool bad = false;
    for (uint32_t i = tid; i + 1u < len; i += THREADS) {
      const K a = s_k[i] & looked, b = s_k[i + 1] & looked;
      if constexpr (INDEX) bad = bad || a > b || (a == b && s_i[i] > s_i[i + 1]);
      else bad = bad || a > b;
    }
    if (!__syncthreads_or(bad)) break;
    if (!careful && tid == 0) count_repair(order);
  }
  // (a test of the length instead left the 1024 x 16 form for 64-bit pairs 40
  // bytes of spills and 5 % slower)
  constexpr bool fit = VB > 0 && S::VALS_FIT;
  V* s_v = reinterpret_cast<V*>(smem + (fit ? S::WH : S::KEYS));
  if (fit) {
    for (uint32_t i = tid; i < len; i += THREADS) s_v[i] = vin[i];
    __syncthreads();
  }
  for (uint32_t i = tid; i < len; i += THREADS) {
    if (!dbg_ok(i, len, kSiteSmallOut)) continue;
    kout[i] = xf.on ? xf_inv(s_k[i], xf) : s_k[i];
    if (fit) vout[i] = s_v[s_i[i]];
  }
  if (VB > 0 && !fit) {
    __syncthreads();  // the keys have left
    for (uint32_t i = tid; i < len; i += THREADS) s_v[i] = vin[i];
    __syncthreads();
    for (uint32_t i = tid; i < len; i += THREADS)
      if (dbg_ok(i, len, kSiteSmallOut)) vout[i] = s_v[s_i[i]];
  }
}

// ctrl (may be null): the caller's workspace, whose status words this call
// resets so that a later status read reports this call.
template <class K, int VB, int RADIX_BITS, int THREADS, int ITEMS, bool INDEX>
__global__ void __launch_bounds__(THREADS, 1)
    k_small_sort(K* keys, ValT<VB>* vals, uint32_t n, int begin_bit, int end_bit, Ctrl* ctrl,
                 KeyXf<K> xf, OrderTest order) {
  extern __shared__ __align__(16) unsigned char smem[];
  const int passes = (end_bit - begin_bit + RADIX_BITS - 1) / RADIX_BITS;
  if (ctrl != nullptr && threadIdx.x == 0) {
    ctrl->error = 0u;
    ctrl->error_info = 0u;
    ctrl->exec_mask = (1u << passes) - 1u;  // every pass runs (in shared memory)
    stat_clear_times(ctrl);
    stat_begin(ctrl, n, uint32_t(sizeof(K)) | uint32_t(VB) << 8 | uint32_t(passes) << 16 |
                            3u << 24);
  }
  cta_sort<K, VB, RADIX_BITS, THREADS, ITEMS, INDEX>(keys, vals, keys, vals, n, begin_bit, end_bit,
                                                     smem, xf, order);
  __syncthreads();
  if (ctrl != nullptr && threadIdx.x == 0) ctrl->t_upsweep = stat_now(ctrl);
}

}  // namespace rs
