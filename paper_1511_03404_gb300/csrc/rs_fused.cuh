// One-launch form of the sort for arrays of moderate size, where the
// separate launches of the upsweep and of each digit pass, each waiting for
// the previous one, cost more than the passes themselves.  A cooperative
// grid (every CTA resident) runs:
//   1. the digit histograms of every pass over a grid-stride share of the
//      keys (shared counters, then one global add per digit), and clears
//      the look-back words;
//   -- grid barrier --
//   2. in every CTA, the exclusive scans (all passes at once) and the set of
//      passes that move data (the same rule as the upsweep's last CTA), kept
//      in shared memory;
//   3. each moving pass: the onesweep tile (rank, look-back, stable scatter)
//      on L2-coherent loads of the previous pass's output.  An array of no
//      more tiles than CTAs gives CTA b tile b (all are resident, so that the
//      look-back makes progress); a larger one takes tiles from the pass's
//      counter;
//   -- grid barrier after each pass --
// Every barrier wait is bounded; a CTA that gives up records
// RS_ERR_TIMEOUT and returns, and the others' bounded waits end as well.
//
// Bound by latency.  A barrier costs about 1.5 us against 2.5 to 3 from one
// kernel to the next, but scans one pass after another (1.2 us each) and two
// tile tickets a pass (0.7 us each) had taken more than that back.
#pragma once

#include <type_traits>

#include "rs_kernels.cuh"

namespace rs {

template <class K, int VB, int RADIX_BITS, int THREADS, int ITEMS, bool INDEX>
struct FusedSmem {
  using S = OnesweepSmem<K, VB, RADIX_BITS, THREADS, ITEMS, INDEX>;
  static constexpr int RADIX = 1 << RADIX_BITS;
  static constexpr int MAXP = (8 * int(sizeof(K)) + RADIX_BITS - 1) / RADIX_BITS;
  static constexpr int OFF = (S::BYTES + 15) / 16 * 16;  // u32 [MAXP][RADIX] digit offsets
  static constexpr int FLAG = OFF + MAXP * RADIX * 4;    // u32: barrier outcome
  static constexpr int ONE = FLAG + 4;                   // u32: passes with one digit value
  static constexpr int BYTES = FLAG + 16;
  // the histograms of step 1 use the warp-counter region of the tile
  static_assert(MAXP <= S::WARPS, "histograms fit the warp counters");
};

// All CTAs of the grid meet; false if the wait ran out or an error was
// reported (CTA-uniform).  Nothing else may write *s_flag: no barrier stands
// between the threads' reads of it here and what thread 0 does next, and a
// thread that read another word's zero would leave the kernel alone.
__device__ __forceinline__ bool grid_barrier(Ctrl* ctrl, uint32_t gen, uint64_t timeout_ns,
                                             uint32_t* s_flag) {
  __syncthreads();
  if (threadIdx.x == 0) {
    // release and acquire order the CTA's stores (before the barrier above)
    // and its later loads; sequentially consistent fences took twice as long
    asm volatile("red.release.gpu.global.add.u32 [%0], %1;" ::"l"(&ctrl->grid_bar), "r"(1u)
                 : "memory");
    const bool ok = wait_geq(&ctrl->grid_bar, gen * gridDim.x, ctrl, timeout_ns, 0xffffffffu);
    *s_flag = ok ? 1u : 0u;
  }
  __syncthreads();
  if constexpr (kDebugChecks) {
    // debug builds: all warps but the first read late, so that a store to the
    // word before they have read it shows
    const uint64_t t0 = global_ns();
    while (threadIdx.x >= 32 && global_ns() - t0 < 20000u) {
    }
  }
  return *s_flag != 0u;
}

template <class K, int VB, int RADIX_BITS, int THREADS, int ITEMS, int MINB, bool INDEX>
__global__ void __launch_bounds__(THREADS, MINB)
    k_fused(K* __restrict__ k0, K* __restrict__ k1, ValT<VB>* __restrict__ v0,
            ValT<VB>* __restrict__ v1, uint32_t n, int begin_bit, int end_bit, int passes,
            uint32_t* __restrict__ counts, Layout lay, uint32_t tiles,
            uint4* __restrict__ zero_base, uint64_t zero_vec4, Ctrl* __restrict__ ctrl, Knobs knobs, KeyXf<K> xf,
            uint32_t shape, bool copy) {
  using F = FusedSmem<K, VB, RADIX_BITS, THREADS, ITEMS, INDEX>;
  using S = typename F::S;
  constexpr int RADIX = F::RADIX, MAXP = F::MAXP;
  extern __shared__ __align__(16) unsigned char smem[];
  uint32_t* s_hist = reinterpret_cast<uint32_t*>(smem + S::WH);
  uint32_t* s_misc = reinterpret_cast<uint32_t*>(smem + S::MISC);
  uint32_t* s_off = reinterpret_cast<uint32_t*>(smem + F::OFF);
  uint32_t* s_flag = reinterpret_cast<uint32_t*>(smem + F::FLAG);
  uint32_t* s_one = reinterpret_cast<uint32_t*>(smem + F::ONE);
  const int tid = threadIdx.x;
  const bool rec = blockIdx.x == 0 && tid == 0;  // keeps the per-call record
  if (rec) stat_begin(ctrl, n, shape);

  // ---- 1. histograms of every pass, and the look-back words cleared
  for (int i = tid; i < passes * RADIX; i += THREADS) s_hist[i] = 0u;
  if (tid == 0) *s_one = 0u;
  __syncthreads();
  // copy: the input is in k1 and v1 and the passes start from a copy in k0 and
  // v0, so that an odd number of them ends where the input was
  const K* kin = copy ? k1 : k0;
  if constexpr (VB > 0) {
    if (copy)
      for (uint32_t i = blockIdx.x * THREADS + tid; i < n; i += gridDim.x * THREADS)
        if (dbg_ok(i, n, kSiteCopyVals)) v0[i] = v1[i];
  }
  auto count_all = [&](auto XF) {
    constexpr int LOADS = 4;  // in flight per thread
    const uint32_t stride = gridDim.x * THREADS;
    for (uint32_t i0 = blockIdx.x * THREADS + tid; i0 < n; i0 += stride * LOADS) {
      K k[LOADS];
#pragma unroll
      for (uint32_t u = 0; u < LOADS; ++u)
        if (i0 + u * stride < n) k[u] = kin[i0 + u * stride];
#pragma unroll
      for (uint32_t u = 0; u < LOADS; ++u) {
        if (i0 + u * stride >= n) break;
        if (copy && dbg_ok(i0 + u * stride, n, kSiteCopyKeys)) k0[i0 + u * stride] = k[u];
        if constexpr (decltype(XF)::value) k[u] = xf_fwd(k[u], xf);
#pragma unroll
        for (int p = 0; p < MAXP; ++p) {
          if (p < passes) {
            const int lo = begin_bit + p * RADIX_BITS;
            const uint32_t mask = (1u << min(RADIX_BITS, end_bit - lo)) - 1u;
            atomicAdd(&s_hist[p * RADIX + int(digit_of(k[u], uint32_t(lo), mask))], 1u);
          }
        }
      }
    }
  };
  if (xf.on)
    count_all(std::true_type{});
  else
    count_all(std::false_type{});
  for (uint64_t i = uint64_t(blockIdx.x) * THREADS + tid; i < zero_vec4;
       i += uint64_t(gridDim.x) * THREADS)
    if (dbg_ok(i, zero_vec4, kSiteFusedClear)) zero_base[i] = make_uint4(0u, 0u, 0u, 0u);
  __syncthreads();
  for (int w = tid; w < passes * RADIX; w += THREADS)
    if (s_hist[w] && dbg_ok(w, uint64_t(passes) * RADIX, kSiteFusedCounts))
      atomicAdd(&counts[w], s_hist[w]);
  uint32_t gen = 1;
  if (!grid_barrier(ctrl, gen, knobs.timeout_ns, s_flag)) return;

  // ---- 2. scans and moving passes, in every CTA: a digit a thread, all
  // passes at once
  static_assert(THREADS >= RADIX && THREADS / 32 <= 32, "one thread per digit");
  const int lane = tid & 31, warp = tid >> 5;
  uint32_t* s_sum = s_hist;  // [MAXP][32] the warps' sums (the histograms are added up)
  uint32_t cnt[MAXP], inc[MAXP];
  uint32_t one = 0u;  // passes in which my digit holds every key
#pragma unroll
  for (int p = 0; p < MAXP; ++p)
    cnt[p] = p < passes && tid < RADIX ? ld_relaxed(&counts[p * RADIX + tid]) : 0u;
#pragma unroll
  for (int p = 0; p < MAXP; ++p) {
    if (p < passes && tid < RADIX && cnt[p] == n) one |= 1u << p;
    inc[p] = warp_inclusive_scan(cnt[p], lane);
    if (lane == 31) s_sum[p * 32 + warp] = inc[p];
  }
  one = __reduce_or_sync(kFull, one);
  __syncthreads();
  if (lane == 0 && one != 0u) atomicOr(s_one, one);
#pragma unroll
  for (int p = 0; p < MAXP; ++p) {
    const uint32_t before =
        __reduce_add_sync(kFull, lane < THREADS / 32 && lane < warp ? s_sum[p * 32 + lane] : 0u);
    if (p < passes && tid < RADIX) s_off[p * RADIX + tid] = before + inc[p] - cnt[p];
  }
  __syncthreads();
  uint32_t exec = ~*s_one & ((1u << passes) - 1u);
  if ((__popc(exec) & 1) != (passes & 1)) {  // keep the result in buffer (passes mod 2)
    const uint32_t skipped = ~exec & ((1u << passes) - 1u);
    exec |= skipped & (0u - skipped);
  }
  if (rec) {
    ctrl->exec_mask = exec;
    ctrl->t_upsweep = stat_now(ctrl);
  }

  // ---- 3. the passes that move data
  for (int p = 0; p < passes; ++p) {
    if (!((exec >> p) & 1u)) continue;
    if (tid == 0) {
      const int lo = begin_bit + p * RADIX_BITS;
      auto* t = reinterpret_cast<TileArgs<K, VB>*>(smem + S::ARGS);
      pass_args<K, VB, RADIX>(t, k0, k1, v0, v1, n, p, exec, uint32_t(lo),
                              (1u << min(RADIX_BITS, end_bit - lo)) - 1u, s_off + p * RADIX,
                              lay.words(ctrl, p), tiles, xf, knobs);
      t->trace = nullptr;
      t->bad_tile = -1;
    }
    if (rec) ctrl->t_pass[p][0] = stat_now(ctrl);
    if (tiles <= gridDim.x) {
      __syncthreads();  // the operands are in place
      if (blockIdx.x < tiles)
        onesweep_tile<K, VB, RADIX_BITS, THREADS, ITEMS, INDEX, true>(blockIdx.x, ctrl,
                                                                      knobs.timeout_ns, smem);
    } else {
      for (;;) {
        __syncthreads();  // the previous tile is done with s_misc
        if (tid == 0) {
          s_misc[2] = ld_relaxed(&ctrl->error);
          s_misc[0] = s_misc[2] ? tiles : atomicAdd(&ctrl->tile_counter[p], 1u);
        }
        __syncthreads();
        const uint32_t tile = s_misc[0];
        if (tile >= tiles) break;  // CTA-uniform
        onesweep_tile<K, VB, RADIX_BITS, THREADS, ITEMS, INDEX, true>(tile, ctrl,
                                                                      knobs.timeout_ns, smem);
      }
    }
    ++gen;
    if (!grid_barrier(ctrl, gen, knobs.timeout_ns, s_flag)) return;
    if (rec) ctrl->t_pass[p][1] = stat_now(ctrl);
  }
}

}  // namespace rs
