// The whole sort inside one thread-block cluster, for arrays up to
// 8 x THREADS x ITEMS elements (65,536), whether on 8 CTAs or 16: every digit
// pass (Sec. 2.6) runs on data held in the cluster's shared memory, with no
// trip through global memory and no kernel boundary between passes.
//
// CTA c of the cluster owns positions [c * slice, (c + 1) * slice) of the
// array; the slice follows the length, so that every CTA takes part.  One
// pass:
//   1. each warp draws its keys' ranks from its counters (draw_rank); per-digit
//      prefixes over the warps give every key's place among the CTA's keys of
//      its digit, and the CTA's digit counts;
//   2. every CTA stores its digit counts into every CTA's count table
//      (remote shared-memory stores), and stages its keys (and their 16-bit
//      input positions) in digit order in its own source buffer; after a
//      cluster barrier each CTA reads its table: the start of digit d is the
//      count of all smaller digits, plus the count of digit d in lower-ranked
//      CTAs;
//   3. the staged keys go, in order, each to its global position, in the
//      destination buffer of the CTA that owns that position (a remote
//      shared-memory store): consecutive threads store consecutive keys of a
//      digit run to consecutive addresses of one CTA;
//   4. cluster barrier; the destination buffer becomes the next source.
// In the end the values are gathered by the positions that came with the
// keys.  A result out of order (the draws' order is the hardware's) is sorted
// again with careful ranks.  The cluster barriers are hardware barriers that
// every CTA passes the same number of times; no CTA waits on a flag.
#pragma once

#include "rs_kernels.cuh"

namespace rs {

__device__ __forceinline__ uint32_t cluster_ctarank() {
  uint32_t r;
  asm volatile("mov.u32 %0, %%cluster_ctarank;" : "=r"(r));
  return r;
}

__device__ __forceinline__ void cluster_sync_all() {
  asm volatile("barrier.cluster.arrive.release.aligned;\n\tbarrier.cluster.wait.acquire.aligned;"
               ::: "memory");
}

// The shared::cluster address of `p` (a shared-memory pointer of this CTA)
// in the CTA of cluster rank `rank`.
__device__ __forceinline__ uint32_t map_shared(const void* p, uint32_t rank) {
  const uint32_t local = static_cast<uint32_t>(__cvta_generic_to_shared(p));
  uint32_t remote;
  asm volatile("mapa.shared::cluster.u32 %0, %1, %2;" : "=r"(remote) : "r"(local), "r"(rank));
  return remote;
}

__device__ __forceinline__ void st_cluster(uint32_t addr, uint32_t v) {
  asm volatile("st.shared::cluster.u32 [%0], %1;" ::"r"(addr), "r"(v) : "memory");
}

__device__ __forceinline__ void st_cluster(uint32_t addr, uint64_t v) {
  asm volatile("st.shared::cluster.u64 [%0], %1;" ::"r"(addr), "l"(v) : "memory");
}

__device__ __forceinline__ uint32_t ld_cluster_u32(uint32_t addr) {
  uint32_t v;
  asm volatile("ld.shared::cluster.u32 %0, [%1];" : "=r"(v) : "r"(addr) : "memory");
  return v;
}

__device__ __forceinline__ void st_cluster(uint32_t addr, uint16_t v) {
  asm volatile("st.shared::cluster.u16 [%0], %1;" ::"r"(addr), "h"(v) : "memory");
}

template <class K, int RADIX_BITS, int THREADS, int ITEMS, bool INDEX>
struct ClusterSmem {
  static constexpr int RADIX = 1 << RADIX_BITS;
  static constexpr int WARPS = THREADS / 32;
  static constexpr int SLICE = THREADS * ITEMS;  // the largest
  static constexpr int KB = int(sizeof(K));
  static constexpr int MAX_CL = 16;
  static constexpr int WH = 0;                             // u32 [2][WARPS][RADIX], by pass parity
  static constexpr int CNT = WH + 2 * WARPS * RADIX * 4;   // u32 [MAX_CL][RADIX] every CTA's counts
  static constexpr int BASE = CNT + MAX_CL * RADIX * 4;    // u32 [RADIX] global digit bases
  static constexpr int TOT = BASE + RADIX * 4;             // u32 [32]
  static constexpr int EDGE = TOT + 32 * 4;                // first key, its position; u32 [4]
  static constexpr int FLAGS = EDGE + 16;                  // u32 [MAX_CL] out of order
  static constexpr int KEYS = FLAGS + MAX_CL * 4;          // K [2][SLICE]
  static constexpr int IDX = KEYS + 2 * SLICE * KB;        // u16 [2][SLICE]
  static constexpr int BYTES = IDX + (INDEX ? 2 * SLICE * 2 : 0);
};

template <class K, int VB, int RADIX_BITS, int THREADS, int ITEMS, bool INDEX>
__global__ void __launch_bounds__(THREADS, 1)
    k_cluster_sort(K* __restrict__ keys, ValT<VB>* __restrict__ vals, uint32_t n, uint32_t slice,
                   int begin_bit, int end_bit, Ctrl* ctrl, KeyXf<K> xf, OrderTest order) {
  using V = ValT<VB>;
  using S = ClusterSmem<K, RADIX_BITS, THREADS, ITEMS, INDEX>;
  constexpr int RADIX = S::RADIX, WARPS = S::WARPS;
  static_assert(INDEX || VB == 0, "values follow their keys' positions");
  extern __shared__ __align__(16) unsigned char smem[];
  uint32_t* s_cnt = reinterpret_cast<uint32_t*>(smem + S::CNT);
  uint32_t* s_base = reinterpret_cast<uint32_t*>(smem + S::BASE);
  uint32_t* s_tot = reinterpret_cast<uint32_t*>(smem + S::TOT);
  uint32_t* s_edge = reinterpret_cast<uint32_t*>(smem + S::EDGE);
  uint32_t* s_flags = reinterpret_cast<uint32_t*>(smem + S::FLAGS);
  const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
  const uint32_t rank = cluster_ctarank();
  const uint32_t ncta = gridDim.x;  // the grid is one cluster
  const int passes = (end_bit - begin_bit + RADIX_BITS - 1) / RADIX_BITS;
  const int items = int(slice / THREADS);
  const uint32_t base0 = rank * slice;
  const uint32_t len = n > base0 ? min(slice, n - base0) : 0u;
  const uint32_t magic = 0xffffffffu / slice + 1u;  // g / slice == mulhi(g, magic): g * slice < 2^32
  constexpr int BATCH = ITEMS < 4 ? ITEMS : 4;
  const K looked = (end_bit - begin_bit == 8 * int(sizeof(K)))
                       ? ~K(0)
                       : K(((K(1) << (end_bit - begin_bit)) - K(1)) << begin_bit);
  if (ctrl != nullptr && blockIdx.x == 0 && tid == 0) {
    ctrl->error = 0u;
    ctrl->error_info = 0u;
    ctrl->exec_mask = (1u << passes) - 1u;  // every pass runs (in shared memory)
    stat_clear_times(ctrl);
    stat_begin(ctrl, n, uint32_t(sizeof(K)) | uint32_t(VB) << 8 | uint32_t(passes) << 16 |
                            3u << 24);
  }
  if constexpr (VB > 0) {  // needed in the end only: into the L2 meanwhile
    for (uint32_t i = tid * (32 / VB); i < len; i += THREADS * (32 / VB))
      asm volatile("prefetch.global.L2 [%0];" ::"l"(vals + base0 + i));
  }
  // exclusive prefix over the CTA of one value per digit (thread d < RADIX); a
  // barrier, and the caller separates two calls by another
  auto scan = [&](uint32_t x) {
    const uint32_t inc = warp_inclusive_scan(x, lane);
    if (lane == 31) s_tot[warp] = inc;
    __syncthreads();
    return __reduce_add_sync(kFull, lane < RADIX / 32 && lane < warp ? s_tot[lane] : 0u) + inc - x;
  };

  // the first remote store waits until every CTA of the cluster has started
  asm volatile("barrier.cluster.arrive.release.aligned;" ::: "memory");
  bool started = false;
  int src = 0;
  for (int attempt = 0; attempt < 2; ++attempt) {
    const bool careful = attempt != 0;
    const uint32_t slot0 = uint32_t(warp * items * 32 + (order.mirror && !careful ? 31 - lane : lane));
    src = 0;
    {
      K* ks = reinterpret_cast<K*>(smem + S::KEYS);
      uint16_t* is = reinterpret_cast<uint16_t*>(smem + S::IDX);
      for (uint32_t i = tid; i < len; i += THREADS) {
        const K k = keys[base0 + i];
        ks[i] = xf.on ? xf_fwd(k, xf) : k;
        if constexpr (INDEX) is[i] = uint16_t(base0 + i);
      }
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
      K* ks = reinterpret_cast<K*>(smem + S::KEYS) + src * S::SLICE;
      uint16_t* is = reinterpret_cast<uint16_t*>(smem + S::IDX) + src * S::SLICE;
      // ---- 1. draws
      K key[ITEMS];
      uint32_t meta[ITEMS];  // rank << 16 | input position
#pragma unroll
      for (int j0 = 0; j0 < ITEMS; j0 += BATCH) {
        if (j0 >= items) break;
#pragma unroll
        for (int j = j0; j < ITEMS && j < j0 + BATCH; ++j) {
          const uint32_t at = slot0 + j * 32;
          const bool in = j < items && at < len;
          key[j] = in ? ks[at] : K(0);
          meta[j] = 0u;
          if constexpr (INDEX) meta[j] = in ? is[at] : 0u;
        }
#pragma unroll
        for (int j = j0; j < ITEMS && j < j0 + BATCH; ++j) {
          const bool in = j < items && slot0 + j * 32 < len;
          meta[j] |= draw_rank(wh, digit_of(key[j], shift, mask), in, careful, lane) << 16;
        }
      }
      __syncthreads();
      if (!started) asm volatile("barrier.cluster.wait.acquire.aligned;" ::: "memory");
      started = true;
      uint32_t c[WARPS], cnt = 0u;
      if (tid < RADIX) {
#pragma unroll
        for (int w = 0; w < WARPS; ++w) {
          c[w] = s_wh[w * RADIX + tid];
          cnt += c[w];
        }
        // ---- 2. this CTA's counts into every CTA's table
        for (uint32_t q = 0; q < ncta; ++q)
          st_cluster(map_shared(s_cnt + rank * RADIX + tid, q), cnt);
      }
      const uint32_t lstart = scan(cnt);
      if (tid < RADIX) {
        uint32_t run = lstart;
#pragma unroll
        for (int w = 0; w < WARPS; ++w) {
          s_wh[w * RADIX + tid] = run;
          run += c[w];
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
            ks[p[j - j0]] = key[j];
            if constexpr (INDEX) is[p[j - j0]] = uint16_t(meta[j]);
          }
        }
      }
      uint4* zero = reinterpret_cast<uint4*>(smem + S::WH) + (parity ^ 1) * WARPS * RADIX / 4;
      for (int i = tid; i < WARPS * RADIX / 4; i += THREADS) zero[i] = make_uint4(0u, 0u, 0u, 0u);
      // every CTA's counts have landed and the stage is complete
      cluster_sync_all();
      uint32_t total = 0u, below = 0u;
      if (tid < RADIX) {
#pragma unroll
        for (uint32_t q = 0; q < S::MAX_CL; ++q) {
          const uint32_t x = q < ncta ? s_cnt[q * RADIX + tid] : 0u;
          total += x;
          if (q < rank) below += x;
        }
      }
      const uint32_t start = scan(total);
      // staged key i of digit d goes to global position s_base[d] + i
      if (tid < RADIX) s_base[tid] = start + below - lstart;
      __syncthreads();
      // ---- 3. remote stores of the staged runs into the owners' destination buffers
      K* kd = reinterpret_cast<K*>(smem + S::KEYS) + (src ^ 1) * S::SLICE;
      uint16_t* id = reinterpret_cast<uint16_t*>(smem + S::IDX) + (src ^ 1) * S::SLICE;
#pragma unroll 4
      for (uint32_t i = tid; i < len; i += THREADS) {
        const K k = ks[i];
        const uint32_t g = s_base[digit_of(k, shift, mask)] + i;
        const uint32_t owner = __umulhi(g, magic), at = g - owner * slice;
        st_cluster(map_shared(kd + at, owner), k);
        if constexpr (INDEX) st_cluster(map_shared(id + at, owner), is[i]);
      }
      // ---- 4. the destination buffers are complete
      cluster_sync_all();
      src ^= 1;
    }

    // in order?  Each CTA checks its slice and, against the next one's first
    // key, its end; every CTA learns every CTA's finding
    const K* ks = reinterpret_cast<const K*>(smem + S::KEYS) + src * S::SLICE;
    const uint16_t* is = reinterpret_cast<const uint16_t*>(smem + S::IDX) + src * S::SLICE;
    if (tid == 0) {
      const uint64_t first = len ? uint64_t(ks[0] & looked) : ~uint64_t(0);
      s_edge[0] = uint32_t(first);
      s_edge[1] = uint32_t(first >> 32);
      s_edge[2] = INDEX && len ? is[0] : 0xffffu;
    }
    bool bad = false;
    for (uint32_t i = tid; i + 1u < len; i += THREADS) {
      const K a = ks[i] & looked, b = ks[i + 1] & looked;
      if constexpr (INDEX) bad = bad || a > b || (a == b && is[i] > is[i + 1]);
      else bad = bad || a > b;
    }
    cluster_sync_all();
    if (tid == 0 && len && rank + 1u < ncta) {
      const uint64_t last = uint64_t(ks[len - 1u] & looked);
      const uint64_t next = uint64_t(ld_cluster_u32(map_shared(s_edge, rank + 1u))) |
                            uint64_t(ld_cluster_u32(map_shared(s_edge + 1, rank + 1u))) << 32;
      const uint32_t next_i = ld_cluster_u32(map_shared(s_edge + 2, rank + 1u));
      bad = bad || last > next || (INDEX && last == next && is[len - 1u] > next_i);
    }
    const int any = __syncthreads_or(bad);
    if (uint32_t(tid) < ncta)
      st_cluster(map_shared(s_flags + rank, uint32_t(tid)), uint32_t(any != 0));
    cluster_sync_all();
    uint32_t found = 0u;
    for (uint32_t q = 0; q < ncta; ++q) found |= s_flags[q];
    if (!found) break;  // the same in every CTA
    if (!careful && rank == 0u && tid == 0) count_repair(order);
  }

  // write this CTA's slice out (untransformed): everything is read before the
  // first write
  const K* ks = reinterpret_cast<const K*>(smem + S::KEYS) + src * S::SLICE;
  [[maybe_unused]] const uint16_t* is =
      reinterpret_cast<const uint16_t*>(smem + S::IDX) + src * S::SLICE;
  V v[VB > 0 ? ITEMS : 1];
  if constexpr (VB > 0) {
#pragma unroll
    for (int j = 0; j < ITEMS; ++j) {
      const uint32_t i = uint32_t(j * THREADS + tid);
      if (i < len) v[j] = vals[is[i]];
    }
    cluster_sync_all();
  }
#pragma unroll
  for (int j = 0; j < ITEMS; ++j) {
    const uint32_t i = uint32_t(j * THREADS + tid);
    if (i < len && dbg_ok(base0 + i, n, kSiteClusterOut)) {
      keys[base0 + i] = xf.on ? xf_inv(ks[i], xf) : ks[i];
      if constexpr (VB > 0) vals[base0 + i] = v[j];
    }
  }
  if (ctrl != nullptr) {
    __syncthreads();
    if (tid == 0) atomicMax(&ctrl->t_upsweep, stat_now(ctrl));
  }
}

}  // namespace rs
