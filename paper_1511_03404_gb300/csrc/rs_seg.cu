// Host side of the batched segmented sort (each of the four data types):
// workspace sizing and the launch sequence memset -> k_seg_plan ->
// k_seg_small (short, then medium) -> k_seg_hist -> k_seg_persistent, all on
// the caller's stream (capturable in a CUDA graph).
#include <algorithm>

#include "../../include/rs.h"
#include "rs_host.h"
#include "rs_segmented.cuh"

namespace rs {

namespace {

// MINB: resident CTAs per SM the short-segment kernel is compiled for (its
// register budget); PASS_MINB: the same for the pass kernel.
template <class K, int VB, int R, int THREADS, int ITEMS, int CHUNK_TILES, int SMALL_ITEMS,
          int MEDIUM_ITEMS, int MINB, int PASS_MINB>
struct SegSort {
  using C = SegKernelCfg<K, VB, R, THREADS, ITEMS, CHUNK_TILES, SMALL_ITEMS>;
  static constexpr int PLAN_THREADS = 256, MEDIUM_THREADS = 1024;

  static SegLayout layout(size_t n, size_t nseg, int passes) {
    return seg_layout(n, nseg, passes, R, C::TILE, C::CHUNK);
  }

  static cudaError_t run(void* keys, void* vals, void* keys_alt, void* vals_alt, size_t n,
                         const uint64_t* d_off, size_t nseg, int begin_bit, int end_bit,
                         void* ws, cudaStream_t s, Knobs knobs) {
    const int passes = num_passes(begin_bit, end_bit, R);
    const SegLayout L = layout(n, nseg, passes);
    char* w = static_cast<char*>(ws);
    Ctrl* ctrl = reinterpret_cast<Ctrl*>(w);
    cudaError_t e = cudaMemsetAsync(w, 0, sizeof(Ctrl), s);
    if (e != cudaSuccess) return e;
    // short segments: one CTA each, before the persistent kernel
    auto small = &k_seg_small<K, VB, R, THREADS, SMALL_ITEMS, true, MINB>;
    int smem_small = SmallSmem<K, VB, R, THREADS, SMALL_ITEMS, true>::BYTES;
    if constexpr (VB == 0) {
      if (begin_bit == 0 && end_bit == 8 * int(sizeof(K))) {  // whole keys need no positions
        small = &k_seg_small<K, VB, R, THREADS, SMALL_ITEMS, false, MINB>;
        smem_small = SmallSmem<K, VB, R, THREADS, SMALL_ITEMS, false>::BYTES;
      }
    }
    const int occ_small = prepare_kernel(reinterpret_cast<const void*>(small), THREADS, smem_small);
    if (occ_small <= 0) return cudaErrorInvalidConfiguration;
    auto medium = &k_seg_small<K, VB, R, MEDIUM_THREADS, MEDIUM_ITEMS, true, 1, true>;
    int smem_medium = SmallSmem<K, VB, R, MEDIUM_THREADS, MEDIUM_ITEMS, true>::BYTES;
    if constexpr (VB == 0) {
      if (begin_bit == 0 && end_bit == 8 * int(sizeof(K))) {
        medium = &k_seg_small<K, VB, R, MEDIUM_THREADS, MEDIUM_ITEMS, false, 1, true>;
        smem_medium = SmallSmem<K, VB, R, MEDIUM_THREADS, MEDIUM_ITEMS, false>::BYTES;
      }
    }
    const int occ_medium =
        prepare_kernel(reinterpret_cast<const void*>(medium), MEDIUM_THREADS, smem_medium);
    if (occ_medium <= 0) return cudaErrorInvalidConfiguration;
    auto hist = &k_seg_hist<K, R, C::HIST_THREADS, C::MAXP, C::HIST_SLOTS, C::CHUNK, C::TILE,
                            CHUNK_TILES, C::HIST_MINB>;
    const int occ_hist =
        prepare_kernel(reinterpret_cast<const void*>(hist), C::HIST_THREADS, C::HIST_BYTES);
    if (occ_hist <= 0) return cudaErrorInvalidConfiguration;
    auto kern = &k_seg_persistent<K, VB, R, THREADS, ITEMS, CHUNK_TILES, PASS_MINB, true>;
    int smem = C::BYTES;
    if constexpr (VB == 0) {
      if (begin_bit == 0 && end_bit == 8 * int(sizeof(K))) {  // whole keys: staged themselves
        kern = &k_seg_persistent<K, VB, R, THREADS, ITEMS, CHUNK_TILES, PASS_MINB, false>;
        smem = SegKernelCfg<K, VB, R, THREADS, ITEMS, CHUNK_TILES, SMALL_ITEMS, false>::BYTES;
      }
    }
    const int occ = prepare_kernel(reinterpret_cast<const void*>(kern), THREADS, smem);
    if (occ <= 0) return cudaErrorInvalidConfiguration;
    SegArgs a;
    a.off = d_off;
    a.begin_bit = begin_bit;
    a.end_bit = end_bit;
    a.passes = passes;
    a.ctrl = ctrl;
    a.small_ids = reinterpret_cast<const uint32_t*>(w + L.small_ids);
    a.medium_ids = reinterpret_cast<const uint32_t*>(w + L.medium_ids);
    a.descs = reinterpret_cast<const SegDesc*>(w + L.descs);
    a.tdesc = reinterpret_cast<TileDesc*>(w + L.tdesc);
    a.chunk_seg = reinterpret_cast<const uint32_t*>(w + L.chunk_seg);
    a.state = reinterpret_cast<uint32_t*>(w + L.state);
    a.counts = reinterpret_cast<uint32_t*>(w + L.counts);
    a.offsets = reinterpret_cast<uint32_t*>(w + L.offsets);
    a.status = reinterpret_cast<uint32_t*>(w + L.status);
    a.tiles_max = L.tiles_max;
    a.nseg = nseg;
    a.knobs = knobs;
    using V = ValT<VB>;
    k_seg_plan<PLAN_THREADS, C::RADIX>
        <<<unsigned((nseg + PLAN_THREADS - 1) / PLAN_THREADS), PLAN_THREADS, 0, s>>>(
            n, uint32_t(C::SMALL_TILE), uint32_t(MEDIUM_THREADS * MEDIUM_ITEMS), uint32_t(C::TILE),
            uint32_t(C::CHUNK), L.chunks_max, reinterpret_cast<uint32_t*>(w + L.small_ids),
            reinterpret_cast<uint32_t*>(w + L.medium_ids),
            reinterpret_cast<SegDesc*>(w + L.descs),
            reinterpret_cast<uint32_t*>(w + L.chunk_seg), a);
    e = cudaGetLastError();
    if (e != cudaSuccess) return e;
    // grids no larger than the work can be: at most tiles_max pass tiles per
    // pass and chunks_max histogram chunks (bounds the host knows without
    // the plan), so that a small batch does not spread idle CTAs over every
    // SM while other streams' kernels want them
    const size_t sms = size_t(device_info().sms);
    const unsigned grid = unsigned(std::max<size_t>(
        1, std::min<size_t>(sms * occ, size_t(passes) * L.tiles_max)));
    const unsigned grid_hist =
        unsigned(std::max<size_t>(1, std::min<size_t>(sms * occ_hist, L.chunks_max)));
    const unsigned grid_small =
        unsigned(std::max<size_t>(1, std::min<size_t>(nseg, sms * occ_small)));
    const unsigned grid_medium = unsigned(std::max<size_t>(
        1, std::min<size_t>(sms * occ_medium, n / (size_t(C::SMALL_TILE) + 1))));
    prof_before(s);
    // each kernel waits for the one before it (pdl_wait), so that it may be
    // launched as that one exits
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
      if (e == cudaSuccess) e = cudaLaunchKernelEx(&cfg, kernel, args...);
    };
    K *k0 = static_cast<K*>(keys), *k1 = static_cast<K*>(keys_alt);
    V *v0 = static_cast<V*>(vals), *v1 = static_cast<V*>(vals_alt);
    launch(small, grid_small, THREADS, smem_small, k0, v0, k1, v1, a);
    // (no segment is longer than the array)
    if (n > size_t(C::SMALL_TILE))
      launch(medium, grid_medium, MEDIUM_THREADS, smem_medium, k0, v0, k1, v1, a);
    if (n > size_t(MEDIUM_THREADS) * MEDIUM_ITEMS) {
      launch(hist, grid_hist, C::HIST_THREADS, passes * C::RADIX * C::HIST_SLOTS * 4,
             static_cast<const K*>(k0), a);
      launch(kern, grid, THREADS, smem, k0, v0, k1, v1, a);
    }
    if (e == cudaSuccess) e = cudaGetLastError();
    prof_after(s, RS_KERNEL_SEGMENTED,
               double(n) * (sizeof(K) + passes * 2.0 * (sizeof(K) + VB)));
    return e;
  }
};

// Short segments are sorted by a CTA of 256 threads up to 256 x SMALL_ITEMS
// elements, medium ones by one of 1024 threads up to 1024 x MEDIUM_ITEMS (its
// counters, keys and positions fill the shared memory of an SM), longer ones in
// passes over tiles of 256 x ITEMS, two CTAs an SM.  The lines lie where the
// next form becomes the faster one: 20,000 log-uniform segments of 2^26 u32
// pairs / keys take 1405 / 1048 us with medium segments up to 16 items a
// thread, 1363 / 1004 up to 20, 1403 / 1052 up to 24; of 2^25 u64 pairs / keys
// 2049 / 1666 up to 8, 1827 / 1441 up to 12, 1715 / 1372 up to 16.  10,000 rows
// of up to 3,000 u64 pairs / keys take 773 / 664 us with short segments up to
// 8 items a thread, 489 / 366 up to 12, 510 / 390 up to 16; rows of up to
// 2,047 take 364 / 285, 388 / 298 and 413 / 320, for the registers; u32 ones
// are the same at 16 and 24.
using SegU32Pairs = SegSort<uint32_t, 4, 8, 256, 41, 12, 16, 20, 4, 2>;
using SegU32Keys = SegSort<uint32_t, 0, 8, 256, 45, 14, 16, 20, 4, 2>;
using SegU64Keys = SegSort<uint64_t, 0, 8, 256, 23, 24, 12, 16, 4, 2>;
using SegU64Pairs = SegSort<uint64_t, 8, 8, 256, 23, 24, 12, 16, 3, 2>;

bool seg_types(int kb, int vb) { return (kb == 4 || kb == 8) && (vb == 0 || vb == kb); }

SegLayout seg_layout_for(int kb, int vb, size_t n, size_t nseg, int passes) {
  if (kb == 4) return vb ? SegU32Pairs::layout(n, nseg, passes) : SegU32Keys::layout(n, nseg, passes);
  return vb ? SegU64Pairs::layout(n, nseg, passes) : SegU64Keys::layout(n, nseg, passes);
}

cudaError_t seg_run(int kb, int vb, void* keys, void* vals, void* keys_alt, void* vals_alt,
                    size_t n, const uint64_t* d_off, size_t nseg, int begin_bit, int end_bit,
                    void* ws, cudaStream_t s, Knobs knobs) {
  if (kb == 4 && vb)
    return SegU32Pairs::run(keys, vals, keys_alt, vals_alt, n, d_off, nseg, begin_bit, end_bit,
                            ws, s, knobs);
  if (kb == 4)
    return SegU32Keys::run(keys, vals, keys_alt, vals_alt, n, d_off, nseg, begin_bit, end_bit,
                           ws, s, knobs);
  if (vb)
    return SegU64Pairs::run(keys, vals, keys_alt, vals_alt, n, d_off, nseg, begin_bit, end_bit,
                            ws, s, knobs);
  return SegU64Keys::run(keys, vals, keys_alt, vals_alt, n, d_off, nseg, begin_bit, end_bit, ws,
                         s, knobs);
}

}  // namespace

Knobs knobs_now();

}  // namespace rs

using namespace rs;

extern "C" {

rs_status rs_segmented_workspace_bytes_typed(int key_bytes, int val_bytes, size_t n, size_t n_seg,
                                             int begin_bit, int end_bit, size_t* bytes) {
  if (!bytes || !seg_types(key_bytes, val_bytes)) return RS_ERR_INVALID;
  if (begin_bit < 0 || begin_bit > end_bit || end_bit > 8 * key_bytes) return RS_ERR_INVALID;
  if (n >= (size_t(1) << 40) || n_seg >= (size_t(1) << 31)) return RS_ERR_INVALID;
  *bytes = 0;
  if (n == 0 || n_seg == 0 || begin_bit == end_bit) return RS_OK;
  const SegLayout L =
      seg_layout_for(key_bytes, val_bytes, n, n_seg, num_passes(begin_bit, end_bit, 8));
  if (L.tiles_max >= (size_t(1) << 32)) return RS_ERR_INVALID;
  *bytes = L.total;
  return RS_OK;
}

rs_status rs_segmented_sort(int key_bytes, int val_bytes, void* keys, void* vals, void* keys_alt,
                            void* vals_alt, size_t n, const uint64_t* d_offsets, size_t n_seg,
                            int begin_bit, int end_bit, void* ws, size_t ws_bytes,
                            rs_stream_t stream, int* result_in_alt) {
  if (!result_in_alt) return RS_ERR_INVALID;
  *result_in_alt = 0;
  size_t need = 0;
  rs_status st = rs_segmented_workspace_bytes_typed(key_bytes, val_bytes, n, n_seg, begin_bit,
                                                    end_bit, &need);
  if (st != RS_OK) return st;
  if (n == 0 || n_seg == 0 || begin_bit == end_bit) return RS_OK;
  if (!keys || !keys_alt || !d_offsets || keys == keys_alt) return RS_ERR_INVALID;
  if ((val_bytes != 0) != (vals != nullptr && vals_alt != nullptr)) return RS_ERR_INVALID;
  if (val_bytes == 0 && (vals || vals_alt)) return RS_ERR_INVALID;
  if (val_bytes && vals == vals_alt) return RS_ERR_INVALID;
  auto al = [](const void* p, size_t a) { return reinterpret_cast<uintptr_t>(p) % a == 0; };
  if (!al(keys, key_bytes) || !al(keys_alt, key_bytes) || !al(d_offsets, 8)) return RS_ERR_INVALID;
  if (val_bytes && (!al(vals, val_bytes) || !al(vals_alt, val_bytes))) return RS_ERR_INVALID;
  if (!ws || ws_bytes < need || !al(ws, 256)) return RS_ERR_WORKSPACE;
  const int passes = num_passes(begin_bit, end_bit, 8);
  const cudaError_t e = seg_run(key_bytes, val_bytes, keys, vals, keys_alt, vals_alt, n,
                                d_offsets, n_seg, begin_bit, end_bit, ws,
                                reinterpret_cast<cudaStream_t>(stream), knobs_now());
  if (e != cudaSuccess) return RS_ERR_CUDA;
  *result_in_alt = passes & 1;
  return RS_OK;
}


rs_status rs_segmented_workspace_bytes(size_t n, size_t n_seg, int begin_bit, int end_bit,
                                       size_t* bytes) {
  return rs_segmented_workspace_bytes_typed(4, 4, n, n_seg, begin_bit, end_bit, bytes);
}

rs_status rs_segmented_sort_pairs(uint32_t* keys, uint32_t* vals, uint32_t* keys_alt,
                                  uint32_t* vals_alt, size_t n, const uint64_t* d_offsets,
                                  size_t n_seg, int begin_bit, int end_bit, void* ws,
                                  size_t ws_bytes, rs_stream_t stream, int* result_in_alt) {
  if (n > 0 && n_seg > 0 && begin_bit != end_bit && (!vals || !vals_alt)) return RS_ERR_INVALID;
  return rs_segmented_sort(4, 4, keys, vals, keys_alt, vals_alt, n, d_offsets, n_seg, begin_bit,
                           end_bit, ws, ws_bytes, stream, result_in_alt);
}

}  // extern "C"
