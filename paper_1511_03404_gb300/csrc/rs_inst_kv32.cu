// Compiled variants of the sort for 32-bit key-value pairs.  Index 0 is the
// default multi-CTA shape; the others are candidates for the autotuner
// (tile shape, registers per thread, digit width).
#include "rs_launch.cuh"

namespace rs {

const Variant* variants_kv32(int* count) {
  static const Variant table[] = {
      OnesweepSort<uint32_t, 4, 8, 256, 16, 4>::describe(),
      SmallSort<uint32_t, 4, 8, 512, 16>::describe(),
      OnesweepSort<uint32_t, 4, 8, 256, 12, 4>::describe(),
      OnesweepSort<uint32_t, 4, 8, 256, 20, 3>::describe(),
      OnesweepSort<uint32_t, 4, 7, 256, 16, 4>::describe(),
      SmallSort<uint32_t, 4, 8, 1024, 8>::describe(),
      OnesweepSort<uint32_t, 4, 8, 256, 16, 4, true>::describe(),
      FusedSort<uint32_t, 4, 8, 256, 16, 2>::describe(),
      FusedSort<uint32_t, 4, 8, 256, 8, 3>::describe(),
      ClusterSort<uint32_t, 4, 8, 512, 16, 8>::describe(),
      OnesweepSort<uint32_t, 4, 8, 256, 18, 4, true>::describe(),
      OnesweepSort<uint32_t, 4, 8, 256, 41, 2, true>::describe(),
      OnesweepSort<uint32_t, 4, 8, 256, 26, 3, true>::describe(),
      OnesweepSort<uint32_t, 4, 8, 384, 26, 2, true>::describe(),
      OnesweepSort<uint32_t, 4, 8, 512, 19, 2, true>::describe(),
      ClusterSort<uint32_t, 4, 8, 512, 16, 16>::describe(),
  };
  *count = int(sizeof(table) / sizeof(table[0]));
  return table;
}

}  // namespace rs
