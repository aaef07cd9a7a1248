// Compiled variants of the sort for 64-bit keys (keys only).  Index 0 is the
// default multi-CTA shape; the others are candidates for the autotuner.
#include "rs_launch.cuh"

namespace rs {

const Variant* variants_k64(int* count) {
  static const Variant table[] = {
      OnesweepSort<uint64_t, 0, 8, 256, 12, 3>::describe(),
      SmallSort<uint64_t, 0, 8, 512, 16>::describe(),
      OnesweepSort<uint64_t, 0, 8, 256, 16, 3>::describe(),
      OnesweepSort<uint64_t, 0, 8, 256, 8, 4>::describe(),
      SmallSort<uint64_t, 0, 8, 1024, 8>::describe(),
      OnesweepSort<uint64_t, 0, 8, 256, 12, 3, true>::describe(),
      FusedSort<uint64_t, 0, 8, 256, 12, 2>::describe(),
      ClusterSort<uint64_t, 0, 8, 512, 16, 8>::describe(),
      OnesweepSort<uint64_t, 0, 8, 256, 16, 3, true>::describe(),
      OnesweepSort<uint64_t, 0, 8, 256, 25, 2, true>::describe(),
      OnesweepSort<uint64_t, 0, 8, 384, 16, 2, true>::describe(),
      OnesweepSort<uint64_t, 0, 8, 256, 11, 4, true>::describe(),
      OnesweepSort<uint64_t, 0, 8, 512, 11, 2, true>::describe(),
      ClusterSort<uint64_t, 0, 8, 512, 16, 16>::describe(),
      FusedSort<uint64_t, 0, 8, 256, 8, 3>::describe(),
  };
  *count = int(sizeof(table) / sizeof(table[0]));
  return table;
}

}  // namespace rs
