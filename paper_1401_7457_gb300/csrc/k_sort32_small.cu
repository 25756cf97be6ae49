// Onesweep digit pass, 32-bit suffix ids, tiles of 256 threads x 4 items, for
// small collections: a pass over a few hundred tiles is one wave of them, as
// long as one tile takes, and most of that is the 16 ranking turns of a
// 4096-item tile (154k suffixes, two passes:
// build 119 -> 107 us; 303k 142 -> 131; 1.01M 160 -> 170, so larger ones do not).
#include "onesweep.cuh"

namespace cxbwt {

cudaError_t launch_onesweep32_small(const PassArgs& a, int mode, bool wk, bool filter, cudaStream_t st) {
  return onesweep::launch_shape<uint32_t, onesweep::ShapeSmall>(a, mode, wk, filter, st);
}

}  // namespace cxbwt
