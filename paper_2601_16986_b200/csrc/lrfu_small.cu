// Algorithm 1's kernel with CTAs of two warps, every group size.
#include "lrfu_kernel.cuh"

namespace ckv {

cudaError_t lrfu_launch_small(int G, const DecodeParams& p, int npb, int heads, cudaStream_t s) {
  switch (G) {
    case 1: return launch_lrfu<1, LRFU_SMALL>(p, npb, heads, s);
    case 2: return launch_lrfu<2, LRFU_SMALL>(p, npb, heads, s);
    case 3: return launch_lrfu<3, LRFU_SMALL>(p, npb, heads, s);
    case 4: return launch_lrfu<4, LRFU_SMALL>(p, npb, heads, s);
    case 5: return launch_lrfu<5, LRFU_SMALL>(p, npb, heads, s);
    case 6: return launch_lrfu<6, LRFU_SMALL>(p, npb, heads, s);
    case 7: return launch_lrfu<7, LRFU_SMALL>(p, npb, heads, s);
    case 8: return launch_lrfu<8, LRFU_SMALL>(p, npb, heads, s);
  }
  return cudaErrorInvalidValue;
}

}  // namespace ckv
