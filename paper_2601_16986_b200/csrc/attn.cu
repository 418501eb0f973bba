// The attention kernel's instantiations.
#include "attn_kernel.cuh"

namespace ckv {

AttnKernel attn_of(bool shared, bool track) {
  return track ? (shared ? attn_kernel<true, true> : attn_kernel<false, true>) : (shared ? attn_kernel<true, false> : attn_kernel<false, false>);
}

}  // namespace ckv
