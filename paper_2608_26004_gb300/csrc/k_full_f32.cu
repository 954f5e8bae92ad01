// Instantiations of the recording row kernel and its decision kernel for
// fp32 logits.
#include "kernel_full.cuh"
#include "kernels.h"

namespace asymspec_impl {

const void* full_kernel_f32(bool stoch, bool edge) {
  if (stoch)
    return edge ? reinterpret_cast<const void*>(&fuse_verify_full<float, true, true>)
                : reinterpret_cast<const void*>(&fuse_verify_full<float, true, false>);
  return edge ? reinterpret_cast<const void*>(&fuse_verify_full<float, false, true>)
              : reinterpret_cast<const void*>(&fuse_verify_full<float, false, false>);
}

const void* decide_full_f32(bool stoch, bool edge) {
  if (stoch)
    return edge ? reinterpret_cast<const void*>(&decide_full<float, true, true>)
                : reinterpret_cast<const void*>(&decide_full<float, true, false>);
  return edge ? reinterpret_cast<const void*>(&decide_full<float, false, true>)
              : reinterpret_cast<const void*>(&decide_full<float, false, false>);
}

}  // namespace asymspec_impl
