// Instantiations of the streaming row kernel and its decision kernel for
// fp32 logits.
#include "kernel_row.cuh"
#include "kernels.h"

namespace asymspec_impl {

const void* row_kernel_f32(bool stoch, bool edge) {
  if (stoch)
    return edge ? reinterpret_cast<const void*>(&fuse_verify_row<float, true, true>)
                : reinterpret_cast<const void*>(&fuse_verify_row<float, true, false>);
  return edge ? reinterpret_cast<const void*>(&fuse_verify_row<float, false, true>)
              : reinterpret_cast<const void*>(&fuse_verify_row<float, false, false>);
}

const void* decide_blocks_f32(bool stoch, bool edge) {
  if (stoch)
    return edge ? reinterpret_cast<const void*>(&decide_blocks<float, true, true>)
                : reinterpret_cast<const void*>(&decide_blocks<float, true, false>);
  return edge ? reinterpret_cast<const void*>(&decide_blocks<float, false, true>)
              : reinterpret_cast<const void*>(&decide_blocks<float, false, false>);
}

}  // namespace asymspec_impl
