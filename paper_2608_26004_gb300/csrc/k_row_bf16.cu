// Instantiations of the streaming row kernel and its decision kernel for
// bf16 logits.
#include "kernel_row.cuh"
#include "kernels.h"

namespace asymspec_impl {

const void* row_kernel_bf16(bool stoch, bool edge) {
  if (stoch)
    return edge ? reinterpret_cast<const void*>(&fuse_verify_row<__nv_bfloat16, true, true>)
                : reinterpret_cast<const void*>(&fuse_verify_row<__nv_bfloat16, true, false>);
  return edge ? reinterpret_cast<const void*>(&fuse_verify_row<__nv_bfloat16, false, true>)
              : reinterpret_cast<const void*>(&fuse_verify_row<__nv_bfloat16, false, false>);
}

const void* decide_blocks_bf16(bool stoch, bool edge) {
  if (stoch)
    return edge ? reinterpret_cast<const void*>(&decide_blocks<__nv_bfloat16, true, true>)
                : reinterpret_cast<const void*>(&decide_blocks<__nv_bfloat16, true, false>);
  return edge ? reinterpret_cast<const void*>(&decide_blocks<__nv_bfloat16, false, true>)
              : reinterpret_cast<const void*>(&decide_blocks<__nv_bfloat16, false, false>);
}

}  // namespace asymspec_impl
