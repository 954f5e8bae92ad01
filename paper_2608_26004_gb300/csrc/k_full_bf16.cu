// Instantiations of the recording row kernel and its decision kernel for
// bf16 logits.
#include "kernel_full.cuh"
#include "kernels.h"

namespace asymspec_impl {

const void* full_kernel_bf16(bool stoch, bool edge) {
  if (stoch)
    return edge ? reinterpret_cast<const void*>(&fuse_verify_full<__nv_bfloat16, true, true>)
                : reinterpret_cast<const void*>(&fuse_verify_full<__nv_bfloat16, true, false>);
  return edge ? reinterpret_cast<const void*>(&fuse_verify_full<__nv_bfloat16, false, true>)
              : reinterpret_cast<const void*>(&fuse_verify_full<__nv_bfloat16, false, false>);
}

const void* decide_full_bf16(bool stoch, bool edge) {
  if (stoch)
    return edge ? reinterpret_cast<const void*>(&decide_full<__nv_bfloat16, true, true>)
                : reinterpret_cast<const void*>(&decide_full<__nv_bfloat16, true, false>);
  return edge ? reinterpret_cast<const void*>(&decide_full<__nv_bfloat16, false, true>)
              : reinterpret_cast<const void*>(&decide_full<__nv_bfloat16, false, false>);
}

}  // namespace asymspec_impl
