// Instantiations of the cross-family row kernel and its decision kernel for
// bf16 logits.
#include "kernel_xrow.cuh"
#include "kernels.h"

namespace asymspec_impl {

const void* xrow_kernel_bf16(bool stoch) {
  return stoch ? reinterpret_cast<const void*>(&fuse_verify_xrow<__nv_bfloat16, true>)
               : reinterpret_cast<const void*>(&fuse_verify_xrow<__nv_bfloat16, false>);
}

const void* decide_xrow_bf16(bool stoch) {
  return stoch ? reinterpret_cast<const void*>(&decide_xrow<__nv_bfloat16, true>)
               : reinterpret_cast<const void*>(&decide_xrow<__nv_bfloat16, false>);
}

}  // namespace asymspec_impl
