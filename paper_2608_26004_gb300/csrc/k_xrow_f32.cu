// Instantiations of the cross-family row kernel and its decision kernel for
// fp32 logits.
#include "kernel_xrow.cuh"
#include "kernels.h"

namespace asymspec_impl {

const void* xrow_kernel_f32(bool stoch) {
  return stoch ? reinterpret_cast<const void*>(&fuse_verify_xrow<float, true>)
               : reinterpret_cast<const void*>(&fuse_verify_xrow<float, false>);
}

const void* decide_xrow_f32(bool stoch) {
  return stoch ? reinterpret_cast<const void*>(&decide_xrow<float, true>)
               : reinterpret_cast<const void*>(&decide_xrow<float, false>);
}

}  // namespace asymspec_impl
