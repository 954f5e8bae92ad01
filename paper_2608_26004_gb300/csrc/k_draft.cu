// Instantiations of the drafter's draw (see kernel_draft.cuh).
#include "kernel_draft.cuh"
#include "kernels.h"

namespace asymspec_impl {

template <typename T>
const void* draft_pick(bool edge, bool stoch) {
  if (edge)
    return stoch ? reinterpret_cast<const void*>(&draft_kernel<T, true, true>)
                 : reinterpret_cast<const void*>(&draft_kernel<T, true, false>);
  return stoch ? reinterpret_cast<const void*>(&draft_kernel<T, false, true>)
               : reinterpret_cast<const void*>(&draft_kernel<T, false, false>);
}

const void* draft_kernel_ptr(int dtype, bool edge, bool stoch) {
  return dtype == ASYMSPEC_FP32 ? draft_pick<float>(edge, stoch)
                                : draft_pick<__nv_bfloat16>(edge, stoch);
}

}  // namespace asymspec_impl
