// The reduction kernel for D = 0: columns of any dimension.
#include "rips_reduce.cuh"

namespace rips {

const void* reduce_kernel_d0() { return (const void*)reduce_persistent_kernel<0>; }

}  // namespace rips
