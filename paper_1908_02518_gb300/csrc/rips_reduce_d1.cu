// The reduction kernel for D = 1: columns are edges.
#include "rips_reduce.cuh"

namespace rips {

const void* reduce_kernel_d1() { return (const void*)reduce_persistent_kernel<1>; }

}  // namespace rips
