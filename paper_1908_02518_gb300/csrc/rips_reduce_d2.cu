// The reduction kernel for D = 2: columns are triangles.
#include "rips_reduce.cuh"

namespace rips {

const void* reduce_kernel_d2() { return (const void*)reduce_persistent_kernel<2>; }

}  // namespace rips
