// The reduction kernel for D = 3: columns are tetrahedra.
#include "rips_reduce.cuh"

namespace rips {

const void* reduce_kernel_d3() { return (const void*)reduce_persistent_kernel<3>; }

}  // namespace rips
