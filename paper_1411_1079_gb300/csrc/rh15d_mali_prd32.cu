// rh15d_mali_prd32.cu -- column kernels: FP32 sweep, partial redistribution, linear solver.
#include "rh15d_mali.cuh"

namespace rh {

const void *mali_kernel_prd32() { return (const void *)mali::mali_kernel<float, true, true, false>; }

}  // namespace rh
