// rh15d_mali_prd32_bez.cu -- column kernels: FP32 sweep, partial redistribution, Bezier solver.
#include "rh15d_mali.cuh"

namespace rh {

const void *mali_kernel_prd32_bez() { return (const void *)mali::mali_kernel<float, true, true, true>; }

}  // namespace rh
