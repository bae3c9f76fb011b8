// rh15d_mali_crd32.cu -- column kernels: FP32 sweep, linear solver, complete redistribution.
#include "rh15d_mali.cuh"

namespace rh {

const void *mali_kernel_crd32(bool cache, int np)
{
    using namespace mali;
    if (!cache) return (const void *)mali_kernel<float, false, false, false, 1>;
    return np == 1   ? (const void *)mali_kernel<float, false, true, false, 1>
           : np == 2 ? (const void *)mali_kernel<float, false, true, false, 2>
                     : (const void *)mali_kernel<float, false, true, false, 3>;
}

}  // namespace rh
