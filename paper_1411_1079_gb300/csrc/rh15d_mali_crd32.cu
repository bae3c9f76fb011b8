// rh15d_mali_crd32.cu -- column kernels: FP32 sweep, linear solver, complete redistribution.
#include "rh15d_mali.cuh"

namespace rh {

const void *mali_kernel_crd32(bool cache, int nv)
{
    using namespace mali;
    if (!cache)
        return nv == 1   ? (const void *)mali_kernel<float, false, false, false, 1>
               : nv == 2 ? (const void *)mali_kernel<float, false, false, false, 2>
                         : (const void *)mali_kernel<float, false, false, false, 3>;
    return nv == 1   ? (const void *)mali_kernel<float, false, true, false, 1>
           : nv == 2 ? (const void *)mali_kernel<float, false, true, false, 2>
                     : (const void *)mali_kernel<float, false, true, false, 3>;
}

}  // namespace rh
