// rh15d_mali_crd32.cu -- column kernels: FP32 sweep, linear solver, complete redistribution.
#include "rh15d_mali.cuh"

namespace rh {

const void *mali_kernel_crd32(bool cache)
{
    using namespace mali;
    return cache ? (const void *)mali_kernel<float, false, true, false>
                 : (const void *)mali_kernel<float, false, false, false>;
}

}  // namespace rh
