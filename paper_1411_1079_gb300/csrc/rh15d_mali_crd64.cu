// rh15d_mali_crd64.cu -- column kernels: FP64, linear solver, complete redistribution.
#include "rh15d_mali.cuh"

namespace rh {

const void *mali_kernel_crd64(bool cache)
{
    using namespace mali;
    return cache ? (const void *)mali_kernel<double, false, true, false>
                 : (const void *)mali_kernel<double, false, false, false>;
}

}  // namespace rh
