// rh15d_mali_prd64.cu -- column kernels: FP64, partial redistribution, linear and Bezier solvers.
#include "rh15d_mali.cuh"

namespace rh {

const void *mali_kernel_prd64(bool bez)
{
    using namespace mali;
    return bez ? (const void *)mali_kernel<double, true, true, true>
               : (const void *)mali_kernel<double, true, true, false>;
}

}  // namespace rh
