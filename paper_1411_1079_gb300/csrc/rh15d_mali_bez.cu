// rh15d_mali_bez.cu -- column kernels: Bezier solver, complete redistribution.
#include "rh15d_mali.cuh"

namespace rh {

const void *mali_kernel_bez(int precision)
{
    using namespace mali;
    return precision == 1 ? (const void *)mali_kernel<float, false, true, true>
                          : (const void *)mali_kernel<double, false, true, true>;
}

}  // namespace rh
