// spline_fused_high.cu -- instantiates the fused spline kernels of degrees 4 and
// 5 (see spline_fused.cuh), apart from the others to compile beside them.
#include "spline_fused.cuh"

namespace bez {
const void* fused_kernel_high(int degree, int dim, bool rat)
{
    return degree == 4 ? fused_kernel<4>(dim, rat) : fused_kernel<5>(dim, rat);
}
}  // namespace bez
