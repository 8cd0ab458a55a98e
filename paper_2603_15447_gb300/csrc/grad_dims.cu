// grad_dims.cu -- instantiates the adjoint kernels of 1D, 2D and 4D points (see
// grad.cuh).
#include "grad.cuh"

namespace bez {

template <bool RAT>
static const void* pick(int degree, int dim)
{
    return dim == 1 ? grad_kernel_dim<1, RAT>(degree)
           : dim == 2 ? grad_kernel_dim<2, RAT>(degree)
                      : grad_kernel_dim<4, RAT>(degree);
}

const void* grad_kernel_dims(int degree, int dim, bool rat)
{
    return rat ? pick<true>(degree, dim) : pick<false>(degree, dim);
}

}  // namespace bez
