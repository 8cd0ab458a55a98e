// grad.cu -- launch of the adjoint kernels (see grad.cuh), and their instances
// for 3D points and runtime degrees.
#include "grad.cuh"

namespace bez {

LaunchResult launch_grad(const GradArgs& a, cudaStream_t s, const LaunchHooks& h)
{
    const bool rat = a.weights != nullptr;
    const void* kern = a.dim != 3 ? grad_kernel_dims(a.degree, a.dim, rat)
                       : rat      ? grad_kernel_dim<3, true>(a.degree)
                                  : grad_kernel_dim<3, false>(a.degree);
    if (!kern) kern = rat ? (const void*)k_grad<0, 0, true> : (const void*)k_grad<0, 0, false>;
    const size_t smem = (a.t_stride == 0 && a.grad_t && a.shared_gt) ? (size_t)a.n_t * sizeof(float) : 0;
    const int grid = persistent_grid(kern, kWarps * 32, smem, h.sm_count, (a.n_curves + kWarps - 1) / kWarps);
    void* args[] = {(void*)&a};
    h.count(h.self);
    h.begin(h.self, s);
    cudaError_t e = cudaLaunchKernel(kern, dim3(grid), dim3(kWarps * 32), args, smem, s);
    h.end(h.self, s);
    return {1, e};
}

}  // namespace bez
