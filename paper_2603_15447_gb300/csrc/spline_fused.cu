// spline_fused.cu -- launch of the fused spline kernels (see spline_fused.cuh),
// and their instances for degrees 1 to 3.
#include "spline_fused.cuh"

namespace bez {

bool spline_fits_fused(const SplineArgs& a)
{
    // (a block per curve at worst: the curves have to fit a grid)
    if (a.degree > kFusedMaxDegree || a.n_ctrl > 100000 || a.n_curves > 2147483647) return false;
    const FusedLayout f = fused_layout(1, a.n_ctrl, a.degree, a.dim, a.weights != nullptr, a.knots != nullptr);
    return (size_t)f.total * sizeof(float) <= kFusedMaxSmem;
}

LaunchResult launch_spline_fused(const SplineArgs& a, int tm, int om, cudaStream_t s, const LaunchHooks& h)
{
    const bool rat = a.weights != nullptr, knots = a.knots != nullptr;
    const void* kern = a.degree == 1   ? fused_kernel<1>(a.dim, rat)
                       : a.degree == 2 ? fused_kernel<2>(a.dim, rat)
                       : a.degree == 3 ? fused_kernel<3>(a.dim, rat)
                                       : fused_kernel_high(a.degree, a.dim, rat);
    // as many curves as give every thread a span, fewer when that leaves the
    // SMs short of blocks (8 each) or does not fit
    int cb = kFusedThreads / a.n_spans;
    cb = cb < 1 ? 1 : cb;
    const int64_t target = (int64_t)h.sm_count * 8;
    while (cb > 1 && (a.n_curves + cb - 1) / cb < target) cb = (cb + 1) / 2;
    while (cb > 1 && (size_t)fused_layout(cb, a.n_ctrl, a.degree, a.dim, rat, knots).total * sizeof(float) >
                         kFusedMaxSmem / 2)
        cb = (cb + 1) / 2;
    int64_t parts = 1, part_len = 0;
    if (cb == 1 && om == OM_POINTS && a.n_curves < target) {
        const int64_t tiles = ((int64_t)a.n_t + kFusedThreads * kFusedRun - 1) / (kFusedThreads * kFusedRun);
        const int64_t want = (target + a.n_curves - 1) / a.n_curves;
        const int64_t per = want >= tiles ? 1 : tiles / want;
        part_len = per * kFusedThreads * kFusedRun;
        parts = ((int64_t)a.n_t + part_len - 1) / part_len;
    }
    const int64_t blocks = (a.n_curves + cb - 1) / cb * parts;
    if (blocks > 2147483647) return {0, cudaErrorInvalidConfiguration};
    const size_t smem = (size_t)fused_layout(cb, a.n_ctrl, a.degree, a.dim, rat, knots).total * sizeof(float);
    int iparts = (int)parts;
    uint32_t ulen = (uint32_t)part_len;
    void* args[] = {(void*)&a, (void*)&tm, (void*)&om, (void*)&cb, (void*)&iparts, (void*)&ulen};
    h.count(h.self);
    h.begin(h.self, s);
    const cudaError_t e = cudaLaunchKernel(kern, dim3((unsigned)blocks), dim3(kFusedThreads), args, smem, s);
    h.end(h.self, s);
    return {1, e};
}

}  // namespace bez
