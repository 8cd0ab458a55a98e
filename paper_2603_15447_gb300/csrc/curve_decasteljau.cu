// curve_decasteljau.cu -- instantiates the decasteljau register evaluator (see curve_tile.cuh).
#include "curve_tile.cuh"

namespace bez {
LaunchResult launch_curve_decasteljau(const CurveArgs& a, int tm, int om, cudaStream_t s, const LaunchHooks& h)
{
    return launch_curve_variant<VAR_DECASTELJAU>(a, tm, om, s, h);
}
}  // namespace bez
