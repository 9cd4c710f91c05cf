// RK4 stage kernels of small boxes with 4 lanes per point.
#include "grf_team.cuh"

namespace grf {
void launch_stage_team4(int stage, cudaStream_t st, const Geom& g, const Coeffs& c, const StageArgs& a) {
    launch_team<4>(stage, st, g, c, a);
}
}  // namespace grf
