// RK4 stage kernels of small boxes with 2 lanes per point.
#include "grf_team.cuh"

namespace grf {
void launch_stage_team2(int stage, cudaStream_t st, const Geom& g, const Coeffs& c, const StageArgs& a) {
    launch_team<2>(stage, st, g, c, a);
}
}  // namespace grf
