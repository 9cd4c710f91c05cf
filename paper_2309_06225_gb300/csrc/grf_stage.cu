// RK4 stage kernels (the hot path): the routing of a stage to its instantiation, and the default one
// (4th order, centred advection, linear or quadratic coupling), one instantiation per stage.
#include "grf_kernels.cuh"
#include "grf_launch.h"

namespace grf {
void launch_stage(int stage, int k0, int planes, cudaStream_t st, const Geom& g, const Coeffs& c, StageArgs a) {
    const long long nxy = (long long)g.nx * g.ny;
    a.q0 = k0 * nxy;
    a.q1 = (k0 + planes) * nxy;
    const unsigned threads = point_threads(a.q1 - a.q0), blocks = point_blocks(a.q1 - a.q0, threads);
    if (g.ng != NG) {
        launch_stage6(stage, blocks, threads, st, g, c, a);
        return;
    }
    if (team_fits(a.q1 - a.q0, 4)) {
        launch_stage_team4(stage, st, g, c, a);
        return;
    }
    if (team_fits(a.q1 - a.q0, 2)) {
        launch_stage_team2(stage, st, g, c, a);
        return;
    }
    if (c.advection) {
        launch_stage_lopsided(stage, blocks, threads, st, g, c, a);
        return;
    }
    if (c.beta_kind == 2 || c.g3 != 0.0) {  // the exponential coupling or the cubic term: the general instantiation
        launch_stage_general(stage, blocks, threads, st, g, c, a);
        return;
    }
    if (c.decoupled) {
        launch_stage_decoupled(stage, blocks, threads, st, g, c, a);
        return;
    }
    switch (stage) {
        case 0: rk4_stage_kernel<0, 0, 0, 0><<<blocks, threads, 0, st>>>(g, c, a); break;
        case 1: rk4_stage_kernel<1, 0, 0, 0><<<blocks, threads, 0, st>>>(g, c, a); break;
        case 2: rk4_stage_kernel<2, 0, 0, 0><<<blocks, threads, 0, st>>>(g, c, a); break;
        default: rk4_stage_kernel<3, 0, 0, 0><<<blocks, threads, 0, st>>>(g, c, a); break;
    }
}
}  // namespace grf
