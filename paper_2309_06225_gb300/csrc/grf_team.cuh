// RK4 stage kernel for small boxes (4th-order scheme): a team of 4 or 2 lanes per point.
//
// A launch of a few warps per SM is bound by the latency of one warp, and the integer code of the gather is
// the larger part of that. Here the lanes of a team each gather a share of the point's fields into shared
// memory and then all evaluate the point's equations (the FP64 pipe is idle enough), so that the gather takes
// a quarter or half of the time. The operations on each value are those of rk4_stage_kernel, and so are the bits.
// 16^3 step: 0.66 ms with one lane a point, 0.53 with 2, 0.46 with 4; 20^3: 0.69, 0.55, 0.68 (the FP64 work of a
// point is done once a lane, so 4 lanes pay only while a scheduler has one warp at most).
#pragma once

#include "grf_kernels.cuh"
#include "grf_launch.h"

namespace grf {

template <int LOP>
struct TeamPoint {
    PointIn in;
    double kos[NFIELDS], adv[LOP ? NFIELDS : 1];
};

// Blocks of one warp: 32 / TEAM points.
template <int TEAM, int STAGE, int LOP>
__global__ void __launch_bounds__(32) rk4_stage_team_kernel(Geom g, Coeffs c, StageArgs a) {
    __shared__ TeamPoint<LOP> team[32 / TEAM];
    const int t = threadIdx.x % TEAM;
    TeamPoint<LOP>& P = team[threadIdx.x / TEAM];
    const long long q = a.q0 + (long long)blockIdx.x * (32 / TEAM) + threadIdx.x / TEAM;
    const bool live = q < a.q1;
    int i, j, k;
    point_of(g, live ? q : a.q1 - 1, i, j, k);  // idle teams of the last block follow its last point
    const long long p = gidx(g, i + NG, j + NG, k + NG);
    gather<LOP, 1, TEAM>(g, a.src, p, P.in, P.kos, P.adv, t);
    __syncwarp();
    double r[NFIELDS];
    bool ok = true;
    point_rhs<double, double, -1, LOP, 1>(c, P.in, r, nullptr, ok, P.adv);
    if (!ok && t == 0) atomicOr(a.status, 1);
    // Every lane forms all output values (enforcement needs them together) and stores its share; the accumulator
    // is read and written by the field's own lane, but for the last stage, which only reads it.
#pragma unroll 1
    for (int f = 0; f < NFIELDS; ++f) {
        const long long o = f * g.fstride + p;
        const double kf = fma(a.ko, P.kos[f], r[f]);
        const double unf = (STAGE == 0) ? P.in.v[f] : a.un[o];
        if (STAGE == 3 || (live && f % TEAM == t)) r[f] = rk4_value<STAGE>(a, o, kf, unf);
        else r[f] = fma(STAGE == 2 ? a.dt : 0.5 * a.dt, kf, unf);
    }
    if (a.enforce) enforce_point(r, a.min_chi, a.min_lapse);
    __syncwarp();  // the last stage's output is the state u_n that the other lanes read
    if (!live) return;
#pragma unroll 1
    for (int f = t; f < NFIELDS; f += TEAM) store_with_images(g, a.dst, f, i, j, k, r[f]);
}

template <int TEAM>
void launch_team(int stage, cudaStream_t st, const Geom& g, const Coeffs& c, const StageArgs& a) {
    const unsigned blocks = point_blocks(a.q1 - a.q0, 32 / TEAM);
    if (c.advection) {
        switch (stage) {
            case 0: rk4_stage_team_kernel<TEAM, 0, kLopsided><<<blocks, 32, 0, st>>>(g, c, a); break;
            case 1: rk4_stage_team_kernel<TEAM, 1, kLopsided><<<blocks, 32, 0, st>>>(g, c, a); break;
            case 2: rk4_stage_team_kernel<TEAM, 2, kLopsided><<<blocks, 32, 0, st>>>(g, c, a); break;
            default: rk4_stage_team_kernel<TEAM, 3, kLopsided><<<blocks, 32, 0, st>>>(g, c, a); break;
        }
        return;
    }
    switch (stage) {
        case 0: rk4_stage_team_kernel<TEAM, 0, 0><<<blocks, 32, 0, st>>>(g, c, a); break;
        case 1: rk4_stage_team_kernel<TEAM, 1, 0><<<blocks, 32, 0, st>>>(g, c, a); break;
        case 2: rk4_stage_team_kernel<TEAM, 2, 0><<<blocks, 32, 0, st>>>(g, c, a); break;
        default: rk4_stage_team_kernel<TEAM, 3, 0><<<blocks, 32, 0, st>>>(g, c, a); break;
    }
}
}  // namespace grf
