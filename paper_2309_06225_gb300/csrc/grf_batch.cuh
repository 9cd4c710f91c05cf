// Batched RK4 over many boxes: the box and tile descriptors and the per-tile stage shared by the
// per-stage kernels (grf_batch.cu) and the persistent kernel (grf_batch_persistent.cu), which are
// compiled in separate translation units so that the library builds in parallel.
#pragma once

#include <vector>

#include "grf.h"
#include "grf_kernels.cuh"

namespace grf {

struct BoxDesc {
    Geom g;
    Coeffs c;
    double* un;
    double* A;
    double* B;
    double* acc;
    double dt, ko, min_chi, min_lapse;
    int enforce;
    int pad_;
};

struct TileDesc {
    int box, pad_;
    long long q0;  // the tile's first interior point (x-fastest order); one point per thread of the block
};

// DEC: 0 full theory, 1 without backreaction, -1 read from the box's coefficients; LOP: lopsided
// advection.
template <int STAGE, int DEC, int LOP>
__device__ __forceinline__ void batch_tile(const BoxDesc* __restrict__ boxes, const TileDesc& td, int* status) {
    const BoxDesc& d = boxes[td.box];
    const long long q = td.q0 + threadIdx.x + (int)blockDim.x * ((int)threadIdx.y + (int)blockDim.y * (int)threadIdx.z);
    if (q >= (long long)d.g.nx * d.g.ny * d.g.nz) return;
    int i, j, k;
    point_of(d.g, q, i, j, k);
    StageArgs a;
    a.un = d.un;
    a.acc = d.acc;
    a.dt = d.dt;
    a.ko = d.ko;
    a.min_chi = d.min_chi;
    a.min_lapse = d.min_lapse;
    a.enforce = d.enforce;
    a.status = status;
    a.src = (STAGE == 0) ? d.un : (STAGE == 1 ? d.A : (STAGE == 2 ? d.B : d.A));
    a.dst = (STAGE == 0) ? d.A : (STAGE == 1 ? d.B : (STAGE == 2 ? d.A : d.un));
    stage_point<STAGE, DEC, LOP>(d.g, d.c, a, i, j, k);
}

// Out-of-line copy of batch_tile for the persistent kernel: with the four stages inlined into one
// kernel, ptxas spilled 52 KB per thread; called, each stage is allocated on its own (13 KB).
template <int STAGE, int DEC, int LOP>
__device__ __noinline__ void batch_tile_call(const BoxDesc* __restrict__ boxes, const TileDesc& td, int* status) {
    batch_tile<STAGE, DEC, LOP>(boxes, td, status);
}

// Shared with the split-box evolution (grf_patches.cu), in grf_batch.cu: the couplings check of
// one parameter set; a box descriptor (geometry, coefficients, dissipation, floors and dt; the
// buffers are left null); the tiles of a box in a work list and their number; one stage launch over
// a tile list.
bool batch_params_ok(const grf_params* p);
void batch_box_desc(BoxDesc& d, const grf_box* b, const grf_params* p, double dt);
inline long long batch_tiles(const Geom& g, int points) { return ((long long)g.nx * g.ny * g.nz + points - 1) / points; }
void batch_append_tiles(std::vector<TileDesc>& tiles, int box, const Geom& g, int points);
void launch_batch_stage(int stage, long long ntiles, dim3 block, cudaStream_t st, const BoxDesc* boxes,
                        const TileDesc* tiles, int* status);

// The persistent cooperative launch (grf_batch_persistent.cu): its function attributes (loads the
// kernel), its resident blocks per SM for `nthreads` threads, and the launch.
cudaError_t batch_persistent_attributes();
cudaError_t batch_persistent_occupancy(int nthreads, int* per_sm);
cudaError_t launch_batch_persistent(dim3 grid, dim3 block, const BoxDesc* boxes, const TileDesc* tiles, int ntiles,
                                    int nsteps, unsigned* bar, int* status, long long timeout, cudaStream_t st);

}  // namespace grf
