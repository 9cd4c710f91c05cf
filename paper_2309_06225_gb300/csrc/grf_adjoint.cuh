// Reverse mode: what the taping kernel (grf_adjoint.cu) and the sweep (grf_adj_sweep.cu) share.
#pragma once

#include "grf_kernels.cuh"
#include "grf_rev.cuh"

namespace grf {

// leaves of the pointwise map: values, first derivatives (24 slots x 3), second derivatives
// (12 slots x 6), KO sums, u_n, acc, lambda, g2
enum : int { kLV = 0, kLD1 = 27, kLD2 = 99, kLKO = 171, kLUN = 198, kLACC = 225, kLLAM = 252, kLG2 = 253, kNLeaf = 254 };
// tape entries per point and stage: the pointwise RHS records about 2,330, the stage update and
// enforcement about 130 more; an overflow is detected and reported
constexpr int kTapeCap = 5120;
constexpr int kAdjThreads = 128;
// tape columns (points per wave): 1024 per SM of a GB300, so that the sweep (28 warps per SM at 72
// registers) has warps to hide its dependent memory operations; the taping kernel is held to 128
// registers for 16 warps per SM (more spills, but it ran faster than at 255 registers with 8)
constexpr long long kAdjCols = 152LL * 1024;
constexpr int kSweepThreads = 128;
// derivative and dissipation adjoints per point (slots of the G buffer): d1 72, d2 72, KO 27
constexpr int kGD2 = 72, kGKO = 144, kGSlots = 171;

struct AdjArgs {
    const double* src;    // u_{s-1} (ghosts valid)
    const double* un;     // u_n
    const double* acc;    // k_1 + 2 k_2 + 2 k_3 (stage 3)
    const double* ubar;   // adjoint of the stage output u_s
    double* abar;         // adjoint of the accumulator: written by stage 3, read by stages 0..2
    double* vbar;         // adjoint of the values of u_{s-1} (stages 1..3, written)
    double* unbar;        // adjoint of u_n (stage 3 writes it, stages 2..0 add)
    double* G;            // kGSlots derivative / KO adjoints, with periodic images
    double* pbar;         // per-column sums of the lambda and g2 adjoints
    int* count;           // tape entries of each column (written by the taping kernel)
    double dt, ko, min_chi, min_lapse;
    int enforce;
    int* status;
    long long npts;
};

// Sweeps the wave's tape columns (points q0 ..).
void launch_adj_sweep(const Geom& g, const AdjArgs& a, const grf_rev::Tape& tape, int stage, long long q0, cudaStream_t st);

}  // namespace grf
