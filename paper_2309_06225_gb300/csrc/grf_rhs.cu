// Single-state RHS and constraint kernels (4th-order scheme).
#include "grf_diag.cuh"
#include "grf_launch.h"

namespace grf {

// One thread per interior point, as rk4_stage_kernel, and bound like it. LOP: lopsided advection.
// Held to 168 registers for 3 blocks per SM (80 x 64 x 72 with its dissipation: 2.35 -> 1.97 ms against 255 and 2).
template <int LOP>
__global__ void __launch_bounds__(128, 3) rhs_kernel(Geom g, Coeffs c, const double* __restrict__ s, double* __restrict__ rhs,
                                                     double ko, int* status) {
    const long long q = (long long)blockIdx.x * blockDim.x + threadIdx.x;
    if (q >= (long long)g.nx * g.ny * g.nz) return;
    int i, j, k;
    point_of(g, q, i, j, k);
    const long long p = gidx(g, i + NG, j + NG, k + NG);
    PointIn in;
    double kos[NFIELDS];
    double adv[LOP ? NFIELDS : 1];
    gather<LOP>(g, s, p, in, kos, adv);
    double r[NFIELDS];
    bool ok = true;
    point_rhs<double, double, -1, LOP>(c, in, r, nullptr, ok, adv);
    if (!ok) atomicOr(status, 1);
#pragma unroll 1
    for (int f = 0; f < NFIELDS; ++f) rhs[f * g.fstride + p] = fma(ko, kos[f], r[f]);
}

void launch_rhs(cudaStream_t st, const Geom& g, const Coeffs& c, const double* s, double* rhs, double ko, int* status) {
    if (g.ng == NG6) {
        launch_rhs6(st, g, c, s, rhs, ko, status);
        return;
    }
    const long long n = (long long)g.nx * g.ny * g.nz;
    const unsigned threads = point_threads(n), blocks = point_blocks(n, threads);
    if (c.advection) rhs_kernel<kLopsided><<<blocks, threads, 0, st>>>(g, c, s, rhs, ko, status);
    else rhs_kernel<0><<<blocks, threads, 0, st>>>(g, c, s, rhs, ko, status);
}
void launch_constraints(cudaStream_t st, const Geom& g, const Coeffs& c, const double* s, double* out4, double* part,
                        double* dens, double* psi4, double3 origin, double* hyp) {
    const dim3 grid(constraint_blocks(g));
    if (g.ng == NG6) launch_constraints6(grid, st, g, c, s, out4, part, dens, psi4, origin, hyp);
    else if (psi4 || hyp) constraints_kernel<4, 1><<<grid, 128, 0, st>>>(g, c, s, out4, part, dens, psi4, origin, hyp);
    else constraints_kernel<4, 0><<<grid, 128, 0, st>>>(g, c, s, out4, part, dens, psi4, origin, hyp);
}
}  // namespace grf
