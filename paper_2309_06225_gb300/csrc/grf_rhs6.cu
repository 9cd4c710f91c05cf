// Single-state RHS and constraint kernels of the 6th-order scheme (4 ghost layers).
#include "grf_diag.cuh"
#include "grf_launch.h"

namespace grf {

// One thread per interior point, held to 168 registers as rhs_kernel. LOP: lopsided advection.
template <int LOP>
__global__ void __launch_bounds__(128, 3) rhs6_kernel(Geom g, Coeffs c, const double* __restrict__ s,
                                                      double* __restrict__ rhs, double ko, int* status) {
    const long long q = (long long)blockIdx.x * blockDim.x + threadIdx.x;
    if (q >= (long long)g.nx * g.ny * g.nz) return;
    int i, j, k;
    point_of(g, q, i, j, k);
    const long long p = gidx(g, i + NG6, j + NG6, k + NG6);
    PointIn in;
    double kos[NFIELDS], adv[LOP ? NFIELDS : 1];
    gather6<LOP>(g, s, p, in, kos, adv);
    double r[NFIELDS];
    bool ok = true;
    point_rhs<double, double, -1, LOP>(c, in, r, nullptr, ok, adv);
    if (!ok) atomicOr(status, 1);
#pragma unroll 1
    for (int f = 0; f < NFIELDS; ++f) rhs[f * g.fstride + p] = fma(ko, kos[f], r[f]);
}

void launch_rhs6(cudaStream_t st, const Geom& g, const Coeffs& c, const double* s, double* rhs, double ko, int* status) {
    const long long n = (long long)g.nx * g.ny * g.nz;
    const unsigned threads = point_threads(n), blocks = point_blocks(n, threads);
    if (c.advection) rhs6_kernel<kLopsided><<<blocks, threads, 0, st>>>(g, c, s, rhs, ko, status);
    else rhs6_kernel<0><<<blocks, threads, 0, st>>>(g, c, s, rhs, ko, status);
}

void launch_constraints6(dim3 grid, cudaStream_t st, const Geom& g, const Coeffs& c, const double* s, double* out4,
                         double* part, double* dens, double* psi4, double3 origin, double* hyp) {
    if (psi4 || hyp) constraints_kernel<6, 1><<<grid, 128, 0, st>>>(g, c, s, out4, part, dens, psi4, origin, hyp);
    else constraints_kernel<6, 0><<<grid, 128, 0, st>>>(g, c, s, out4, part, dens, psi4, origin, hyp);
}

}  // namespace grf
