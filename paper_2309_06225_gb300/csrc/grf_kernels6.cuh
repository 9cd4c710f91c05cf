// 6th-order scheme ("Accuracy": 4th- and 6th-order finite differences) on boxes with 4 ghost
// layers: centred 6th-order first, second and mixed differences, Kreiss-Oliger dissipation with
// the 8th difference, and the 6th-order lopsided advection stencil (offsets -2..4 towards the
// side the shift points to). The sums are in block fixed point as the 4th-order ones.
#pragma once

#include "grf_kernels.cuh"

namespace grf {

constexpr int NG6 = 4;  // ghost layers of the 6th-order scheme

// 6th-order centred first difference times 60 dx at offset p along stride t:
//   (u_3 - u_-3) - 9 (u_2 - u_-2) + 45 (u_1 - u_-1)
__device__ __forceinline__ double fd1_6(const double* __restrict__ u, long long p, long long t) {
    return fma(45.0, __ldg(u + p + t) - __ldg(u + p - t),
               fma(-9.0, __ldg(u + p + 2 * t) - __ldg(u + p - 2 * t), __ldg(u + p + 3 * t) - __ldg(u + p - 3 * t)));
}

// Values, first and second derivatives, lopsided advection terms adv[f] (LOP = 1) and the 8th
// differences sum_d Delta^8_d u of all fields at ghosted offset p.
//   first:  ((u_3 - u_-3) - 9 (u_2 - u_-2) + 45 (u_1 - u_-1)) / (60 dx)
//   second: (2 (u_3 + u_-3) - 27 (u_2 + u_-2) + 270 (u_1 + u_-1) - 490 u_0) / (180 dx^2)
//   mixed:  the first-difference stencil along s applied to first differences along t
//   KO:     (u_4 + u_-4) - 8 (u_3 + u_-3) + 28 (u_2 + u_-2) - 56 (u_1 + u_-1) + 70 u_0 per axis
//   lopsided, beta^d >= 0 (mirrored for beta^d < 0; a_n = u at n points towards the side beta^d
//   points to, b_n = u at n points away from it):
//           beta^d D_d u = |beta^d| (2 b_2 - 24 b_1 - 35 u_0 + 80 a_1 - 30 a_2 + 8 a_3 - a_4) / (60 dx)
// In FP64, for points whose fields leave the fixed-point range. `fields` as for gather_fp64.
template <int LOP, int KO>
__device__ __noinline__ void gather6_fp64(const Geom& g, const double* __restrict__ s, long long p, PointIn& in,
                                          double* kos, double* adv, unsigned fields) {
    const double i60 = 1.0 / (60.0 * g.dx), i180s = 1.0 / (180.0 * g.dx * g.dx);
    const long long st[3] = {1, g.pitch, g.plane};
    double bet[3] = {0.0, 0.0, 0.0};
    if (LOP) {
#pragma unroll
        for (int d = 0; d < 3; ++d) bet[d] = __ldg(s + (F_SHIFT + d) * g.fstride + p);
    }
#pragma unroll 1
    for (int f = 0; f < NFIELDS; ++f) {
        if (!(fields >> f & 1u)) continue;
        const double* u = s + f * g.fstride;
        const double u0 = __ldg(u + p);
        in.v[f] = u0;
        double t[5] = {0.0, 0.0, 0.0, 0.0, 0.0};  // pair sums at distance 1..4 over the three axes
        double pr[3][5];
        double av = 0.0;
#pragma unroll
        for (int d = 0; d < 3; ++d) {
            double m[5], q[5];
#pragma unroll
            for (int r = 1; r <= 4; ++r) {
                m[r] = __ldg(u + p - r * st[d]);
                q[r] = __ldg(u + p + r * st[d]);
                pr[d][r] = m[r] + q[r];
            }
            const double d1 = fma(45.0, q[1] - m[1], fma(-9.0, q[2] - m[2], q[3] - m[3])) * i60;
            if (!(f >= F_B && f < F_B + 3)) in.d1[d1slot(f)][d] = d1;
            if (LOP) {
                const bool fw = bet[d] >= 0.0;
                const double a1 = fw ? q[1] : m[1], a2 = fw ? q[2] : m[2], a3 = fw ? q[3] : m[3], a4 = fw ? q[4] : m[4];
                const double b1 = fw ? m[1] : q[1], b2 = fw ? m[2] : q[2];
                const double x = fma(80.0, a1, fma(-30.0, a2, fma(8.0, a3, -a4))) + fma(2.0, b2, fma(-24.0, b1, -35.0 * u0));
                av = fma(fabs(bet[d]), x * i60, av);
            }
        }
        if (LOP) adv[f] = av;
        if (has_d2(f)) {
            const int b = d2slot(f);
#pragma unroll
            for (int d = 0; d < 3; ++d)
                in.d2[b][d == 0 ? 0 : (d == 1 ? 3 : 5)] =
                    fma(270.0, pr[d][1], fma(-27.0, pr[d][2], fma(2.0, pr[d][3], -490.0 * u0))) * i180s;
            const int pairs[3][3] = {{0, 1, 1}, {0, 2, 2}, {1, 2, 4}};  // (s, t, slot)
#pragma unroll
            for (int c = 0; c < 3; ++c) {
                const long long so = st[pairs[c][0]], to = st[pairs[c][1]];
                const double dp1 = fd1_6(u, p + so, to) * i60, dm1 = fd1_6(u, p - so, to) * i60;
                const double dp2 = fd1_6(u, p + 2 * so, to) * i60, dm2 = fd1_6(u, p - 2 * so, to) * i60;
                const double dp3 = fd1_6(u, p + 3 * so, to) * i60, dm3 = fd1_6(u, p - 3 * so, to) * i60;
                in.d2[b][pairs[c][2]] = fma(45.0, dp1 - dm1, fma(-9.0, dp2 - dm2, dp3 - dm3)) * i60;
            }
        }
#pragma unroll
        for (int r = 1; r <= 4; ++r) t[r] = (pr[0][r] + pr[1][r]) + pr[2][r];
        if (KO) kos[f] = fma(210.0, u0, fma(-56.0, t[1], fma(28.0, t[2], fma(-8.0, t[3], t[4]))));
    }
}

// ---- the gather in block fixed point

// The values axis_diffs6 reads; the outermost ones only where they count (KO, LOP).
template <int OUTER>
__device__ __forceinline__ void load_axes6(const Geom& g, const double* __restrict__ u, AxisValues6& v) {
    const long long st[3] = {1, g.pitch, g.plane};
    v.c = __ldg(u);
#pragma unroll
    for (int d = 0; d < 3; ++d)
#pragma unroll
        for (int k = 0; k < (OUTER ? 4 : 3); ++k) {
            v.m[d][k] = __ldg(u - (k + 1) * st[d]);
            v.q[d][k] = __ldg(u + (k + 1) * st[d]);
        }
}

__device__ __forceinline__ void load_plane6(const double* __restrict__ u, long long sa, long long sb, PlaneValues6& v) {
#pragma unroll
    for (int a = 0; a < 6; ++a)
#pragma unroll
        for (int b = 0; b < 6; ++b) v.x[a][b] = __ldg(u + (a < 3 ? a - 3 : a - 2) * sa + (b < 3 ? b - 3 : b - 2) * sb);
}

// As gather() (LOP, ALL and KO likewise), 6th order; kos[f] = sum_d Delta^8_d u. Rolled loops over the fields and
// over the three planes of a field.
template <int LOP = 0, int ALL = 1, int KO = 1>
__device__ __forceinline__ void gather6(const Geom& g, const double* __restrict__ s, long long p, PointIn& in,
                                        double kos[NFIELDS], double* adv = nullptr) {
    const long long st[3] = {1, g.pitch, g.plane};
    constexpr unsigned kFields = ALL ? (1u << NFIELDS) - 1 : kMetricScalarFields;
    double bet[3] = {0.0, 0.0, 0.0};
    if (LOP) {
#pragma unroll
        for (int d = 0; d < 3; ++d) bet[d] = __ldg(s + (F_SHIFT + d) * g.fstride + p);
    }
    int mag = 0;
#pragma unroll 1
    for (int f = 0; f < NFIELDS; ++f) {
        if (!(kFields >> f & 1u)) continue;
        const double* u = s + f * g.fstride + p;
        const bool first = has_d1(f), second = has_d2(f);
        AxisValues6 ax;
        load_axes6<LOP || KO>(g, u, ax);
        FieldDiffs r;
        in.v[f] = ax.c;
        mag = fx_max(mag, axis_diffs6<LOP, KO>(g, ax, first, second, bet, r));
        if (KO) kos[f] = r.ko;
        if (first) {
#pragma unroll
            for (int d = 0; d < 3; ++d) in.d1[d1slot(f)][d] = r.d1[d];
        }
        if (second) {
            const int b = d2slot(f);
            in.d2[b][0] = r.d2[0];
            in.d2[b][3] = r.d2[3];
            in.d2[b][5] = r.d2[5];
#pragma unroll 1
            for (int c = 0; c < 3; ++c) {
                PlaneValues6 pl;
                load_plane6(u, c < 2 ? 1 : st[1], c == 0 ? st[1] : st[2], pl);
                in.d2[b][c < 2 ? c + 1 : 4] = plane_diff6(g, pl, mag);
            }
        }
        if (LOP) adv[f] = fma(fabs(bet[2]), r.up[2], fma(fabs(bet[1]), r.up[1], fabs(bet[0]) * r.up[0]));
    }
    if (mag >> 20 > g.fx.emax) gather6_fp64<LOP, KO>(g, s, p, in, kos, adv, kFields);
}

// One RK4 stage at one point of a 6th-order box, as stage_point (a.ko = -sigma/(256 dx)).
template <int STAGE, int LOP>
__device__ __forceinline__ void stage_point6(const Geom& g, const Coeffs& c, const StageArgs& a, int i, int j, int k) {
    const long long p = gidx(g, i + NG6, j + NG6, k + NG6);
    PointIn in;
    double kos[NFIELDS], adv[LOP ? NFIELDS : 1];
    gather6<LOP>(g, a.src, p, in, kos, adv);
    double r[NFIELDS];
    bool ok = true;
    point_rhs<double, double, -1, LOP>(c, in, r, nullptr, ok, adv);
    if (!ok) atomicOr(a.status, 1);
#pragma unroll 1
    for (int f = 0; f < NFIELDS; ++f) {
        const double kf = fma(a.ko, kos[f], r[f]);
        const double unf = (STAGE == 0) ? in.v[f] : a.un[f * g.fstride + p];
        r[f] = rk4_value<STAGE>(a, f * g.fstride + p, kf, unf);
    }
    if (a.enforce) enforce_point(r, a.min_chi, a.min_lapse);
#pragma unroll 1
    for (int f = 0; f < NFIELDS; ++f) store_with_images<NG6>(g, a.dst, f, i, j, k, r[f]);
}

// One thread per interior point of [q0, q1), as rk4_stage_kernel. The decoupled mode is read from c.
template <int STAGE, int LOP>
__global__ void __launch_bounds__(128, 3) rk4_stage6_kernel(Geom g, Coeffs c, StageArgs a) {
    const long long q = a.q0 + (long long)blockIdx.x * blockDim.x + threadIdx.x;
    if (q >= a.q1) return;
    int i, j, k;
    point_of(g, q, i, j, k);
    stage_point6<STAGE, LOP>(g, c, a, i, j, k);
}

// sum_d Delta^8_d u at ghosted offset p (pair sums added x, y, z)
__device__ __forceinline__ double ko8(const double* __restrict__ u, long long p, long long sy, long long sz) {
    const long long st[3] = {1, sy, sz};
    double t[5];
#pragma unroll
    for (int r = 1; r <= 4; ++r)
        t[r] = ((__ldg(u + p - r * st[0]) + __ldg(u + p + r * st[0])) + (__ldg(u + p - r * st[1]) + __ldg(u + p + r * st[1]))) +
               (__ldg(u + p - r * st[2]) + __ldg(u + p + r * st[2]));
    return fma(210.0, __ldg(u + p), fma(-56.0, t[1], fma(28.0, t[2], fma(-8.0, t[3], t[4]))));
}

}  // namespace grf
