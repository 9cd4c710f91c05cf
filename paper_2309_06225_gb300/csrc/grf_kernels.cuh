// Grid kernels of the GB300 path: stencil gather, fused RK4 stage, RHS, KO dissipation,
// periodic ghost fill, constraints and their norms.
#pragma once

#include <cuda_runtime.h>

#include "grf_diffs.cuh"
#include "grf_point.cuh"

// Loads of stencil sources. By default the read-only, non-coherent path (__ldg): every kernel
// that reads a state through these helpers leaves it unwritten for the rest of its launch. A
// kernel that reads, in one launch, buffers that other blocks wrote earlier in the same launch
// (the persistent batched kernel, across its grid barriers) defines GRF_COHERENT_LOADS before
// including this header: the loads then go through L2 only (__ldcg), which is coherent.
#ifdef GRF_COHERENT_LOADS
#define GRF_LDG(p) __ldcg(p)
#else
#define GRF_LDG(p) __ldg(p)
#endif

namespace grf {

struct Geom {
    int nx, ny, nz;          // interior points
    int NX, NY, NZ;          // ghosted extents (n + 2 ng)
    long long pitch;         // doubles per x row
    long long plane;         // pitch * NY
    long long fstride;       // plane * NZ
    double dx;
    int periodic;            // ghosts are periodic images (written by the owner of each value)
    int reflect;             // the three low faces are mirror planes (images written by the owner)
    int ng;                  // ghost layers: 3 (4th-order scheme) or 4 (6th-order scheme)
    // the scheme's factors of first, second and mixed differences (4th order: 1/(12 dx), 1/(12 dx^2),
    // 1/(144 dx^2); 6th order: 1/(60 dx), 1/(180 dx^2), 1/(3600 dx^2)), and the fixed-point sums' range
    FxScale f1, f2, f11;
    FxRange fx;
};

inline void set_spacing(Geom& g, double dx, int ng) {
    g.ng = ng;
    g.dx = dx;
    spacing_factors(g, dx, ng);
}

constexpr int NG = 3;        // ghost layers of the 4th-order kernels (those of this header)

// Blocks (of 128 points) of the constraint kernel, each with one set of partial norms.
inline unsigned constraint_blocks(const Geom& g) { return (unsigned)(((long long)g.nx * g.ny * g.nz + 127) / 128); }

__device__ __forceinline__ long long gidx(const Geom& g, int i, int j, int k) {  // ghosted indices
    return (long long)k * g.plane + (long long)j * g.pitch + i;
}

// Centred 4th-order differences at ghosted offset p in FP64 (the adjoint's transposed stencils).
// first: (u_-2 - 8 u_-1 + 8 u_+1 - u_+2)/(12 dx) ; second: (-u_-2 + 16 u_-1 - 30 u_0 + 16 u_+1 - u_+2)/(12 dx^2)
// mixed: the first-derivative stencil along s applied to first derivatives along t.
__device__ __forceinline__ double fd1(const double* __restrict__ u, long long p, long long s, double i12) {
    return fma(8.0, GRF_LDG(u + p + s) - GRF_LDG(u + p - s), GRF_LDG(u + p - 2 * s) - GRF_LDG(u + p + 2 * s)) * i12;
}
__device__ __forceinline__ double fd2(const double* __restrict__ u, long long p, long long s, double u0, double i12s) {
    return fma(-30.0, u0, fma(16.0, GRF_LDG(u + p + s) + GRF_LDG(u + p - s), -(GRF_LDG(u + p + 2 * s) + GRF_LDG(u + p - 2 * s)))) * i12s;
}
__device__ __forceinline__ double mixed_local(const double* __restrict__ u, long long p, long long so, long long t,
                                              double i12) {
    const double m2 = fd1(u, p - 2 * so, t, i12), m1 = fd1(u, p - so, t, i12);
    const double p1 = fd1(u, p + so, t, i12), p2 = fd1(u, p + 2 * so, t, i12);
    return fma(8.0, p1 - m1, m2 - p2) * i12;
}

// sum_d (u_-3 - 6 u_-2 + 15 u_-1 - 20 u_0 + 15 u_+1 - 6 u_+2 + u_+3), pair sums added x, y, z
__device__ __forceinline__ double ko6(const double* __restrict__ u, long long p, long long sy, long long sz) {
    const long long st[3] = {1, sy, sz};
    double t[4];
#pragma unroll
    for (int r = 1; r <= 3; ++r)
        t[r] = ((GRF_LDG(u + p - r * st[0]) + GRF_LDG(u + p + r * st[0])) + (GRF_LDG(u + p - r * st[1]) + GRF_LDG(u + p + r * st[1]))) +
               (GRF_LDG(u + p - r * st[2]) + GRF_LDG(u + p + r * st[2]));
    return fma(-60.0, GRF_LDG(u + p), fma(15.0, t[1], fma(-6.0, t[2], t[3])));
}

__device__ __forceinline__ bool has_d2(int f) {
    return f == F_CHI || (f >= F_H && f < F_H + 6) || f == F_LAPSE || (f >= F_SHIFT && f < F_SHIFT + 3) || f == F_PHI;
}
__device__ __forceinline__ bool has_d1(int f) { return !(f >= F_B && f < F_B + 3); }

// ---- the gather: differences of the fields at one point, the sums in block fixed point (grf_fixed.cuh)

// The values axis_diffs reads; the outermost ones only where they count (KO, LOP).
template <int OUTER>
__device__ __forceinline__ void load_axes(const Geom& g, const double* __restrict__ u, AxisValues& v) {
    const long long st[3] = {1, g.pitch, g.plane};
    v.c = GRF_LDG(u);
#pragma unroll
    for (int d = 0; d < 3; ++d)
#pragma unroll
        for (int k = 0; k < (OUTER ? 3 : 2); ++k) {
            v.m[d][k] = GRF_LDG(u - (k + 1) * st[d]);
            v.q[d][k] = GRF_LDG(u + (k + 1) * st[d]);
        }
}
__device__ __forceinline__ void load_plane(const double* __restrict__ u, long long sa, long long sb, PlaneValues& v) {
#pragma unroll
    for (int a = 0; a < 4; ++a)
#pragma unroll
        for (int b = 0; b < 4; ++b)
            v.x[a][b] = GRF_LDG(u + (a < 2 ? a - 2 : a - 1) * sa + (b < 2 ? b - 2 : b - 1) * sb);
}

// The fields that the constraints take derivatives of: all but Theta, Gamma-hat, the lapse, the shift and B.
constexpr unsigned kMetricScalarFields = ((1u << F_TH) - 1) | 1u << F_PHI | 1u << F_PI;

// Where a gather's results go: a point's data, dissipation sums and (LOP) advection terms.
struct PointSink {
    PointIn& in;
    double* kos;
    double* adv;
    __device__ __forceinline__ void value(int f, double x) const { in.v[f] = x; }
    __device__ __forceinline__ void first(int slot, int d, double x) const { in.d1[slot][d] = x; }
    __device__ __forceinline__ void second(int slot, int m, double x) const { in.d2[slot][m] = x; }
    __device__ __forceinline__ void dissipation(int f, double x) const { kos[f] = x; }
    __device__ __forceinline__ void advection(int f, double x) const { adv[f] = x; }
};

// The differences in FP64, for a point whose fields leave the fixed-point range (values near overflow,
// infinities, NaNs): rewrites what gather() took.
template <int LOP, int KO, typename Sink>
__device__ __noinline__ void gather_fp64(const Geom& g, const double* __restrict__ s, long long p, const Sink& out,
                                         unsigned fields) {
    const double i12 = 1.0 / (12.0 * g.dx), i12s = 1.0 / (12.0 * g.dx * g.dx);
    const long long st[3] = {1, g.pitch, g.plane};
#pragma unroll 1
    for (int f = 0; f < NFIELDS; ++f) {
        if (!(fields >> f & 1u)) continue;
        const double* u = s + f * g.fstride + p;
        const double u0 = GRF_LDG(u);
        double av = 0.0;
        if (KO) out.dissipation(f, ko6(u, 0, g.pitch, g.plane));
#pragma unroll 1
        for (int d = 0; d < 3; ++d) {
            if (has_d1(f)) out.first(d1slot(f), d, fd1(u, 0, st[d], i12));
            if (has_d2(f)) {
                out.second(d2slot(f), d == 0 ? 0 : (d == 1 ? 3 : 5), fd2(u, 0, st[d], u0, i12s));
                out.second(d2slot(f), d == 2 ? 4 : d + 1, mixed_local(u, 0, st[d == 2], st[d == 0 ? 1 : 2], i12));
            }
            if (LOP) {
                const double b = GRF_LDG(s + (F_SHIFT + d) * g.fstride + p);
                const long long t = b >= 0.0 ? st[d] : -st[d];
                const double x = fma(18.0, GRF_LDG(u + t), fma(-6.0, GRF_LDG(u + 2 * t), GRF_LDG(u + 3 * t))) -
                                 fma(3.0, GRF_LDG(u - t), 10.0 * u0);
                av = fma(fabs(b), x * i12, av);
            }
        }
        if (LOP) out.advection(f, av);
    }
}

// The 15 fields without second derivatives, in their order: K, A, Theta, Gamma-hat, B, Pi.
__host__ __device__ constexpr int plainfield(int b) { return b < 11 ? b + 7 : (b < 14 ? b + 11 : F_PI); }
// Field index of d2 slot b (inverse of d2slot).
__host__ __device__ constexpr int d2field(int b) { return b < 7 ? b : (b == 7 ? F_LAPSE : (b < 11 ? b + 11 : F_PHI)); }

// Values, first derivatives and second derivatives of all fields at ghosted offset p, and each field's
// Kreiss-Oliger sum sum_d (u_-3 - 6 u_-2 + 15 u_-1 - 20 u_0 + 15 u_+1 - 6 u_+2 + u_+3).
//   LOP = 1: also the lopsided advection terms adv[f] = sum_d |beta^d| D_d u_f.
//   ALL = 0: only the kMetricScalarFields (the others' entries are left alone).
//   KO = 0: no Kreiss-Oliger sums; the outermost points, at +-3, are then read for LOP only.
// Two rolled loops (the 12 fields with second derivatives, the 15 without): unrolled threefold, the integer
// code of a field no longer stays in the instruction cache (128^3 step 44 -> 50 ms). Each block's values are
// loaded one block ahead of their use, so that the loads' latency lies under the previous block's arithmetic.
//   TEAM > 1: the point's fields are shared out over TEAM consecutive lanes, of which this is lane t (every
//   lane of the warp calls this; in, kos and adv are the team's).
template <int LOP, int ALL, int TEAM, int KO, typename Sink>
__device__ __forceinline__ void gather_to(const Geom& g, const double* __restrict__ s, long long p, const Sink& out, int t) {
    const long long st[3] = {1, g.pitch, g.plane};
    double bet[3] = {0.0, 0.0, 0.0};
    if (LOP) {
#pragma unroll
        for (int d = 0; d < 3; ++d) bet[d] = GRF_LDG(s + (F_SHIFT + d) * g.fstride + p);
    }
    // slots 0..6 (chi, h) and phi; with ALL also lapse and shift (slots 7..10); K, A; with ALL the rest
    constexpr int kLastSecond = ALL ? 10 : 6, kLastPlain = ALL ? 13 : 6;
    auto next_second = [](int b) { return TEAM > 1 ? b + TEAM : (b == kLastSecond ? 11 : b + 1); };
    auto next_plain = [](int b) { return TEAM > 1 ? b + TEAM : (b == kLastPlain ? 14 : b + 1); };
    const double* u = s + d2field(t) * g.fstride + p;
    AxisValues ax;
    load_axes<LOP || KO>(g, u, ax);
    int mag = 0;
#pragma unroll 1
    for (int b = t; b < 12; b = next_second(b)) {
        FieldDiffs r;
        const int f = d2field(b);
        out.value(f, ax.c);
        mag = fx_max(mag, axis_diffs<LOP, KO>(g, ax, true, true, bet, r));
        out.second(b, 0, r.d2[0]);
        out.second(b, 3, r.d2[3]);
        out.second(b, 5, r.d2[5]);
#pragma unroll 1
        for (int c = 0; c < 3; ++c) {
            PlaneValues pl;
            load_plane(u, c < 2 ? 1 : st[1], c == 0 ? st[1] : st[2], pl);
            out.second(b, c < 2 ? c + 1 : 4, plane_diff(g, pl, mag));
        }
        const int nb = next_second(b), next = nb < 12 ? d2field(nb) : plainfield(t);
        u = s + next * g.fstride + p;
        load_axes<LOP || KO>(g, u, ax);
        if (KO) out.dissipation(f, r.ko);
#pragma unroll
        for (int d = 0; d < 3; ++d) out.first(d1slot(f), d, r.d1[d]);
        if (LOP) out.advection(f, fma(fabs(bet[2]), r.up[2], fma(fabs(bet[1]), r.up[1], fabs(bet[0]) * r.up[0])));
    }
#pragma unroll 1
    for (int b = t; b < 15; b = next_plain(b)) {
        FieldDiffs r;
        const AxisValues now = ax;
        if (next_plain(b) < 15) load_axes<LOP || KO>(g, s + plainfield(next_plain(b)) * g.fstride + p, ax);
        const int f = plainfield(b);
        out.value(f, now.c);
        mag = fx_max(mag, axis_diffs<LOP, KO>(g, now, has_d1(f), false, bet, r));
        if (KO) out.dissipation(f, r.ko);
        if (has_d1(f)) {
#pragma unroll
            for (int d = 0; d < 3; ++d) out.first(d1slot(f), d, r.d1[d]);
        }
        if (LOP) out.advection(f, fma(fabs(bet[2]), r.up[2], fma(fabs(bet[1]), r.up[1], fabs(bet[0]) * r.up[0])));
    }
    unsigned fields = ALL ? (1u << NFIELDS) - 1 : kMetricScalarFields;
    if (TEAM > 1) {
#pragma unroll
        for (int o = 1; o < TEAM; o *= 2) mag = fx_max(mag, __shfl_xor_sync(0xffffffffu, mag, o));
        fields = 0;
        for (int b = t; b < 12; b += TEAM) fields |= 1u << d2field(b);
        for (int b = t; b < 15; b += TEAM) fields |= 1u << plainfield(b);
    }
    if (mag >> 20 > g.fx.emax) {
        gather_fp64<LOP, KO>(g, s, p, out, fields);
    }
}

template <int LOP = 0, int ALL = 1, int TEAM = 1, int KO = 1>
__device__ __forceinline__ void gather(const Geom& g, const double* __restrict__ s, long long p, PointIn& in,
                                       double kos[NFIELDS], double* adv = nullptr, int t = 0) {
    gather_to<LOP, ALL, TEAM, KO>(g, s, p, PointSink{in, kos, adv}, t);
}

__device__ __forceinline__ bool interior_thread(const Geom& g, int& i, int& j, int& k) {
    i = blockIdx.x * blockDim.x + threadIdx.x;
    j = blockIdx.y * blockDim.y + threadIdx.y;
    k = blockIdx.z * blockDim.z + threadIdx.z;
    return i < g.nx && j < g.ny && k < g.nz;
}

// Parity of field f under the reflections x_d -> -x_d of the axes in `mask` (bit d): -1 when
// the component has an odd number of indices along the reflected axes (the d-components of
// Gamma-hat, shift and B; h_ab and A_ab with exactly one index reflected), +1 otherwise.
__host__ __device__ __forceinline__ double mirror_sign(int f, int mask) {
    int odd = 0;
    if (f >= F_GAM && f < F_GAM + 3) odd = (mask >> (f - F_GAM)) & 1;
    else if (f >= F_SHIFT && f < F_SHIFT + 3) odd = (mask >> (f - F_SHIFT)) & 1;
    else if (f >= F_B && f < F_B + 3) odd = (mask >> (f - F_B)) & 1;
    else if ((f >= F_H && f < F_H + 6) || (f >= F_A && f < F_A + 6)) {
        const int m = (f < F_A) ? f - F_H : f - F_A;  // sym index of (a, b), a <= b
        const int a = m < 3 ? 0 : (m < 5 ? 1 : 2);
        const int b = m < 3 ? m : (m < 5 ? m - 2 : 2);
        odd = ((mask >> a) & 1) ^ ((mask >> b) & 1);
    }
    return odd ? -1.0 : 1.0;
}

// Writes value x of field f for interior point (i,j,k) and to every ghost location that is an
// image of it: periodic images, or for mirror boxes its reflections in the low faces (the
// mirror plane lies half a cell below the first point; ghost NG-1-i mirrors interior i), with
// the component's parity.
template <int NGT = NG>
__device__ __forceinline__ void store_with_images(const Geom& g, double* __restrict__ dst, int f, int i, int j, int k,
                                                  double x) {
    constexpr int NG = NGT;
    double* d = dst + f * g.fstride;
    if (!g.periodic) {
        d[gidx(g, i + NG, j + NG, k + NG)] = x;
        if (g.reflect) {
            const int near = (i < NG ? 1 : 0) | (j < NG ? 2 : 0) | (k < NG ? 4 : 0);
            for (int m = 1; m < 8; ++m) {
                if (m & ~near) continue;
                d[gidx(g, (m & 1) ? NG - 1 - i : i + NG, (m & 2) ? NG - 1 - j : j + NG, (m & 4) ? NG - 1 - k : k + NG)] =
                    mirror_sign(f, m) * x;
            }
        }
        return;
    }
    int xi[3], yi[3], zi[3];
    int nxi = 0, nyi = 0, nzi = 0;
    xi[nxi++] = i + NG;
    if (i < NG) xi[nxi++] = i + NG + g.nx;
    if (i >= g.nx - NG) xi[nxi++] = i + NG - g.nx;
    yi[nyi++] = j + NG;
    if (j < NG) yi[nyi++] = j + NG + g.ny;
    if (j >= g.ny - NG) yi[nyi++] = j + NG - g.ny;
    zi[nzi++] = k + NG;
    if (k < NG) zi[nzi++] = k + NG + g.nz;
    if (k >= g.nz - NG) zi[nzi++] = k + NG - g.nz;
    for (int c = 0; c < nzi; ++c)
        for (int b = 0; b < nyi; ++b)
            for (int a = 0; a < nxi; ++a) d[gidx(g, xi[a], yi[b], zi[c])] = x;
}

// Trace-free A_ij with respect to h_ij, and the chi / lapse floors, on one point's values.
__device__ __forceinline__ void enforce_point(double u[NFIELDS], double min_chi, double min_lapse) {
    double hh[6], hi[6], id;
#pragma unroll
    for (int m = 0; m < 6; ++m) hh[m] = u[F_H + m];
    sym3_inv(hh, hi, id);
    const double off = dot3(hi[1], u[F_A + 1], hi[2], u[F_A + 2], hi[4], u[F_A + 4]);
    const double tr3 = fma(2.0, off, dot3(hi[0], u[F_A], hi[3], u[F_A + 3], hi[5], u[F_A + 5])) * (1.0 / 3.0);
#pragma unroll
    for (int m = 0; m < 6; ++m) u[F_A + m] = fnma(hh[m], tr3, u[F_A + m]);
    u[F_CHI] = fmax(u[F_CHI], min_chi);
    u[F_LAPSE] = fmax(u[F_LAPSE], min_lapse);
}

struct StageArgs {
    const double* src;   // state whose RHS is evaluated (ghosts valid)
    const double* un;    // u_n (pointwise)
    double* acc;         // k1 + 2 k2 + 2 k3 accumulator (pointwise)
    double* dst;         // state written by this stage
    double dt;
    double ko;           // sigma / (64 dx)
    double min_chi, min_lapse;
    int enforce;
    int* status;
    long long q0, q1;    // the launch's interior points in x-fastest order: [q0, q1)
};

// Lopsided advection: the ADV terms of point_rhs come from in.adv (filled by the gather).
constexpr int kLopsided = 1;

// RK4 stage arithmetic for one value at offset q (u_1 = u_n + dt/2 k_1, u_2 = u_n + dt/2 k_2,
// u_3 = u_n + dt k_3, u_{n+1} = u_n + dt/6 (k_1 + 2 k_2 + 2 k_3 + k_4)): kf the stage's right-hand
// side, unf = u_n; the accumulator a.acc[q] is read (STAGE > 0) and written (STAGE < 3). Returns
// the stage's output value.
template <int STAGE>
__device__ __forceinline__ double rk4_value(const StageArgs& a, long long q, double kf, double unf) {
    double accf;
    if (STAGE == 0) accf = kf;
    else if (STAGE == 3) accf = a.acc[q] + kf;
    else accf = fma(2.0, kf, a.acc[q]);
    if (STAGE < 3) a.acc[q] = accf;
    const double cs = (STAGE == 0 || STAGE == 1) ? 0.5 * a.dt : (STAGE == 2 ? a.dt : a.dt * (1.0 / 6.0));
    return (STAGE == 3) ? fma(cs, accf, unf) : fma(cs, kf, unf);
}

// Interior point q (x fastest) as (i, j, k); 32-bit divisions where the box allows them.
__device__ __forceinline__ void point_of(const Geom& g, long long q, int& i, int& j, int& k) {
    const unsigned nx = (unsigned)g.nx, ny = (unsigned)g.ny;
    long long row;  // q / nx
    if (q < (1LL << 32)) row = (unsigned)q / nx;
    else row = q / nx;
    i = (int)(q - row * nx);
    k = (int)((unsigned)row / ny);  // rows of a box that fits the device are below 2^32
    j = (int)((unsigned)row - (unsigned)k * ny);
}

// One RK4 stage at one point, fused: gather -> pointwise RHS -> + KO -> stage update ->
// enforcement -> store (with periodic images). STAGE 0..3.
template <int STAGE, int DEC = -1, int LOP = 0, int COUP = 1>
__device__ __forceinline__ void stage_point(const Geom& g, const Coeffs& c, const StageArgs& a, int i, int j, int k) {
    const long long p = gidx(g, i + NG, j + NG, k + NG);
    PointIn in;
    double kos[NFIELDS];
    double adv[LOP ? NFIELDS : 1];
    gather<LOP>(g, a.src, p, in, kos, adv);
    double r[NFIELDS];
    bool ok = true;
    point_rhs<double, double, DEC, LOP, COUP>(c, in, r, nullptr, ok, adv);
    if (!ok) atomicOr(a.status, 1);
#pragma unroll 1
    for (int f = 0; f < NFIELDS; ++f) {  // r becomes the stage's output values
        const double kf = fma(a.ko, kos[f], r[f]);
        const double unf = (STAGE == 0) ? in.v[f] : a.un[f * g.fstride + p];
        r[f] = rk4_value<STAGE>(a, f * g.fstride + p, kf, unf);
    }
    if (a.enforce) enforce_point(r, a.min_chi, a.min_lapse);
#pragma unroll 1
    for (int f = 0; f < NFIELDS; ++f) store_with_images(g, a.dst, f, i, j, k, r[f]);
}

// One thread per interior point of [q0, q1), consecutive threads consecutive points in x-fastest order,
// so that every lane of every warp but the last works whatever the box's extents (no derivative is
// exchanged between lanes, so the mapping is free). Blocks of point_threads() threads (grf_launch.h).
// What bounds it: the FP64 pipe (80% of its issue slots), 2,292 instructions a point and stage. 12 resident
// warps per SM (168 registers a thread) hide its latency; more would spill more: 128^3 step 51.1 ms with 8
// warps, 38.8 with 12, 42.0 with 16, 45.8 with 20. (256^3 step 506 -> 317 ms since the stencils are summed in
// integers, grf_fixed.cuh, and the equations need fewer operations, grf_point.cuh.)
// DEC: 0 full theory, 1 without backreaction (a separate instantiation each, so the full
// theory's kernel carries no test of the mode), -1 the mode read from c. LOP: lopsided advection.
// COUP = 0: the linear and quadratic couplings only.
template <int STAGE, int DEC = 0, int LOP = 0, int COUP = 1>
__global__ void __launch_bounds__(128, 3) rk4_stage_kernel(Geom g, Coeffs c, StageArgs a) {
    const long long q = a.q0 + (long long)blockIdx.x * blockDim.x + threadIdx.x;
    if (q >= a.q1) return;
    int i, j, k;
    point_of(g, q, i, j, k);
    stage_point<STAGE, DEC, LOP, COUP>(g, c, a, i, j, k);
}

}  // namespace grf
