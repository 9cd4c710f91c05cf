// Finite differences and dissipation sums of one field at one point, from its values around the point, in block
// fixed point (grf_fixed.cuh). 4th- and 6th-order schemes. The functions compile for the host too.
//
// Blocks: the points of one difference along one grid line. A difference across a line's neighbours (a mixed
// derivative, the dissipation's sum over the axes) is taken of the lines' sums, brought to a common unit that
// the largest of them fills. So a sum's error is bounded by its own points' magnitudes, as an FP64 sum's is, and
// it is the smaller of the two: in the tail of 1e-2 exp(-r^2), 8 to 16 cells out, mean relative errors of first
// and mixed derivatives 1.2e-16 and 4.4e-16 where FP64 has 2.4e-16 and 1.9e-15 (one exponent for the lines of all
// three axes left 2e-10 at r = 6, and took 3% of a 256^3 step less).
#pragma once

#include "grf_fixed.cuh"

namespace grf {

// A box's factors and fixed-point range from its spacing, for a type with members f1, f2, f11 and fx.
template <typename Spacing>
void spacing_factors(Spacing& g, double dx, int ng) {
    const double d1 = ng == 4 ? 60.0 : 12.0, d2 = ng == 4 ? 180.0 : 12.0;
    g.f1 = fx_scale_of(1.0 / (d1 * dx));
    g.f2 = fx_scale_of(1.0 / (d2 * dx * dx));
    g.f11 = fx_scale_of(1.0 / (d1 * d1 * dx * dx));
    const int lo = g.f11.e < g.f1.e ? g.f11.e : g.f1.e, hi = g.f2.e > g.f1.e ? g.f2.e : g.f1.e;
    g.fx = fx_range(lo, hi, ng == 4 ? 10 : 0);
}

// Differences of one field at one point.
struct FieldDiffs {
    double d1[3], d2[6], ko;  // first and second derivatives, Kreiss-Oliger sum
    double up[3];             // lopsided first differences (LOP)
};

constexpr int kGuard4 = 5, kGuard6 = 8;  // guard bits of a line's values: below 2^58, 2^61

// x >> s rounded to nearest, s >= 1.
GRF_HD long long fx_sar_round(long long x, int s) { return (fx_sar_any(x, s - 1) + 1) >> 1; }

// ---- 4th order

// One field on the three axes through the point (19 values), and on one coordinate plane (16).
struct AxisValues {
    double c, m[3][3], q[3][3];  // the point; at -(k+1) and +(k+1) along axis d
};
struct PlaneValues {
    double x[4][4];  // at offsets -2, -1, 1, 2 along both axes
};

// The axis part: first derivatives, unmixed second derivatives and (KO = 1) the Kreiss-Oliger sum. Returns the
// largest magnitude word of the values read; the outermost ones, at +-3, are read for KO and LOP only.
//   LOP = 1: also the differences biased towards the side the shift component bet[d] points to (offsets
//   -1..3, mirrored for bet[d] < 0): (-3 b1 - 10 u0 + 18 a1 - 6 a2 + a3) / (12 dx) with a_n = u at n
//   points towards that side, b1 = u one point away from it.
// The bounds, of values below 2^58: first 18 x 2^58; a quarter of the second 16 x 2^58 and of the dissipation's
// 15.5 x 2^58; half the lopsided sum 18.5 x 2^58: all below 2^63.
template <int LOP, int KO, typename Spacing>
GRF_HD int axis_diffs(const Spacing& g, const AxisValues& v, bool first, bool second, const double* bet, FieldDiffs& r) {
    constexpr int G = kGuard4;
    const int mc = fx_mag(v.c);
    int mag = mc, e[3];
    long long inner[3];
#pragma unroll
    for (int d = 0; d < 3; ++d) {
        const int near = fx_max(fx_max(mc, fx_max(fx_mag(v.m[d][0]), fx_mag(v.q[d][0]))), fx_max(fx_mag(v.m[d][1]), fx_mag(v.q[d][1])));
        mag = fx_max(mag, near);
        const int ed = fx_max(near >> 20, g.fx.emin), lim = fx_lim<G>(ed);
        const long long c0 = fx_int(v.c, lim), c2 = c0 + c0;
        const long long m1 = fx_int(v.m[d][0], lim), q1 = fx_int(v.q[d][0], lim);
        const long long m2 = fx_int(v.m[d][1], lim), q2 = fx_int(v.q[d][1], lim);
        if (first) r.d1[d] = fx_value<G>(((q1 - m1) << 3) + (m2 - q2), ed, g.f1);
        if (second || KO) {
            const long long p1 = q1 + m1 - c2, p2 = q2 + m2 - c2;  // pair sums less 2 u0
            // a quarter of the sums: what their constant shifts drop is below 2^-57 of the largest value
            if (second) r.d2[d == 0 ? 0 : (d == 1 ? 3 : 5)] = fx_value<G - 2>((p1 << 2) - (p2 >> 2), ed, g.f2);
            // the dissipation's 15 p1 - 6 p2 - 2 u0, without u_-3 + u_3
            inner[d] = (p1 << 2) - (p1 >> 2) - p2 - (p2 >> 1) - (c0 >> 1);
            e[d] = ed;
        }
        if (LOP) {
            const bool fw = bet[d] >= 0.0;
            const double far = fw ? v.q[d][2] : v.m[d][2];
            long long u0 = c0, a1 = fw ? q1 : m1, a2 = fw ? q2 : m2, b1 = fw ? m1 : q1;
            int eb = fx_max(fx_max(fx_max(mc, fx_max(fx_mag(v.m[d][0]), fx_mag(v.q[d][0]))), fx_mag(fw ? v.q[d][1] : v.m[d][1])) >> 20, g.fx.emin);
            if (ed - eb > 2) {  // the point two away on the other side is not read: its size does not count
                const int lb = fx_lim<G>(eb);
                u0 = fx_int(v.c, lb);
                a1 = fx_int(fw ? v.q[d][0] : v.m[d][0], lb);
                a2 = fx_int(fw ? v.q[d][1] : v.m[d][1], lb);
                b1 = fx_int(fw ? v.m[d][0] : v.q[d][0], lb);
            } else {
                eb = ed;
            }
            const long long x = 9 * a1 - 3 * a2 - 5 * u0 - b1 - (b1 >> 1);  // half the sum without the far point
            const int eu = fx_max(eb, fx_mag(far) >> 20);  // the unit of the far point, three guard bits: 38 x 2^56
            r.up[d] = fx_value<3>(fx_sar_round(x, eu - eb + 1) + fx_int(far, fx_lim<3>(eu)), eu, g.f1);
            mag = fx_max(mag, fx_mag(far));
        }
    }
    if (KO) {  // the lines' sums and the six outermost points, two guard bits: 192 x 2^55
#pragma unroll
        for (int d = 0; d < 3; ++d) mag = fx_max(mag, fx_max(fx_mag(v.m[d][2]), fx_mag(v.q[d][2])));
        const int E = fx_max(mag >> 20, g.fx.emin), lim = fx_lim<2>(E);
        long long t = 0;
#pragma unroll
        for (int d = 0; d < 3; ++d)
            t += fx_int(v.m[d][2], lim) + fx_int(v.q[d][2], lim) + fx_sar_round(inner[d], E - e[d] + 1);
        r.ko = fx_value<2>(t, E);
    }
    return mag;
}

// The lines' sums d[a], in units of exponent e[a] each, in the finest common unit in which every |d[a]| is at
// most 2^bits[a]; E becomes its exponent.
template <int N>
GRF_HD void align_lines(long long (&d)[N], const int (&e)[N], const int (&bits)[N], int& E) {
    E = e[0];
#pragma unroll
    for (int a = 1; a < N; ++a) E = fx_max(E, e[a]);
    int left = 1 << 20;
#pragma unroll
    for (int a = 0; a < N; ++a) {
        const int z = fx_clz32(fx_top(d[a])) + (E - e[a]) - (64 - bits[a]);
        left = z < left ? z : left;
    }
#pragma unroll
    for (int a = 0; a < N; ++a) d[a] = fx_aligned(d[a], left - (E - e[a]));
    E -= left;
}

// A mixed derivative: the tensor product of the first-difference weights (1, -8, 8, -1) on its 16 points, the
// lines' differences (below 18 x 2^58), then the same of those (16 x 2^58 + 2 x 2^60 after alignment). mag collects the
// largest magnitude word.
template <typename Spacing>
GRF_HD double plane_diff(const Spacing& g, const PlaneValues& v, int& mag) {
    constexpr int G = kGuard4;
    long long d[4];
    int e[4], E;
#pragma unroll
    for (int a = 0; a < 4; ++a) {
        const int top = fx_max(fx_max(fx_mag(v.x[a][0]), fx_mag(v.x[a][1])), fx_max(fx_mag(v.x[a][2]), fx_mag(v.x[a][3])));
        mag = fx_max(mag, top);
        e[a] = fx_max(top >> 20, g.fx.emin);
        const int lim = fx_lim<G>(e[a]);
        d[a] = ((fx_int(v.x[a][2], lim) - fx_int(v.x[a][1], lim)) << 3) + (fx_int(v.x[a][0], lim) - fx_int(v.x[a][3], lim));
    }
    const int bits[4] = {60, 58, 58, 60};
    align_lines(d, e, bits, E);
    return fx_value<G>(((d[2] - d[1]) << 3) + (d[0] - d[3]), E, g.f11);
}

// ---- 6th order

struct AxisValues6 {
    double c, m[3][4], q[3][4];  // the point; at -(k+1) and +(k+1) along axis d
};
struct PlaneValues6 {
    double x[6][6];  // at offsets -3, -2, -1, 1, 2, 3 along both axes
};

// A 32nd of 45 d1 - 9 d2 + d3 of differences below 2^62 (110/32 x 2^61 < 2^63).
GRF_HD long long first6(long long d1, long long d2, long long d3) {
    return d1 + (d1 >> 2) + (d1 >> 3) + (d1 >> 5) - (d2 >> 2) - (d2 >> 5) + (d3 >> 5);
}

// As axis_diffs, 6th order; the outermost values are those at +-4.
//   second: |p1| < 2^54, |p2| < 2^56, |p3| < 2^59: 270 x 2^54 + 27 x 2^56 + 2^60 < 2^63;
//   a 64th of the dissipation's line sum 254/64 x 2^61, of the lopsided sum 179/64 x 2^61: below 2^63.
template <int LOP, int KO, typename Spacing>
GRF_HD int axis_diffs6(const Spacing& g, const AxisValues6& v, bool first, bool second, const double* bet, FieldDiffs& r) {
    constexpr int G = kGuard6;
    const int mc = fx_mag(v.c);
    int mag = mc, e[3];
    long long inner[3];
#pragma unroll
    for (int d = 0; d < 3; ++d) {
        int near = mc;
#pragma unroll
        for (int k = 0; k < 3; ++k) near = fx_max(near, fx_max(fx_mag(v.m[d][k]), fx_mag(v.q[d][k])));
        mag = fx_max(mag, near);
        const int ed = fx_max(near >> 20, g.fx.emin), lim = fx_lim<G>(ed);
        const long long c0 = fx_int(v.c, lim), c2 = c0 + c0;
        const long long m1 = fx_int(v.m[d][0], lim), q1 = fx_int(v.q[d][0], lim);
        const long long m2 = fx_int(v.m[d][1], lim), q2 = fx_int(v.q[d][1], lim);
        const long long m3 = fx_int(v.m[d][2], lim), q3 = fx_int(v.q[d][2], lim);
        const long long p1 = q1 + m1 - c2, p2 = q2 + m2 - c2, p3 = q3 + m3 - c2;  // pair sums less 2 u0
        if (first) r.d1[d] = fx_value<G - 5>(first6(q1 - m1, q2 - m2, q3 - m3), ed, g.f1);
        if (second) {
            const int sh = fx_room(fx_top(p1) | fx_top(p2) >> 2 | fx_top(p3) >> 5, 54);
            r.d2[d == 0 ? 0 : (d == 1 ? 3 : 5)] =
                fx_value<G>(270 * fx_sar(p1, sh) - 27 * fx_sar(p2, sh) + 2 * fx_sar(p3, sh), ed + sh, g.f2);
        }
        if (KO) {
            // a 64th of 28 p2 - 56 p1 - 8 p3 - 2 u0, the dissipation without u_-4 + u_4
            inner[d] = (p2 >> 1) - (p2 >> 4) - p1 + (p1 >> 3) - (p3 >> 3) - (c0 >> 5);
            e[d] = ed + 6;
        }
        if (LOP) {
            const bool fw = bet[d] >= 0.0;
            const double far = fw ? v.q[d][3] : v.m[d][3];
            long long u0 = c0, a1 = fw ? q1 : m1, a2 = fw ? q2 : m2, a3 = fw ? q3 : m3, b1 = fw ? m1 : q1, b2 = fw ? m2 : q2;
            int eb = mc;
#pragma unroll
            for (int k = 0; k < 2; ++k) eb = fx_max(eb, fx_max(fx_mag(v.m[d][k]), fx_mag(v.q[d][k])));
            eb = fx_max(fx_max(eb, fx_mag(fw ? v.q[d][2] : v.m[d][2])) >> 20, g.fx.emin);
            if (ed - eb > 2) {  // the point three away on the other side is not read: its size does not count
                const int lb = fx_lim<G>(eb);
                u0 = fx_int(v.c, lb);
                a1 = fx_int(fw ? v.q[d][0] : v.m[d][0], lb);
                a2 = fx_int(fw ? v.q[d][1] : v.m[d][1], lb);
                a3 = fx_int(fw ? v.q[d][2] : v.m[d][2], lb);
                b1 = fx_int(fw ? v.m[d][0] : v.q[d][0], lb);
                b2 = fx_int(fw ? v.m[d][1] : v.q[d][1], lb);
            } else {
                eb = ed;
            }
            // a 64th of 80 a1 - 30 a2 + 8 a3 - 24 b1 + 2 b2 - 35 u0
            const long long x = (a1 + (a1 >> 2)) - ((a2 >> 1) - (a2 >> 5)) + (a3 >> 3) - ((b1 >> 2) + (b1 >> 3)) + (b2 >> 5) -
                                ((u0 >> 1) + (u0 >> 5) + (u0 >> 6));
            const int eu = fx_max(eb, fx_mag(far) >> 20);  // the unit of the far point, one guard bit: 180 x 2^54
            r.up[d] = fx_value<1>(fx_sar_round(x, eu - eb + 1) - fx_int(far, fx_lim<1>(eu)), eu, g.f1);
            mag = fx_max(mag, fx_mag(far));
        }
    }
    if (KO) {  // the lines' sums, and that of the six outermost points with five guard bits
        int out = 0;
#pragma unroll
        for (int d = 0; d < 3; ++d) out = fx_max(out, fx_max(fx_mag(v.m[d][3]), fx_mag(v.q[d][3])));
        mag = fx_max(mag, out);
        const int eo = fx_max(out >> 20, g.fx.emin), lim = fx_lim<5>(eo);
        long long t[4] = {inner[0], inner[1], inner[2], 0};
#pragma unroll
        for (int d = 0; d < 3; ++d) t[3] += fx_int(v.m[d][3], lim) + fx_int(v.q[d][3], lim);
        const int et[4] = {e[0], e[1], e[2], eo + G - 5};
        int E;
        const int bits[4] = {60, 60, 60, 60};
        align_lines(t, et, bits, E);
        r.ko = fx_value<G>((t[0] + t[1]) + (t[2] + t[3]), E);
    }
    return mag;
}

// As plane_diff, 6th order: weights (-1, 9, -45, 45, -9, 1) on 36 points, 90 x 2^55 + 18 x 2^57 + 2 x 2^60 after
// alignment: < 2^63.
template <typename Spacing>
GRF_HD double plane_diff6(const Spacing& g, const PlaneValues6& v, int& mag) {
    constexpr int G = kGuard6;
    long long d[6];
    int e[6], E;
#pragma unroll
    for (int a = 0; a < 6; ++a) {
        int top = 0;
#pragma unroll
        for (int b = 0; b < 6; ++b) top = fx_max(top, fx_mag(v.x[a][b]));
        mag = fx_max(mag, top);
        const int ed = fx_max(top >> 20, g.fx.emin), lim = fx_lim<G>(ed);
        d[a] = first6(fx_int(v.x[a][3], lim) - fx_int(v.x[a][2], lim), fx_int(v.x[a][4], lim) - fx_int(v.x[a][1], lim),
                      fx_int(v.x[a][5], lim) - fx_int(v.x[a][0], lim));
        e[a] = ed;
    }
    const int bits[6] = {60, 57, 55, 55, 57, 60};
    align_lines(d, e, bits, E);
    return fx_value<G - 5>(45 * (d[3] - d[2]) - 9 * (d[4] - d[1]) + (d[5] - d[0]), E, g.f11);
}

}  // namespace grf
