// Pointwise right-hand side of the modified CCZ4 + 4dST system (FP64, one grid point per
// thread, everything in registers / local memory).
//
// The 4dST sources are written in explicit 3+1 form. With the basis (n, d_i) the 4D
// Riemann tensor splits into
//     S_ij  = gamma^kl R_kilj           = R_ij + K K_ij - K_ik K^k_j          (Gauss block)
//     B_kij = R_{n k i j}               = D_i K_kj - D_j K_ki                (Codazzi block)
//     C_ij  = R_{n i n j}               = (d_t K_ij - L_beta K_ij + D_i D_j lapse)/lapse
//                                          + K_ik K^k_j                        (Ricci equation)
// and the double dual P has the closed form
//     P_ninj = S_ij - gamma_ij S / 2,   P_nkij = B_kij - gamma_ki B_j + gamma_kj B_i,
//     P_ijkl = gamma_ik C_jl - gamma_il C_jk - gamma_jk C_il + gamma_jl C_ik - C (g_ik g_jl - g_il g_jk),
// with B_j = gamma^ab B_abj. Then
//     L_GB   = 8 G_S^ij C_ij - 4 B_kij B^kij + 8 B_i B^i            (G_S = S - gamma S/2)
//     8 pi rho  = rho1 - 4 G_S^ij Phi_ij
//     8 pi S_i  = S1_i + 4 [G_S ik Phi_n^k + B_kil Phi^kl - Phi_i^l B_l + tr(Phi) B_i]
//     8 pi S_ij = S1_ij - 4 [G_S ij Phi_nn + Y_ij + Q_ij(C)]
// where Phi_ab = nabla_a nabla_b beta(phi) and the first-order (X, X^2) parts rho1, S1 are
// those of (1/16 pi)(X + g2 X^2). C_ij (through d_t K_ij) and Phi_nn (through d_t Pi) are
// the only places the unknowns enter, affinely: the 7x7 system M v = r for v = (C_ij, H_nn), which hold
// d_t K_ij and d_t Pi, is assembled from these expressions and solved by LU with partial pivoting.
//
// What bounds it: the FP64 pipe (2 lanes per SM and clock), one instruction at a time, so the formulas are
// chosen by their instruction count. The curvature goes through the six components of the 3D Riemann
// tensor (its double dual is the raised Einstein tensor), the derivatives of Gt^k that cancel between
// R_ij and D_(i Z_j) are never formed, and C_ij and H_nn are the unknowns, in which the lapse's
// derivatives and the shift terms cancel. About 2,000 FP64 instructions where the forms through
// d_m (h^ij Gt_lij) and d_t K_ij took 2,900: by itself 256^3 step 506 -> 412 ms, 36 x 32 x 30 gradient (whose
// tape has one entry per operation) 76.9 -> 52.7 ms, 72^2 x 60 diagnostics 6.57 -> 4.97 ms.
// Products and sums are fused only where fma is written (-fmad=false), so all instantiations round alike.
//
// Rounding: near a puncture the curvature's chi part is large and cancels, so the order counts. The small terms of
// R^Z_ij are summed before the chi part is added, the scalar curvature's chi part is taken in closed form, the
// system is solved for the departure of (C_ij, H_nn) from its right-hand side, and K and A_ij take that right-hand
// side and the departure apart. Errors against long double, near one of two punctures, over those of the plain
// formulation (Ricci tensor and D_i Z_j term by term, S_ij from the solution): off-diagonal d_t A_ij 1.0 (2.1 to 2.6
// with the chi part summed first and A_ij from the eliminated C_ij), K 1.07 (1.4), Theta 1.03 (1.5), all fields 0.9.
// It takes about 80 instructions more: 256^3 step 296 -> 306 ms when it came in.
//
// The cubic Horndeski term (1/16 pi) g3 X box(phi) (general instantiation, COUP = 1) adds, with
// H = nabla nabla phi in the same basis (H_nn holding d_t Pi, H_ni, H_ij = D_i D_j phi + K_ij Pi),
//     8 pi rho3  = g3/2 (Pi^2 tr H - H(dphi, dphi))
//     8 pi S3_i  = -g3/2 [(Pi tr H - H_n(dphi)) d_i phi + Pi^2 H_ni - Pi H_ik d^k phi]
//     8 pi S3_ij = g3 [1/2 H_nn (Pi^2 gamma_ij - d_i phi d_j phi) + 1/2 tr H d_i phi d_j phi
//                      + Pi H_n(i d_j) phi - H_(i|k d^k phi d_|j) phi + gamma_ij (H(dphi, dphi)/2 - Pi H_n(dphi))]
// to the metric equations, and to the scalar equation
//     g3 [box(phi)^2 - H_ab H^ab - R_ab d^a phi d^b phi],
// in which H_nn^2 cancels: -2 H_nn tr H + (tr H)^2 + 2 H_n.H_n - H_ij H^ij
// - (Pi^2 gamma^kl - d^k phi d^l phi) C_kl - 2 Pi B^i d_i phi - S_ij d^i phi d^j phi
// (4D Ricci: R_nn = tr C, R_ni = -B_i, R_ij = S_ij - C_ij). The system stays affine in the unknowns.
#pragma once

#include <type_traits>

#ifdef __CUDACC__
#include <cuda_runtime.h>
#define GRF_HD __host__ __device__ __forceinline__
#else
#include <cmath>
#define GRF_HD inline
#define __host__
#define __device__
#endif

// Section markers: no-ops in the CUDA build; the host operation-counting build defines them
// to attribute FP64 operations to the parts of the algorithm.
#ifndef GRF_SECTION
#define GRF_SECTION(id)
#endif
// Marks a value as data (not a known constant) in the counting build: compare-and-exchange
// pivoting turns every swapped entry into a runtime value.
#ifndef GRF_OPAQUE
#define GRF_OPAQUE(x)
#endif

namespace grf {

// d1 slots: fields 0..21 keep their index, phi -> 22, Pi -> 23 (B^i has no derivative)
__host__ __device__ constexpr int d1slot(int f) { return f < 22 ? f : (f == 25 ? 22 : 23); }
// d2 slots: chi 0, h 1..6, lapse 7, shift 8..10, phi 11
__host__ __device__ constexpr int d2slot(int f) { return f < 7 ? f : (f == 18 ? 7 : (f < 22 ? f - 11 : 11)); }
__host__ __device__ constexpr int sidx(int i, int j) {
    return i <= j ? (i == 0 ? j : (i == 1 ? 2 + j : 5)) : (j == 0 ? i : (j == 1 ? 2 + i : 5));
}

enum { F_CHI = 0, F_H = 1, F_K = 7, F_A = 8, F_TH = 14, F_GAM = 15, F_LAPSE = 18, F_SHIFT = 19,
       F_B = 22, F_PHI = 25, F_PI = 26, NFIELDS = 27 };

// Per-launch coefficients. P is the type of the two couplings (double, or a dual number when
// their tangents are propagated).
template <typename P>
struct CoeffsT {
    double kappa1, kappa2, kappa3, shift_F, eta;
    P lam, g2;
    double inv_1pa, a_1pa;        // 1/(1+a), a/(1+a)
    double bK, bTh;               // 3b/(4(1+b)), 1/(2(1+b))
    int beta_kind;
    double beta_kappa;  // kappa of the exponential coupling (beta_kind 2)
    int decoupled;  // 1: the scalar's stress-energy is left out of the metric equations
    int advection;  // 1: lopsided advection derivatives (kernels instantiated with LOP = 1)
    double g3;      // cubic Horndeski coupling (read only by COUP = 1 instances)
};
using Coeffs = CoeffsT<double>;

template <typename T>
struct PointInT {
    T v[NFIELDS];
    T d1[24][3];
    T d2[12][6];
};
using PointIn = PointInT<double>;

// Output diagnostics besides the RHS (constraints come out as by-products).
template <typename T>
struct PointExtraT {
    T ham;      // H = S - 2 (8 pi rho)
    T mom[3];   // M_i = B_i - 8 pi S_i
    T rho8[3];  // 8 pi rho of the X, g2 X^2 and beta(phi) L_GB terms of the action (their sum is
                // the 8 pi rho of the equations when g3 = 0; reported with and without backreaction)
    // Weyl scalar Psi_4 (double instances only), computed when want_psi4 is set: xyz are the
    // point's coordinates relative to the origin of the tetrad's triad.
    int want_psi4 = 0;
    double xyz[3];
    T psi4[2];
    // Hyperbolicity diagnostics (double instances only), computed when want_hyp is set:
    //   hyp[0] = det M of the coupled system for (d_t K_ij, d_t Pi), normalised so that each
    //            unknown's own coefficient is 1 (M = identity without coupling); where it
    //            vanishes the equations no longer determine the time derivatives;
    //   hyp[1] = det(g_eff^ab) / det(g^ab) of the scalar equation's principal symbol
    //            g_eff^ab = (1 + 2 g2 X) g^ab - 2 g2 d^a phi d^b phi + 2 g3 (box(phi) g^ab - H^ab);
    //            for g3 = 0, by the matrix determinant lemma, (1 + 2 g2 X)^3 (1 + 6 g2 X);
    //   hyp[2] = -g_eff^nn = 1 + 2 g2 X + 2 g2 Pi^2 + 2 g3 tr H (the coefficient of d_t Pi; the
    //            normal is timelike for the scalar's characteristic cone while it is positive);
    //   hyp[3] = the smallest pivot of partial-pivoting elimination of M over its largest entry.
    int want_hyp = 0;
    double hyp[4];
};
using PointExtra = PointExtraT<double>;

// a0 b0 + a1 b1 + a2 b2, and c - a b
template <typename T>
GRF_HD T dot3(const T& a0, const T& b0, const T& a1, const T& b1, const T& a2, const T& b2) {
    return fma(a2, b2, fma(a1, b1, a0 * b0));
}
template <typename T>
GRF_HD T fnma(const T& a, const T& b, const T& c) { return fma(-a, b, c); }

// x / 2 and 2 x. For doubles on the device these step the exponent on the integer pipe, which runs
// beside the FP64 pipe (2 lanes per SM and clock against 64); zeros, infinities, NaNs and the ends of
// the exponent range pass through unchanged.
template <typename T>
GRF_HD T half_of(const T& x) { return 0.5 * x; }
template <typename T>
GRF_HD T twice_of(const T& x) { return 2.0 * x; }
// 1 / x. For doubles on the device: the approximate reciprocal (20 bits) and three Newton-Raphson steps
// y <- y + y (1 - x y), 6 FP64 instructions in place of a division's 9. After two steps y is within one unit in the
// last place, so that 1 - x y is exact and the third gives the correctly rounded reciprocal, but for x of a mantissa
// of all ones (P. Markstein, IBM J. Res. Dev. 34, 1990, theorem 7.2). Outside 2^-1022 .. 2^1021 the approximation
// itself is the result: infinities of zeros (and of subnormal x), zeros of infinities, NaNs, and of larger finite x
// 20 bits or zero. (The choice is made on the integer pipe; a branch to a scaled path cost 4% of a 128^3 step, the
// third step nothing measurable.)
template <typename T>
GRF_HD T recip(const T& x) { return 1.0 / x; }
#ifdef __CUDA_ARCH__
__device__ __forceinline__ double recip(const double& x) {
    double y0;
    asm("rcp.approx.ftz.f64 %0, %1;" : "=d"(y0) : "d"(x));
    double y = fma(y0, fma(-x, y0, 1.0), y0);
    y = fma(y, fma(-x, y, 1.0), y);
    y = fma(y, fma(-x, y, 1.0), y);
    const unsigned e = ((unsigned)__double2hiint(x) << 1) - (1u << 21);
    return e < (2043u << 21) ? y : y0;
}
__device__ __forceinline__ double exponent_step(double x, int step) {
    const int hi = __double2hiint(x);
    const unsigned e = ((unsigned)hi << 1) - (2u << 21);
    return __hiloint2double(e < (0x7fcu << 21) ? hi + step : hi, __double2loint(x));
}
__device__ __forceinline__ double half_of(const double& x) { return exponent_step(x, -(1 << 20)); }
__device__ __forceinline__ double twice_of(const double& x) { return exponent_step(x, 1 << 20); }
#endif

template <typename T>
GRF_HD T sym3_det(const T h[6]) {
    const T a = fnma(h[4], h[4], h[3] * h[5]), b = fnma(h[1], h[5], h[4] * h[2]), d = fnma(h[3], h[2], h[1] * h[4]);
    return dot3(h[0], a, h[1], b, h[2], d);
}

// A value of the point's data, read where it is used. For doubles on the device the read is volatile: kept in
// registers from an early read, the 198 values of a point would only be spilled and read back from there.
template <typename T>
GRF_HD T at_use(const T& x) { return x; }
#ifdef __CUDA_ARCH__
__device__ __forceinline__ double at_use(const double& x) { return *(const volatile double*)&x; }
#endif

// Symmetric inverse; returns the determinant. For h near the unit matrix, as here: the small products are
// rounded first, the large ones enter in a fused step.
template <typename T>
GRF_HD T sym3_inv(const T h[6], T hi[6], T& id) {
    const T c00 = fma(h[3], h[5], -(h[4] * h[4]));
    const T c01 = fnma(h[1], h[5], h[2] * h[4]);
    const T c02 = fnma(h[2], h[3], h[1] * h[4]);
    const T det = dot3(h[2], c02, h[1], c01, h[0], c00);
    id = recip(det);
    hi[0] = c00 * id;
    hi[1] = c01 * id;
    hi[2] = c02 * id;
    hi[3] = fma(h[0], h[5], -(h[2] * h[2])) * id;
    hi[4] = fnma(h[0], h[4], h[1] * h[2]) * id;
    hi[5] = fma(h[0], h[3], -(h[1] * h[1])) * id;
    return det;
}

// |a| > |b|, and the largest |M_ij| of the 7x7 block. For doubles on the device both run on the
// integer pipe: with the sign bit cleared, the bit patterns of non-NaN doubles order like their
// magnitudes (a NaN entry makes the maximum a NaN, which then fails every pivot test).
template <typename T>
GRF_HD bool abs_gt(const T& a, const T& b) { return fabs(a) > fabs(b); }
template <typename T>
GRF_HD T abs_max7(const T M[7][8]) {
    T mx = 0.0;
#pragma unroll
    for (int i = 0; i < 7; ++i)
#pragma unroll
        for (int j = 0; j < 7; ++j) mx = fmax(mx, fabs(M[i][j]));
    return mx;
}
#ifdef __CUDA_ARCH__
__device__ __forceinline__ long long abs_bits(double x) { return __double_as_longlong(x) & 0x7fffffffffffffffLL; }
__device__ __forceinline__ bool abs_gt(double a, double b) { return abs_bits(a) > abs_bits(b); }
__device__ __forceinline__ double abs_max7(const double M[7][8]) {
    long long m = 0;
#pragma unroll
    for (int i = 0; i < 7; ++i)
#pragma unroll
        for (int j = 0; j < 7; ++j) m = max(m, abs_bits(M[i][j]));
    return __longlong_as_double(m);
}
#endif

// Determinant of the 7x7 block of M (a copy, Gaussian elimination with partial pivoting and the
// sign of each row exchange), and in *ratio the smallest pivot magnitude over the block's largest
// entry magnitude. Diagnostics only.
GRF_HD double det7(const double M[7][8], double* ratio) {
    double A[7][7], mx = 0.0, mn = -1.0;
    for (int i = 0; i < 7; ++i)
        for (int j = 0; j < 7; ++j) { A[i][j] = M[i][j]; mx = fmax(mx, fabs(A[i][j])); }
    *ratio = 0.0;
    double det = 1.0;
    for (int k = 0; k < 7; ++k) {
        int piv = k;
        for (int i = k + 1; i < 7; ++i)
            if (fabs(A[i][k]) > fabs(A[piv][k])) piv = i;
        const double pm = fabs(A[piv][k]);
        mn = (mn < 0.0 || pm < mn) ? pm : mn;
        if (A[piv][k] == 0.0) return 0.0;
        if (piv != k) {
            for (int j = 0; j < 7; ++j) {
                const double t = A[k][j];
                A[k][j] = A[piv][j];
                A[piv][j] = t;
            }
            det = -det;
        }
        det *= A[k][k];
        for (int i = k + 1; i < 7; ++i) {
            const double f = A[i][k] / A[k][k];
            for (int j = k + 1; j < 7; ++j) A[i][j] = fma(-f, A[k][j], A[i][j]);
        }
    }
    *ratio = mx > 0.0 ? mn / mx : 0.0;
    return det;
}

// 7x7 LU with partial pivoting (row swaps by compare-and-exchange, so every index stays a
// compile-time constant and the matrix stays in registers); the pivot rows are not normalised,
// the back substitution multiplies by the stored pivot reciprocals. Returns false on a pivot
// not larger than 1e-300 times the largest entry.
template <typename T>
GRF_HD bool solve7(T M[7][8]) {
    const T thr = 1e-300 * abs_max7(M);
    bool ok = true;
    T ipv[7];
#pragma unroll
    for (int k = 0; k < 7; ++k) {
#pragma unroll
        for (int i = k + 1; i < 7; ++i) {
            const bool sw = abs_gt(M[i][k], M[k][k]);
#pragma unroll
            for (int j = k; j < 8; ++j) {
                const T a = M[k][j], b = M[i][j];
                M[k][j] = sw ? b : a;
                M[i][j] = sw ? a : b;
                GRF_OPAQUE(M[k][j]);
                GRF_OPAQUE(M[i][j]);
            }
        }
        ok = ok && abs_gt(M[k][k], thr);
        const T ip = recip(M[k][k]);
        ipv[k] = ip;
#pragma unroll
        for (int i = k + 1; i < 7; ++i) {
            const T f = M[i][k] * ip;
#pragma unroll
            for (int j = k + 1; j < 8; ++j) M[i][j] = fma(-f, M[k][j], M[i][j]);
        }
    }
#pragma unroll
    for (int k = 6; k >= 0; --k) {
        T x = M[k][7];
#pragma unroll
        for (int j = k + 1; j < 7; ++j) x = fma(-M[k][j], M[j][7], x);
        M[k][7] = x * ipv[k];
    }
    return ok;
}

// sum_ij a_ij b^ij for symmetric a, b stored as 6 components, with `bw` = b with the three
// off-diagonal components pre-multiplied by 2.
template <typename T>
GRF_HD T sdotw(const T a[6], const T bw[6]) {
    return fma(a[5], bw[5], fma(a[4], bw[4], fma(a[3], bw[3], dot3(a[0], bw[0], a[1], bw[1], a[2], bw[2]))));
}

// Levi-Civita bookkeeping of the Codazzi block: B_kij (antisymmetric in ij) is stored through
// its dual bb[k][m] = B_{k,(m+1)%3,(m+2)%3}; B_kij = +-bb[k][3-i-j] for i != j.
__host__ __device__ constexpr int third(int i, int j) { return 3 - i - j; }
__host__ __device__ constexpr bool cyclic(int i, int j) { return (j - i + 3) % 3 == 1; }

// DEC: the decoupled mode as a compile-time constant (0: full theory, 1: no backreaction), or -1
// to read c.decoupled at run time.
// LOP = 1: every advection term beta^k d_k u of an evolved field (the CCZ4 advection terms and
// the shift-contracted derivatives of K_ij and Pi inside the coupled system) is taken from
// adv[27], the lopsided differences; all other derivatives stay centred. adv is not read when
// LOP = 0. COUP = 0 compiles the linear and quadratic couplings only (the exponential one is then
// routed to another instantiation by the host).
template <typename T, typename P = double, int DEC = -1, int LOP = 0, int COUP = 1>
GRF_HD void point_rhs(const CoeffsT<P>& c, const PointInT<T>& in, T rhs[NFIELDS], PointExtraT<T>* extra, bool& ok,
                      const T* adv = nullptr) {
    GRF_SECTION(0);
    const T* v = in.v;
    const T chi = v[F_CHI], K = v[F_K], Th = v[F_TH], al = v[F_LAPSE], phi = v[F_PHI], Pi = v[F_PI];
    T h[6], A[6];
#pragma unroll
    for (int m = 0; m < 6; ++m) { h[m] = v[F_H + m]; A[m] = v[F_A + m]; }
    T hi[6], ideth;
    sym3_inv(h, hi, ideth);
    const T ichi = recip(chi);
    // weighted inverses (off-diagonals doubled) for symmetric contractions; gamma^ij = chi h^ij
    T hw[6], gu[6], gw[6], gd[6];
#pragma unroll
    for (int m = 0; m < 6; ++m) {
        const bool off = (m == 1 || m == 2 || m == 4);
        hw[m] = off ? twice_of(hi[m]) : hi[m];
        gu[m] = chi * hi[m];
        gw[m] = off ? twice_of(gu[m]) : gu[m];
        gd[m] = h[m] * ichi;
    }

    GRF_SECTION(1);
#define D1(f, k) at_use(in.d1[d1slot(f)][k])
#define D2(f, m) at_use(in.d2[d2slot(f)][m])
#define DH1(k, m) D1(F_H + (m), k) /* d_k h_m */
    T dchi[3], dphi[3];
#pragma unroll
    for (int k = 0; k < 3; ++k) {
        dchi[k] = D1(F_CHI, k); dphi[k] = D1(F_PHI, k);
    }
    const T divb = D1(F_SHIFT, 0) + D1(F_SHIFT + 1, 1) + D1(F_SHIFT + 2, 2);
    
#define ADV(f) (LOP ? adv[f] : dot3(at_use(v[F_SHIFT]), D1(f, 0), at_use(v[F_SHIFT + 1]), D1(f, 1), at_use(v[F_SHIFT + 2]), D1(f, 2)))

    // ---- the right-hand sides that need no curvature
    {
        const T divb23 = (2.0 / 3.0) * divb, al2 = twice_of(al);
        rhs[F_CHI] = fma((2.0 / 3.0) * chi, fma(al, K, -divb), ADV(F_CHI));
        T db[3][3];  // db[j][i] = d_j beta^i
#pragma unroll
        for (int j = 0; j < 3; ++j)
#pragma unroll
            for (int i = 0; i < 3; ++i) db[j][i] = D1(F_SHIFT + i, j);
#pragma unroll
        for (int i = 0; i < 3; ++i)
#pragma unroll
            for (int j = i; j < 3; ++j) {
                T x = fnma(h[sidx(i, j)], divb23, fnma(al2, A[sidx(i, j)], ADV(F_H + sidx(i, j))));
                if (i == j) {
                    x = fma(2.0, dot3(h[sidx(i, 0)], db[i][0], h[sidx(i, 1)], db[i][1], h[sidx(i, 2)], db[i][2]), x);
                } else {
#pragma unroll
                    for (int k = 0; k < 3; ++k) x = fma(h[sidx(i, k)], db[j][k], fma(h[sidx(j, k)], db[i][k], x));
                }
                rhs[F_H + sidx(i, j)] = x;
            }
        const T dal[3] = {D1(F_LAPSE, 0), D1(F_LAPSE, 1), D1(F_LAPSE, 2)};
#pragma unroll
        for (int i = 0; i < 3; ++i)
            rhs[F_SHIFT + i] = fma(c.shift_F * c.inv_1pa, v[F_B + i],
                                   -((c.a_1pa * al * chi) * dot3(hi[sidx(i, 0)], dal[0], hi[sidx(i, 1)], dal[1],
                                                                 hi[sidx(i, 2)], dal[2])));
    }
    const T K2Th = K - twice_of(Th);
    rhs[F_LAPSE] = fma(-2.0 * c.inv_1pa * al, K2Th, ADV(F_LAPSE));
    rhs[F_PHI] = fma(al, Pi, ADV(F_PHI));

    // ---- conformal Christoffels: G1[l][ij] = Gt_{l ij}, G2[k][ij] = Gt^k_ij,
    //      Gl_l = h^ij Gt_lij (= h_lk Gt^k), Gtc^k = h^kl Gl_l. Where two of the indices of Gt_lij agree
    //      two of its three derivatives cancel: Gt_llj = d_j h_ll / 2, Gt_lii = d_i h_li - d_l h_ii / 2.
    GRF_SECTION(2);
    T G1[3][6], G2[3][6], Gl[3], Gtc[3];
#pragma unroll
    for (int l = 0; l < 3; ++l)
#pragma unroll
        for (int i = 0; i < 3; ++i)
#pragma unroll
            for (int j = i; j < 3; ++j) {
                const int m = sidx(i, j);
                if (i == l || j == l) G1[l][m] = half_of(DH1(i == l ? j : i, sidx(l, l)));
                else if (i == j) G1[l][m] = fma(-0.5, DH1(l, m), DH1(i, sidx(l, i)));
                else G1[l][m] = half_of(DH1(i, sidx(l, j)) + DH1(j, sidx(l, i)) - DH1(l, m));
            }
#pragma unroll
    for (int l = 0; l < 3; ++l) Gl[l] = sdotw(G1[l], hw);
#pragma unroll
    for (int k = 0; k < 3; ++k) {
        Gtc[k] = dot3(hi[sidx(k, 0)], Gl[0], hi[sidx(k, 1)], Gl[1], hi[sidx(k, 2)], Gl[2]);
#pragma unroll
        for (int m = 0; m < 6; ++m)
            G2[k][m] = dot3(hi[sidx(k, 0)], G1[0][m], hi[sidx(k, 1)], G1[1][m], hi[sidx(k, 2)], G1[2][m]);
    }

    // ---- the six components of the conformal Riemann tensor (1212, 1213, 1223, 1313, 1323, 2323)
    //   Rt_iklm = (d_k d_l h_im + d_i d_m h_kl - d_k d_m h_il - d_i d_l h_km)/2 + Gt^n_kl Gt_nim - Gt^n_km Gt_nil.
    // In three dimensions they hold the whole curvature: its contraction takes 21 products, where the
    // Ricci tensor written through d_m (h^ij Gt_lij) differentiates h^ij and takes about 300 more.
    GRF_SECTION(3);
#define DH(a, b, c, d) D2(F_H + sidx(a, b), sidx(c, d)) /* d_c d_d h_ab */
    T Rm[6];
    {
        auto riem = [&](int i, int k, int l, int m) -> T {
            T x = (i == l && k == m) ? twice_of(DH(i, k, i, k)) - (DH(i, i, k, k) + DH(k, k, i, i))
                                     : (DH(i, m, k, l) + DH(k, l, i, m)) - (DH(i, l, k, m) + DH(k, m, i, l));
            x = half_of(x);
#pragma unroll
            for (int n = 0; n < 3; ++n)
                x = fma(G2[n][sidx(k, l)], G1[n][sidx(i, m)], fnma(G2[n][sidx(k, m)], G1[n][sidx(i, l)], x));
            return x;
        };
        Rm[0] = riem(0, 1, 0, 1);
        Rm[1] = riem(0, 1, 0, 2);
        Rm[2] = riem(0, 1, 1, 2);
        Rm[3] = riem(0, 2, 0, 2);
        Rm[4] = riem(0, 2, 1, 2);
        Rm[5] = riem(1, 2, 1, 2);
    }

    // ---- physical Christoffels Gp^k_ij = Gt^k_ij - (delta^k_i d_j chi + delta^k_j d_i chi - h_ij h^kl d_l chi)/(2 chi)
    GRF_SECTION(4);
    const T hichi = half_of(ichi);
    T hidchi[3], c1[3], c2[3];
#pragma unroll
    for (int k = 0; k < 3; ++k) {
        hidchi[k] = dot3(hi[sidx(k, 0)], dchi[0], hi[sidx(k, 1)], dchi[1], hi[sidx(k, 2)], dchi[2]);
        c1[k] = hichi * dchi[k];
        c2[k] = hichi * hidchi[k];
    }
    T Gp[3][6];
#pragma unroll
    for (int k = 0; k < 3; ++k)
#pragma unroll
        for (int i = 0; i < 3; ++i)
#pragma unroll
            for (int j = i; j < 3; ++j) {
                T t = fma(h[sidx(i, j)], c2[k], G2[k][sidx(i, j)]);
                if (k == j) t = t - c1[i];
                if (k == i) t = t - c1[j];
                Gp[k][sidx(i, j)] = t;
            }

    // ---- the chi part of the curvature of gamma = h/chi: with
    //   T_ij = D~_i D~_j chi/(2 chi) - d_i chi d_j chi/(4 chi^2) - h_ij |d chi|^2/(8 chi^2) = Pc_ij + ch8 h_ij
    // chi Riem_iklm = Rt_iklm + h_il T_km + h_km T_il - h_im T_kl - h_kl T_im.
    GRF_SECTION(5);
    T Pc[6], chiLap, dchi2;
    const T qichi2 = -(hichi * hichi);
    const T chidet = chi * ideth;
    // The Einstein tensor is minus the double dual of Riemann, G^11 = -Riem_2323/det gamma and so on, so the
    // scalar curvature is -2 gamma_ij G^ij. Its conformal part, chi R~, is taken here; the chi part follows in
    // closed form, 2 D~^2 chi - 5 |d chi|^2/(2 chi): near a puncture its two terms cancel, and their rounding
    // stays out of D_i Z^i = (R^Z - R)/2, which needs the conformal parts only.
    T Rconf;
    {
        T dg = dot3(h[0], Rm[5], h[3], Rm[3], h[5], Rm[0]);
        const T off = fnma(h[1], Rm[4], fnma(h[4], Rm[1], h[2] * Rm[2]));
        dg = fma(2.0, off, dg);
        Rconf = twice_of(chidet) * dg;
    }
    {
        T DDchi[6];
#pragma unroll
        for (int m = 0; m < 6; ++m)
            DDchi[m] = fnma(G2[0][m], dchi[0], fnma(G2[1][m], dchi[1], fnma(G2[2][m], dchi[2], D2(F_CHI, m))));
        {
            T d2chi[6];
#pragma unroll
            for (int m = 0; m < 6; ++m) d2chi[m] = D2(F_CHI, m);
            chiLap = sdotw(d2chi, hw) - dot3(Gtc[0], dchi[0], Gtc[1], dchi[1], Gtc[2], dchi[2]);
        }
        dchi2 = dot3(dchi[0], hidchi[0], dchi[1], hidchi[1], dchi[2], hidchi[2]);
#pragma unroll
        for (int i = 0; i < 3; ++i) {
            const T qd = qichi2 * dchi[i];
#pragma unroll
            for (int j = i; j < 3; ++j) Pc[sidx(i, j)] = fma(hichi, DDchi[sidx(i, j)], qd * dchi[j]);
        }
        const T ch8 = half_of(qichi2 * dchi2);
        T Tc[6];
#pragma unroll
        for (int m = 0; m < 6; ++m) Tc[m] = fma(ch8, h[m], Pc[m]);
        auto wedge = [&](int i, int k, int l, int m, T x) -> T {
            if (i == l && k == m)
                return fma(h[sidx(i, i)], Tc[sidx(k, k)], fma(h[sidx(k, k)], Tc[sidx(i, i)],
                           fnma(twice_of(h[sidx(i, k)]), Tc[sidx(i, k)], x)));
            x = fma(h[sidx(i, l)], Tc[sidx(k, m)], fma(h[sidx(k, m)], Tc[sidx(i, l)], x));
            return fnma(h[sidx(i, m)], Tc[sidx(k, l)], fnma(h[sidx(k, l)], Tc[sidx(i, m)], x));
        };
        Rm[0] = wedge(0, 1, 0, 1, Rm[0]);
        Rm[1] = wedge(0, 1, 0, 2, Rm[1]);
        Rm[2] = wedge(0, 1, 1, 2, Rm[2]);
        Rm[3] = wedge(0, 2, 0, 2, Rm[3]);
        Rm[4] = wedge(0, 2, 1, 2, Rm[4]);
        Rm[5] = wedge(1, 2, 1, 2, Rm[5]);
    }
    const T Rs = Rconf + fma(-5.0 * hichi, dchi2, twice_of(chiLap));

    // ---- Z terms: Zl_i = h_ik (Gamma-hat^k - Gt^k)/2, R^Z_ij = R_ij + D_i Z_j + D_j Z_i. Written out, the
    // derivatives of Gt^k in R_ij and in D_(i Z_j) cancel, as do the Gt_kij Gt^k and Gt_kij Gamma-hat^k terms:
    //   R^Z_ij = -1/2 h^lm d_l d_m h_ij + U^km_i d_m h_jk + U^km_j Gt_ikm + Gamma-hat^k d_k h_ij/2
    //            + h_k(i d_j) Gamma-hat^k + chi part, U^km_i = h^lm Gt^k_li
    GRF_SECTION(6);
    T dG[3], Zl[3];
    const T Gh[3] = {v[F_GAM], v[F_GAM + 1], v[F_GAM + 2]};
#pragma unroll
    for (int k = 0; k < 3; ++k) dG[k] = Gh[k] - Gtc[k];
    {
        const T hdG[3] = {half_of(dG[0]), half_of(dG[1]), half_of(dG[2])};
#pragma unroll
        for (int i = 0; i < 3; ++i)
            Zl[i] = dot3(h[sidx(i, 0)], hdG[0], h[sidx(i, 1)], hdG[1], h[sidx(i, 2)], hdG[2]);
    }
    T RZ[6], DivZ2, chz;  // R^Z_ij without its chi part Pc_ij + chz h_ij; 2 D_i Z^i
    {
        T dh[3][6];
#pragma unroll
        for (int k = 0; k < 3; ++k)
#pragma unroll
            for (int m = 0; m < 6; ++m) dh[k][m] = DH1(k, m);
        T U[3][3][3];  // U[k][m][i] = h^lm Gt^k_li
#pragma unroll
        for (int k = 0; k < 3; ++k)
#pragma unroll
            for (int m = 0; m < 3; ++m)
#pragma unroll
                for (int i = 0; i < 3; ++i)
                    U[k][m][i] = dot3(hi[sidx(0, m)], G2[k][sidx(0, i)], hi[sidx(1, m)], G2[k][sidx(1, i)],
                                      hi[sidx(2, m)], G2[k][sidx(2, i)]);
        T mhw[6];
#pragma unroll
        for (int q = 0; q < 6; ++q) mhw[q] = half_of(hw[q]);
        const T hGh[3] = {half_of(Gh[0]), half_of(Gh[1]), half_of(Gh[2])};
        const T dGd = dot3(dG[0], dchi[0], dG[1], dchi[1], dG[2], dchi[2]);
        chz = fma(hichi, chiLap - dGd, 3.0 * (qichi2 * dchi2));
        const T dci[3] = {twice_of(c1[0]), twice_of(c1[1]), twice_of(c1[2])};  // d_i chi / chi
        T hdGam[3][3];  // d_j Gamma-hat^k / 2
#pragma unroll
        for (int k = 0; k < 3; ++k)
#pragma unroll
            for (int j = 0; j < 3; ++j) hdGam[k][j] = half_of(D1(F_GAM + k, j));
#pragma unroll
        for (int j = 0; j < 3; ++j) {
            const T us01 = U[0][1][j] + U[1][0][j], us02 = U[0][2][j] + U[2][0][j], us12 = U[1][2][j] + U[2][1][j];
#pragma unroll
            for (int i = 0; i <= j; ++i) {
                const int ij = sidx(i, j);
                T r = fma(dci[i], Zl[j], dci[j] * Zl[i]);
#pragma unroll
                for (int k = 0; k < 3; ++k) {
                    r = fma(hGh[k], dh[k][ij], r);
                    if (i == j) r = fma(h[sidx(i, k)], D1(F_GAM + k, i), r);
                    else r = fma(h[sidx(i, k)], hdGam[k][j], fma(h[sidx(j, k)], hdGam[k][i], r));
                }
                r = fma(U[0][0][j], G1[i][0], fma(us01, G1[i][1], fma(us02, G1[i][2], r)));
                r = fma(U[1][1][j], G1[i][3], fma(us12, G1[i][4], fma(U[2][2][j], G1[i][5], r)));
#pragma unroll
                for (int k = 0; k < 3; ++k)
#pragma unroll
                    for (int m = 0; m < 3; ++m) r = fma(U[k][m][i], dh[m][sidx(j, k)], r);
#pragma unroll
                for (int q = 0; q < 6; ++q) r = fnma(mhw[q], D2(F_H + ij, q), r);
                RZ[ij] = r;
            }
        }
        DivZ2 = fma(-1.5, dGd, sdotw(RZ, gw)) - Rconf;
    }

    // ---- D_i D_j lapse, D_i D_j phi (physical)
    GRF_SECTION(7);
    T DDa[6], DDp[6];
#pragma unroll
    for (int m = 0; m < 6; ++m) {
        DDa[m] = fnma(Gp[0][m], D1(F_LAPSE, 0), fnma(Gp[1][m], D1(F_LAPSE, 1), fnma(Gp[2][m], D1(F_LAPSE, 2), D2(F_LAPSE, m))));
        DDp[m] = fnma(Gp[0][m], dphi[0], fnma(Gp[1][m], dphi[1], fnma(Gp[2][m], dphi[2], D2(F_PHI, m))));
    }
    const T lapal = sdotw(DDa, gw);

    // ---- extrinsic curvature K_ij = Ah_ij/chi, Ah_ij = A_ij + h_ij K/3, and friends
    GRF_SECTION(8);
    const T K3 = K * (1.0 / 3.0);
    T Ah[6], Kp[6], Aud[3][3];
#pragma unroll
    for (int m = 0; m < 6; ++m) {
        Ah[m] = fma(h[m], K3, A[m]);
        Kp[m] = Ah[m] * ichi;
    }
#pragma unroll
    for (int i = 0; i < 3; ++i)
#pragma unroll
        for (int j = 0; j < 3; ++j)
            Aud[i][j] = dot3(hi[sidx(i, 0)], A[sidx(0, j)], hi[sidx(i, 1)], A[sidx(1, j)], hi[sidx(i, 2)], A[sidx(2, j)]);
    // K^i_j = A^i_j + delta^i_j K/3
    const T Kdg[3] = {Aud[0][0] + K3, Aud[1][1] + K3, Aud[2][2] + K3};
    auto Kud = [&](int i, int j) -> T { return i == j ? Kdg[i] : Aud[i][j]; };
    T Au[6], Auw[6], AAud[6];  // A^ij, with off-diagonals doubled, A_ik A^k_j
#pragma unroll
    for (int i = 0; i < 3; ++i)
#pragma unroll
        for (int j = i; j < 3; ++j) {
            const int m = sidx(i, j);
            Au[m] = dot3(Aud[i][0], hi[sidx(0, j)], Aud[i][1], hi[sidx(1, j)], Aud[i][2], hi[sidx(2, j)]);
            Auw[m] = (i == j) ? Au[m] : twice_of(Au[m]);
            AAud[m] = dot3(A[sidx(i, 0)], Aud[0][j], A[sidx(i, 1)], Aud[1][j], A[sidx(i, 2)], Aud[2][j]);
        }
    const T AA = sdotw(A, Auw);
    // ---- the sources' share apart (rho, S_i and C_ij come below): d_t K, d_t A_ij, d_t Theta, d_t Gamma-hat and
    // the right-hand side of C_ij, formed where their inputs are at hand, since values kept for later are
    // spilled. C_ij holds all of (d_t K_ij - L_beta K_ij + D_i D_j alpha)/alpha + K_ik K^k_j, S_ij included:
    //   d_t K = beta.dK - D^2 alpha + alpha (tr C + K_ij K^ij), and d_t A_ij from the trace-free part of
    //   alpha C_ij - D_i D_j alpha. The damping and Theta terms, and a non-zero tr A, are those of C's own
    //   right-hand side (a1: the coefficient of A_ij in it).
    T Cr[6];  // R^Z_ij + (a1 A_ij - A_ik A^k_j)/chi
    {
        const T divb23 = (2.0 / 3.0) * divb, al2 = twice_of(al);
        const T a1 = fma(-2.0 / 3.0, K, K2Th);
        const T trA = Aud[0][0] + Aud[1][1] + Aud[2][2], AAt = fnma(a1, trA, AA);
        rhs[F_K] = fma(al, Rs + DivZ2, ADV(F_K) - lapal);
        // h_ij's coefficient: minus a third of the trace of the K_ij K^ij terms
        const T hc = (-1.0 / 3.0) * (al * AAt);
        const T aA = fma(al, K2Th - a1, -divb23);  // 2/3 (alpha K - div beta)
        T db[3][3];
#pragma unroll
        for (int j = 0; j < 3; ++j)
#pragma unroll
            for (int i = 0; i < 3; ++i) db[j][i] = D1(F_SHIFT + i, j);
#pragma unroll
        for (int i = 0; i < 3; ++i)
#pragma unroll
            for (int j = i; j < 3; ++j) {
                const int m = sidx(i, j);
                // the chi part, large near a puncture, comes last, so that the small terms are not rounded to its
                // last place one by one
                Cr[m] = fma(chz, h[m], fma(ichi, fma(a1, A[m], -AAud[m]), RZ[m]) + Pc[m]);
                T x = fma(h[m], hc, ADV(F_A + m));
                x = fma(aA, A[m], fnma(al, AAud[m], x));
                if (i == j) {
                    x = fma(2.0, dot3(A[sidx(i, 0)], db[i][0], A[sidx(i, 1)], db[i][1], A[sidx(i, 2)], db[i][2]), x);
                } else {
#pragma unroll
                    for (int k = 0; k < 3; ++k) x = fma(A[sidx(i, k)], db[j][k], fma(A[sidx(j, k)], db[i][k], x));
                }
                rhs[F_A + m] = x;
            }
        // d_t Theta = beta.dTheta + alpha (D_i Z^i - Theta K) - Z^i d_i alpha + alpha Hb / (2 (1 + b)),
        // with Z^i = chi (Gamma-hat^i - Gt^i)/2; Hb is added below
        const T dal[3] = {D1(F_LAPSE, 0), D1(F_LAPSE, 1), D1(F_LAPSE, 2)};
        const T Zda = half_of(chi) * dot3(dG[0], dal[0], dG[1], dal[1], dG[2], dal[2]);
        rhs[F_TH] = fma(al, fnma(Th, K, half_of(DivZ2)), ADV(F_TH) - Zda);
        // d_t Gamma-hat^i with everything contracted with h^ij in one covector V_j, with A^ij in va_j and
        // with d_k beta^i in Gk: h^ij Z_j = (Gamma-hat^i - Gt^i)/2. The b(x) part of d_t Z_j is
        // -(b/(1+b)) alpha wb_j, wb_j = M_j + d_j Theta - K^k_j Z_k - kappa1 Z_j with the momentum constraint
        // M_j = B_j - 8 pi S_j (added below); Gamma-hat^i carries 2 h^ij Z_j, so d_t Gamma-hat^i gains
        // -(2b/(1+b)) alpha h^ij wb_j (2b/(1+b) = 2 - 4 bTh)
        const T abG = (2.0 - 4.0 * c.bTh) * al;
        const T m3 = -3.0 * (al * ichi), alK43 = (4.0 / 3.0) * (al * K), al43 = (4.0 / 3.0) * al, Th2 = twice_of(Th);
        const T cTh = al2 - abG, cZ = fma(abG, c.kappa1, -alK43);
        T va[3], V[3], Gk[3];
#pragma unroll
        for (int j = 0; j < 3; ++j) {
            va[j] = fma(m3, dchi[j], -2.0 * dal[j]);
            Gk[j] = fma(c.kappa3, dG[j], Gtc[j]);
            const T ddbk = D2(F_SHIFT, sidx(j, 0)) + D2(F_SHIFT + 1, sidx(j, 1)) + D2(F_SHIFT + 2, sidx(j, 2));
            const T kz = dot3(Kud(0, j), Zl[0], Kud(1, j), Zl[1], Kud(2, j), Zl[2]);
            T x = fma(1.0 / 3.0, ddbk, fma(cTh, D1(F_TH, j), cZ * Zl[j]));
            x = fnma(Th2, dal[j], fnma(al43, D1(F_K, j), x));
            V[j] = fma(abG, kz, x);
        }
        const T kz2 = fma((2.0 / 3.0) * c.kappa3, divb, -(c.kappa1 * al));
#pragma unroll
        for (int i = 0; i < 3; ++i) {
            T x = fma(al2, sdotw(G2[i], Auw), ADV(F_GAM + i));
            x = fma(kz2, dG[i], fma(divb23, Gtc[i], x));
#pragma unroll
            for (int k = 0; k < 3; ++k) {
                x = fma(Au[sidx(i, k)], va[k], x);
                x = fma(hi[sidx(i, k)], V[k], x);
                x = fnma(Gk[k], db[k][i], x);
            }
#pragma unroll
            for (int q = 0; q < 6; ++q) x = fma(hw[q], D2(F_SHIFT + i, q), x);
            rhs[F_GAM + i] = x;
        }
    }
    // Codazzi block through its dual: bb[k][m] = B_{k,(m+1),(m+2)} = D_a K_kb - D_b K_ka with
    // (a, b) = (m+1, m+2). The connection's symmetric part cancels between the two covariant
    // derivatives, and with K_ij = (A_ij + h_ij K/3)/chi (D~_a h_kb = 0) so do the derivatives of h:
    //   chi B_kab = d_a A_kb - d_b A_ka - Gt^l_ak A_lb + Gt^l_bk A_la + h_kb e_a - h_ka e_b - q_a A_kb + q_b A_ka,
    //   q_a = d_a chi/(2 chi), e_a = d_a K/3 + h^lm q_m A_la;
    // the q terms are carried by the l = k Christoffels.
    T bb[3][3], Bv[3];  // Bv_j = B_j = gamma^ab B_abj
#define BC(k, i, j) (cyclic(i, j) ? bb[k][third(i, j)] : -bb[k][third(i, j)])
#define BCFMA(B, k, i, j, x, s) (cyclic(i, j) ? fma(B[k][third(i, j)], x, s) : fnma(B[k][third(i, j)], x, s))
    {
        T ev[3], Gk[3][3], bx3[3][3];
#pragma unroll
        for (int a = 0; a < 3; ++a) {
            ev[a] = fma(c2[0], A[sidx(0, a)], fma(c2[1], A[sidx(1, a)], fma(c2[2], A[sidx(2, a)], D1(F_K, a) * (1.0 / 3.0))));
#pragma unroll
            for (int k = 0; k < 3; ++k) Gk[k][a] = G2[k][sidx(a, k)] + c1[a];
        }
#pragma unroll
        for (int k = 0; k < 3; ++k)
#pragma unroll
            for (int m = 0; m < 3; ++m) {
                const int a = (m + 1) % 3, b = (m + 2) % 3;
                T s = D1(F_A + sidx(k, b), a) - D1(F_A + sidx(k, a), b);
                s = fma(h[sidx(k, b)], ev[a], fnma(h[sidx(k, a)], ev[b], s));
#pragma unroll
                for (int l = 0; l < 3; ++l)
                    s = fnma(l == k ? Gk[k][a] : G2[l][sidx(a, k)], A[sidx(l, b)],
                             fma(l == k ? Gk[k][b] : G2[l][sidx(b, k)], A[sidx(l, a)], s));
                bx3[k][m] = s;
                bb[k][m] = s * ichi;
            }
#pragma unroll
        for (int j = 0; j < 3; ++j) {
            const int p = (j + 1) % 3, q = (j + 2) % 3;
            T s = fnma(hi[sidx(j, p)], bx3[j][q], hi[sidx(j, q)] * bx3[j][p]);
            s = fma(hi[sidx(q, q)], bx3[q][p], fnma(hi[sidx(p, p)], bx3[p][q], s));
            s = fma(hi[sidx(p, q)], bx3[p][p], fnma(hi[sidx(p, q)], bx3[q][q], s));
            Bv[j] = s;
        }
    }

    // ---- Gauss block S_iklm = Riem_iklm + K_il K_km - K_im K_kl: its contraction S_ij and the double
    // dual G_S^ij (the raised Einstein tensor), both from the six components
    GRF_SECTION(9);
    Rm[0] = fma(Kp[0], Ah[3], fnma(Kp[1], Ah[1], Rm[0]));
    Rm[1] = fma(Kp[0], Ah[4], fnma(Kp[2], Ah[1], Rm[1]));
    Rm[2] = fma(Kp[1], Ah[4], fnma(Kp[2], Ah[3], Rm[2]));
    Rm[3] = fma(Kp[0], Ah[5], fnma(Kp[2], Ah[2], Rm[3]));
    Rm[4] = fma(Kp[1], Ah[5], fnma(Kp[2], Ah[4], Rm[4]));
    Rm[5] = fma(Kp[3], Ah[5], fnma(Kp[4], Ah[4], Rm[5]));
    T S[6], GSuw[6];
    S[0] = dot3(hi[3], Rm[0], hw[4], Rm[1], hi[5], Rm[3]);
    S[3] = fma(hi[0], Rm[0], fnma(hw[2], Rm[2], hi[5] * Rm[5]));
    S[5] = dot3(hi[0], Rm[3], hw[1], Rm[4], hi[3], Rm[5]);
    S[1] = fnma(hi[1], Rm[0], fnma(hi[2], Rm[1], fma(hi[4], Rm[2], hi[5] * Rm[4])));
    S[2] = fnma(hi[1], Rm[1], fnma(hi[3], Rm[2], fnma(hi[2], Rm[3], fnma(hi[4], Rm[4], T(0.0)))));
    S[4] = fnma(hi[2], Rm[4], fnma(hi[4], Rm[5], fma(hi[0], Rm[1], hi[1] * Rm[2])));
    const T Ss = sdotw(S, gw);
    T GS[6];
    const T hSs = half_of(Ss);
#pragma unroll
    for (int m = 0; m < 6; ++m) GS[m] = fnma(hSs, gd[m], S[m]);
    {
        const T cd = chi * chidet, cd2 = twice_of(cd);  // off-diagonals doubled
        GSuw[0] = fnma(cd, Rm[5], T(0.0));
        GSuw[3] = fnma(cd, Rm[3], T(0.0));
        GSuw[5] = fnma(cd, Rm[0], T(0.0));
        GSuw[1] = cd2 * Rm[4];
        GSuw[2] = fnma(cd2, Rm[2], T(0.0));
        GSuw[4] = cd2 * Rm[1];
    }

    // ---- scalar: nabla nabla phi blocks, Phi = nabla nabla beta(phi)
    GRF_SECTION(10);
    T b1, b2;
    // beta' and beta'' of the coupling: lam phi, lam phi^2 / 2, or lam / (2 kappa) (1 - e^{-kappa phi^2})
    // (beta' = lam phi e^{-kappa phi^2}, beta'' = lam e^{-kappa phi^2} (1 - 2 kappa phi^2))
    if (c.beta_kind == 1) {
        b1 = c.lam * phi; b2 = c.lam;
    } else if (COUP && c.beta_kind == 2) {
        const T kp2 = c.beta_kappa * (phi * phi);
        const T e = exp(-kp2);
        b1 = c.lam * (phi * e);
        b2 = c.lam * (e * fma(-2.0, kp2, 1.0));
    } else {
        b1 = c.lam; b2 = 0.0;
    }
    T dphiu[3];
#pragma unroll
    for (int i = 0; i < 3; ++i)
        dphiu[i] = dot3(gu[sidx(i, 0)], dphi[0], gu[sidx(i, 1)], dphi[1], gu[sidx(i, 2)], dphi[2]);
    const T dphi2 = dot3(dphi[0], dphiu[0], dphi[1], dphiu[1], dphi[2], dphiu[2]);
    const T Pi2 = Pi * Pi;
    const T X = half_of(Pi2 - dphi2);
    const T g2 = c.g2;
    T Hij[6], Hn[3];
#pragma unroll
    for (int m = 0; m < 6; ++m) Hij[m] = fma(Kp[m], Pi, DDp[m]);
#pragma unroll
    for (int i = 0; i < 3; ++i)
        Hn[i] = fma(Kud(0, i), dphi[0], fma(Kud(1, i), dphi[1], fma(Kud(2, i), dphi[2], D1(F_PI, i))));
    T Phd[6], Phn[3];
    const T b2Pi = b2 * Pi;
#pragma unroll
    for (int i = 0; i < 3; ++i) {
        Phn[i] = fma(b1, Hn[i], b2Pi * dphi[i]);
        const T b2d = b2 * dphi[i];
#pragma unroll
        for (int j = i; j < 3; ++j) Phd[sidx(i, j)] = fma(b1, Hij[sidx(i, j)], b2d * dphi[j]);
    }
    T Phm[3][3], Phuw[6], Phnu[3];  // Phi_i^k, Phi^ij (off-diagonals doubled), Phi_n^k
#pragma unroll
    for (int i = 0; i < 3; ++i)
#pragma unroll
        for (int k = 0; k < 3; ++k)
            Phm[i][k] = dot3(Phd[sidx(i, 0)], gu[sidx(0, k)], Phd[sidx(i, 1)], gu[sidx(1, k)], Phd[sidx(i, 2)], gu[sidx(2, k)]);
#pragma unroll
    for (int i = 0; i < 3; ++i) {
#pragma unroll
        for (int j = i; j < 3; ++j) {
            const T x = dot3(gu[sidx(i, 0)], Phm[0][j], gu[sidx(i, 1)], Phm[1][j], gu[sidx(i, 2)], Phm[2][j]);
            Phuw[sidx(i, j)] = (i == j) ? x : twice_of(x);
        }
        Phnu[i] = dot3(gu[sidx(i, 0)], Phn[0], gu[sidx(i, 1)], Phn[1], gu[sidx(i, 2)], Phn[2]);
    }
    const T trP = Phm[0][0] + Phm[1][1] + Phm[2][2];

    // ---- sources that do not depend on the unknowns
    GRF_SECTION(11);
    const T fX = fma(2.0 * g2, X, 1.0);
    const T XX = fma(g2 * X, X, X);  // X + g2 X^2
    // decoupled mode: the scalar's stress-energy is left out of the metric equations (rho, S_i,
    // S_ij and their coupling to d_t K_ij); the scalar equation below is unchanged
    const bool dec = (DEC < 0) ? (c.decoupled != 0) : (DEC == 1);
    const T fXh = half_of(fX), XXh = half_of(XX);
    T rho8 = dec ? T(0.0) : fma(fXh, Pi2, fma(-4.0, sdotw(GS, Phuw), -XXh));
    T S8[3];
    const T BPn = dot3(Bv[0], Phnu[0], Bv[1], Phnu[1], Bv[2], Phnu[2]);
    T Phuh[6];  // Phi^ij
#pragma unroll
    for (int m = 0; m < 6; ++m) Phuh[m] = (m == 1 || m == 2 || m == 4) ? half_of(Phuw[m]) : Phuw[m];
#pragma unroll
    for (int i = 0; i < 3; ++i) {
        T s = dot3(GS[sidx(i, 0)], Phnu[0], GS[sidx(i, 1)], Phnu[1], GS[sidx(i, 2)], Phnu[2]);
        s = fma(trP, Bv[i], fnma(Phm[i][0], Bv[0], fnma(Phm[i][1], Bv[1], fnma(Phm[i][2], Bv[2], s))));
#pragma unroll
        for (int k = 0; k < 3; ++k)
#pragma unroll
            for (int l = 0; l < 3; ++l)
                if (l != i) s = BCFMA(bb, k, i, l, Phuh[sidx(k, l)], s);
        S8[i] = dec ? T(0.0) : fnma(fXh * Pi, dphi[i], 4.0 * s);
    }
    // cubic term: the n-n and n-i parts of its stress tensor (no unknown in them)
    const bool cub = COUP && c.g3 != 0.0;
    T trH3 = 0.0, Hnd3 = 0.0, Hdd3 = 0.0, Hdv3[3];
    if (cub) {
        trH3 = sdotw(Hij, gw);
        Hnd3 = dot3(dphiu[0], Hn[0], dphiu[1], Hn[1], dphiu[2], Hn[2]);
#pragma unroll
        for (int i = 0; i < 3; ++i)
            Hdv3[i] = dot3(Hij[sidx(i, 0)], dphiu[0], Hij[sidx(i, 1)], dphiu[1], Hij[sidx(i, 2)], dphiu[2]);
        Hdd3 = dot3(dphiu[0], Hdv3[0], dphiu[1], Hdv3[1], dphiu[2], Hdv3[2]);
        if (!dec) {
            const double g3h = 0.5 * c.g3;
            rho8 = fma(g3h, fma(Pi2, trH3, -Hdd3), rho8);
            const T a3 = fma(Pi, trH3, -Hnd3);
#pragma unroll
            for (int i = 0; i < 3; ++i) S8[i] = fma(-g3h, fma(a3, dphi[i], Pi * fma(Pi, Hn[i], -Hdv3[i])), S8[i]);
        }
    }
    // LS_ij = L(8 pi S_ij) without its C and N parts, L(X) = X - gamma tr(X)/2, from the X terms
    // fX d_i phi d_j phi/2 + XX gamma_ij/2 and -4 Y_ij; the traces are known (gamma^ij B_ijl = B_l, so
    // tr Y = -2 B_l Phi_n^l):
    //   L(Y)_ij = B_i Phi_nj + B_j Phi_ni + B_ijl Phi_n^l + B_jil Phi_n^l - gamma_ij B_l Phi_n^l
    T LS[6], trS = 0.0;  // trS: minus the trace of LS
    if (dec) {
#pragma unroll
        for (int m = 0; m < 6; ++m) LS[m] = T(0.0);
    } else {
        const T tg = half_of(fma(fXh, dphi2, XXh));
        trS = fma(4.0, BPn, fma(3.0, tg, -(fXh * dphi2)));
#pragma unroll
        for (int i = 0; i < 3; ++i) {
            const T fd = fXh * dphi[i];
#pragma unroll
            for (int j = i; j < 3; ++j) {
                T y = fma(Bv[j], Phn[i], fnma(BPn, gd[sidx(i, j)], Bv[i] * Phn[j]));
#pragma unroll
                for (int l = 0; l < 3; ++l) {
                    if (l != j) y = BCFMA(bb, i, j, l, Phnu[l], y);
                    if (l != i) y = BCFMA(bb, j, i, l, Phnu[l], y);
                }
                LS[sidx(i, j)] = fma(-4.0, y, fnma(tg, gd[sidx(i, j)], fd * dphi[j]));
            }
        }
    }

    GRF_SECTION(12);
    const T bdPi = LOP ? adv[F_PI] : dot3(at_use(v[F_SHIFT]), D1(F_PI, 0), at_use(v[F_SHIFT + 1]), D1(F_PI, 1), at_use(v[F_SHIFT + 2]), D1(F_PI, 2));
    const T dadp = dot3(D1(F_LAPSE, 0), dphiu[0], D1(F_LAPSE, 1), dphiu[1], D1(F_LAPSE, 2), dphiu[2]);

    // L_GB without its 8 G_S^ij C_ij: -4 B_kij B^kij + 8 B_i B^i, with
    // B_kij B^kij = 2 chi^3 / det(h) h^kk' h_mm' bb[k][m] bb[k'][m']
    GRF_SECTION(13);
    T L0;
    {
        T N[3][3];
#pragma unroll
        for (int k = 0; k < 3; ++k)
#pragma unroll
            for (int q = 0; q < 3; ++q)
                N[k][q] = dot3(h[sidx(0, q)], bb[k][0], h[sidx(1, q)], bb[k][1], h[sidx(2, q)], bb[k][2]);
        T tt[6];
#pragma unroll
        for (int k = 0; k < 3; ++k)
#pragma unroll
            for (int kk = k; kk < 3; ++kk)
                tt[sidx(k, kk)] = dot3(N[k][0], bb[kk][0], N[k][1], bb[kk][1], N[k][2], bb[kk][2]);
        const T BB = (chi * (chi * chidet)) * sdotw(tt, hw);  // half of B_kij B^kij
        const T Bvu0 = dot3(gu[0], Bv[0], gu[1], Bv[1], gu[2], Bv[2]);
        const T Bvu1 = dot3(gu[1], Bv[0], gu[3], Bv[1], gu[4], Bv[2]);
        const T Bvu2 = dot3(gu[2], Bv[0], gu[4], Bv[1], gu[5], Bv[2]);
        const T BvBv = dot3(Bv[0], Bvu0, Bv[1], Bvu1, Bv[2], Bvu2);
        L0 = 8.0 * (BvBv - BB);
    }

    // ---- rho and S_i in d_t Theta and d_t Gamma-hat
    GRF_SECTION(14);
    // b(x) of the modified gauge enters through the auxiliary metric g^ab - b n^a n^b of the Z terms
    // of the covariant equation; its 3+1 projection is carried by Hb = H - 16 pi rho
    // - 2 kappa1 (2 + kappa2) Theta (plain H = R - A_ij A^ij + 2/3 K^2) in d_t K and d_t Theta, and
    // by the momentum-constraint combination in d_t Gamma-hat.
    const T Hb = fma(-2.0 * c.kappa1 * (2.0 + c.kappa2), Th, fma(-2.0, rho8, fma((2.0 / 3.0) * K, K, Rs - AA)));
    // (d_t K without advection, the lapse's Laplacian, alpha R^Z and S_ij) / alpha
    const T kS = fma(K, K2Th, fma(-3.0 * c.kappa1 * (1.0 + c.kappa2), Th, fma(-1.5, rho8, -c.bK * Hb)));
    rhs[F_TH] = fma(c.bTh * al, Hb, rhs[F_TH]);
    rhs[F_K] = fma(al, kS, rhs[F_K]);
    {
        const T abG = (2.0 - 4.0 * c.bTh) * al, cTh = twice_of(al) - abG;
        T V[3];
#pragma unroll
        for (int j = 0; j < 3; ++j) V[j] = fma(cTh, S8[j], abG * Bv[j]);
#pragma unroll
        for (int i = 0; i < 3; ++i) {
            T x = fnma(hi[sidx(i, 0)], V[0], fnma(hi[sidx(i, 1)], V[1], fnma(hi[sidx(i, 2)], V[2], rhs[F_GAM + i])));
            rhs[F_GAM + i] = x;
            rhs[F_B + i] = fma(-c.eta, v[F_B + i], x);
        }
    }

    // ---- coupled system, in the curvature components that hold the unknowns: C_ij = R_ninj (d_t K_ij) and
    // N = H_nn = (d_t Pi - beta^k d_k Pi - d^k alpha d_k phi)/alpha (d_t Pi):
    //   C - 4 L(Q(C)) - 4 b1 L(G_S) N = r,   N - (8 b1 / D) G_S^ij C_ij = r_N,   L(X) = X - gamma tr(X)/2.
    // Without S_ij, C = R^Z + (K - 2 Theta) K_ij - K_ik K^k_j + a trace: the lapse's derivatives and every
    // shift term of d_t K_ij cancel in it.
    GRF_SECTION(15);
    T Msys[7][8];
    T rs[7];   // the right-hand side r, r_N
    T PPc[6];  // cubic term: Pi^2 gamma^ij - d^i phi d^j phi
    {
        const T a0 = ((1.0 / 3.0) * ichi) * fma((-1.0 / 3.0) * K, K, kS);
        const T Ss4 = 0.25 * Ss;
        const T four_b1 = 4.0 * b1, b2Pi2x4 = 4.0 * (b2Pi * Pi);
#pragma unroll
        for (int m = 0; m < 6; ++m) {
            T r = a0 * h[m];
            T w6 = T(0.0);
            if (!dec) {
                const T LGS = fnma(Ss4, gd[m], S[m]);
                r = fma(b2Pi2x4, LGS, r - LS[m]);
                w6 = fnma(four_b1, LGS, T(0.0));
            }
            rs[m] = Cr[m] + r;
            Msys[m][6] = w6;
        }
        if (!dec) trS = fma(b2Pi2x4, Ss4, trS);  // tr L(G_S) = S/4
        // 6x6 block, column (a,b): -4 L(Q(E_ab)) with E_ab the unit symmetric matrix and
        //   Q_ij(X) = gamma_ij (X.Phi) - Phi_i^k X_kj - Phi_j^k X_ik + tr(Phi) X_ij - tr(X)(gamma_ij tr(Phi) - Phi_ij)
        //   = -2 gamma_ij w_ab (Phi^ab - gamma^ab tr Phi) - 4 w_ab gamma^ab Phi_ij + 4 P_ij,ab - 4 tr(Phi) [ij == ab]
        //   P_ij,ab = Phi_i^k E_kj + Phi_j^k E_ik
        const T trP4 = -4.0 * trP;
        T gd2[6], Ph4[3][3];
#pragma unroll
        for (int m = 0; m < 6; ++m) gd2[m] = twice_of(gd[m]);
#pragma unroll
        for (int i = 0; i < 3; ++i)
#pragma unroll
            for (int k = 0; k < 3; ++k) Ph4[i][k] = twice_of(twice_of(Phm[i][k]));
#pragma unroll
        for (int a = 0; a < 3; ++a)
#pragma unroll
            for (int b = a; b < 3; ++b) {
                const int col = sidx(a, b);
                const T sab = fnma(gw[col], trP, Phuw[col]);    // w_ab (Phi^ab - gamma^ab trP)
                const T tab = twice_of(twice_of(gw[col]));      // 4 w_ab gamma^ab
#pragma unroll
                for (int i = 0; i < 3; ++i)
#pragma unroll
                    for (int j = i; j < 3; ++j) {
                        const int row = sidx(i, j);
                        T p = 0.0;
                        bool any = false;
                        // 4 Phi_i^k E_kj: E_kj = [k==a][j==b] + [k==b][j==a] (single term when a == b)
                        if (j == b && i == j) { p = twice_of(Ph4[i][a]); any = true; }
                        else {
                            if (j == b) { p = Ph4[i][a]; any = true; }
                            if (i == b) { p = any ? p + Ph4[j][a] : Ph4[j][a]; any = true; }
                        }
                        if (a != b && j == a && i == j) { p = any ? p + twice_of(Ph4[i][b]) : twice_of(Ph4[i][b]); any = true; }
                        else if (a != b) {
                            if (j == a) { p = any ? p + Ph4[i][b] : Ph4[i][b]; any = true; }
                            if (i == a) { p = any ? p + Ph4[j][b] : Ph4[j][b]; any = true; }
                        }
                        if (row == col) { p = any ? p + trP4 : trP4; any = true; }
                        T e = any ? fnma(tab, Phd[row], p) : fnma(tab, Phd[row], T(0.0));
                        e = fnma(gd2[row], sab, e);
                        Msys[row][col] = dec ? T(0.0) : e;  // M - 1
                    }
            }
        T Dphi = fma(2.0 * g2, Pi2, fX);
        T E3 = 0.0;  // the cubic term's share of the scalar equation without N and C
        if (cub) {
            Dphi = fma(2.0 * c.g3, trH3, Dphi);
            T Hm[3][3], ppw[6], PPuw[6];  // H_i^k, d^i phi d^j phi and Pi^2 gamma^ij - d^i phi d^j phi (weighted)
#pragma unroll
            for (int i = 0; i < 3; ++i)
#pragma unroll
                for (int k = 0; k < 3; ++k)
                    Hm[i][k] = dot3(Hij[sidx(i, 0)], gu[sidx(0, k)], Hij[sidx(i, 1)], gu[sidx(1, k)], Hij[sidx(i, 2)], gu[sidx(2, k)]);
            T HH = 0.0;
#pragma unroll
            for (int i = 0; i < 3; ++i)
#pragma unroll
                for (int k = 0; k < 3; ++k) HH = fma(Hm[i][k], Hm[k][i], HH);
            T HnHn = 0.0, BdP = 0.0;
#pragma unroll
            for (int i = 0; i < 3; ++i) {
                const T hnu = dot3(gu[sidx(i, 0)], Hn[0], gu[sidx(i, 1)], Hn[1], gu[sidx(i, 2)], Hn[2]);
                HnHn = fma(Hn[i], hnu, HnHn);
                BdP = fma(Bv[i], dphiu[i], BdP);
            }
#pragma unroll
            for (int i = 0; i < 3; ++i)
#pragma unroll
                for (int j = i; j < 3; ++j) {
                    const T pp = dphiu[i] * dphiu[j];
                    ppw[sidx(i, j)] = (i == j) ? pp : twice_of(pp);
                    PPuw[sidx(i, j)] = fma(Pi2, gw[sidx(i, j)], -ppw[sidx(i, j)]);
                }
            T e3 = fma(trH3, trH3, fma(2.0, HnHn, -HH));
            e3 = fma(-2.0 * Pi, BdP, e3);
            e3 = e3 - sdotw(S, ppw);
            E3 = c.g3 * e3;
            if (!dec) {
                // 8 pi S3_ij without its N part, and that part's coefficient in the metric rows:
                // S3_ij = S3_0 + g3 N / 2 (Pi^2 gamma_ij - d_i phi d_j phi)
                T S3[6];
                const T pcoef = half_of(trH3);                        // of d_i phi d_j phi
                const T gcoef = fma(0.5, Hdd3, -(Pi * Hnd3));         // of gamma_ij
#pragma unroll
                for (int i = 0; i < 3; ++i)
#pragma unroll
                    for (int j = i; j < 3; ++j) {
                        T x = fma(gcoef, gd[sidx(i, j)], pcoef * (dphi[i] * dphi[j]));
                        x = fma(half_of(Pi), fma(Hn[i], dphi[j], Hn[j] * dphi[i]), x);
                        x = fma(-0.5, fma(Hdv3[i], dphi[j], Hdv3[j] * dphi[i]), x);
                        S3[sidx(i, j)] = c.g3 * x;
                    }
                const T trS3h = half_of(sdotw(S3, gw));
                const T wc = half_of(dphi2 - Pi2);
                trS = trS + trS3h;
#pragma unroll
                for (int m = 0; m < 6; ++m) {
                    const int i = (m < 3) ? 0 : (m < 5 ? 1 : 2);
                    const int j = (m < 3) ? m : (m < 5 ? m - 2 : 2);
                    rs[m] = rs[m] - fnma(trS3h, gd[m], S3[m]);
                    Msys[m][6] = fma(0.5 * c.g3, fma(wc, gd[m], -(dphi[i] * dphi[j])), Msys[m][6]);
                }
            }
#pragma unroll
            for (int col = 0; col < 6; ++col) PPc[col] = PPuw[col];
        }
        const T iD = recip(Dphi);
        const T c8 = -8.0 * (b1 * iD);
#pragma unroll
        for (int col = 0; col < 6; ++col) Msys[6][col] = c8 * GSuw[col];
        if (cub) {
#pragma unroll
            for (int col = 0; col < 6; ++col) Msys[6][col] = fma(c.g3 * iD, PPc[col], Msys[6][col]);
        }
        const T trH = sdotw(Hij, gw);
        const T Hnd = dot3(dphiu[0], Hn[0], dphiu[1], Hn[1], dphiu[2], Hn[2]);
        T Hdd = 0.0;
#pragma unroll
        for (int i = 0; i < 3; ++i) {
            const T t = dot3(Hij[sidx(i, 0)], dphiu[0], Hij[sidx(i, 1)], dphiu[1], Hij[sidx(i, 2)], dphiu[2]);
            Hdd = (i == 0) ? dphiu[0] * t : fma(dphiu[i], t, Hdd);
        }
        T src = fma(fX, trH, fma(4.0 * (g2 * Pi), Hnd, fma(-2.0 * g2, Hdd, b1 * L0)));
        if (cub) src = src + E3;
        rs[6] = iD * src;
        // The unknowns are C - r and N - r_N, M (v - r) = -(M - 1) r: the elimination's rounding then enters the
        // solution in proportion to the coupling, and without coupling v is r to the last bit.
        if (dec) {
#pragma unroll
            for (int i = 0; i < 6; ++i) Msys[i][7] = T(0.0);
        } else {
#pragma unroll
            for (int i = 0; i < 6; ++i) {
                T x = fnma(Msys[i][6], rs[6], T(0.0));
#pragma unroll
                for (int j = 0; j < 6; ++j) x = fnma(Msys[i][j], rs[j], x);
                Msys[i][7] = x;
            }
        }
        {
            T x = fnma(Msys[6][0], rs[0], T(0.0));
#pragma unroll
            for (int j = 1; j < 6; ++j) x = fnma(Msys[6][j], rs[j], x);
            Msys[6][7] = x;
        }
#pragma unroll
        for (int i = 0; i < 6; ++i) Msys[i][i] = Msys[i][i] + 1.0;
        Msys[6][6] = 1.0;
        if constexpr (std::is_same<T, double>::value) {
            if (extra && extra->want_hyp) {
                extra->hyp[0] = det7(Msys, &extra->hyp[3]);
                extra->hyp[1] = fX * fX * fX * fma(6.0 * g2, X, 1.0);  // g3 = 0; the cubic case below
                extra->hyp[2] = Dphi;
            }
        }
    }
    GRF_SECTION(16);
    ok = solve7(Msys);
    T C[6], dC[6];
#pragma unroll
    for (int m = 0; m < 6; ++m) {
        dC[m] = Msys[m][7];
        C[m] = rs[m] + dC[m];
    }
    const T Hnn = rs[6] + Msys[6][7];
    if constexpr (std::is_same<T, double>::value) {
        if (cub && extra && extra->want_hyp) {
            // g_eff in the basis (n, e_i) at the solution: g_eff^nn = -D (stored above),
            // g_eff^ni = 2 g2 Pi d^i phi + 2 g3 H_n^i, g_eff^ij = (1 + 2 g2 X) gamma^ij
            // - 2 g2 d^i phi d^j phi + 2 g3 (box(phi) gamma^ij - H^ij); by the Schur complement on the
            // n-n entry, det g_eff / det g = D det(g_eff^ij + g_eff^ni g_eff^nj / D) det(gamma_ij)
            const double D = extra->hyp[2];
            const double box = trH3 - Hnn;
            double e0[3], Hu[3][3], Sc[6];
            for (int i = 0; i < 3; ++i) {
                const double hnu = gu[sidx(i, 0)] * Hn[0] + gu[sidx(i, 1)] * Hn[1] + gu[sidx(i, 2)] * Hn[2];
                e0[i] = 2.0 * (g2 * Pi * dphiu[i] + c.g3 * hnu);
                for (int k = 0; k < 3; ++k)
                    Hu[i][k] = Hij[sidx(i, 0)] * gu[sidx(0, k)] + Hij[sidx(i, 1)] * gu[sidx(1, k)] + Hij[sidx(i, 2)] * gu[sidx(2, k)];
            }
            for (int i = 0; i < 3; ++i)
                for (int j = i; j < 3; ++j) {
                    const double huij = gu[sidx(i, 0)] * Hu[0][j] + gu[sidx(i, 1)] * Hu[1][j] + gu[sidx(i, 2)] * Hu[2][j];
                    const double eij = fX * gu[sidx(i, j)] - 2.0 * g2 * dphiu[i] * dphiu[j]
                                       + 2.0 * c.g3 * (box * gu[sidx(i, j)] - huij);
                    Sc[sidx(i, j)] = eij + e0[i] * e0[j] / D;
                }
            extra->hyp[1] = D * sym3_det(Sc) * sym3_det(gd);
        }
    }

    // ---- the final K, A_ij, Pi right-hand sides
    GRF_SECTION(17);
    {
        rhs[F_K] = fma(al, trS + sdotw(dC, gw), rhs[F_K]);
        T Y[6];
#pragma unroll
        for (int m = 0; m < 6; ++m) Y[m] = fma(al, rs[m], fma(al, dC[m], -DDa[m]));
        const T trY3 = (1.0 / 3.0) * sdotw(Y, hw);
#pragma unroll
        for (int m = 0; m < 6; ++m) rhs[F_A + m] = fma(chi, fnma(h[m], trY3, Y[m]), rhs[F_A + m]);
        rhs[F_PI] = fma(al, Hnn, bdPi + dadp);
    }
    if (extra) {
        extra->ham = fma(-2.0, rho8, Ss);
#pragma unroll
        for (int i = 0; i < 3; ++i) extra->mom[i] = Bv[i] - S8[i];
        const T X2 = X * X;
        extra->rho8[0] = 0.5 * (Pi * Pi - X);
        extra->rho8[1] = g2 * fma(X, Pi * Pi, -0.5 * X2);
        extra->rho8[2] = -4.0 * sdotw(GS, Phuw);
        if constexpr (std::is_same<T, double>::value) {
            if (extra->want_psi4) {
                // Psi_4 = R(n, mbar, n, mbar) with n = (u - e_r)/sqrt2, m = (e_theta + i e_phi)/sqrt2: the
                // Ricci and scalar terms of the Weyl tensor vanish on a null tetrad with g(n, mbar) = 0,
                // so with the Riemann blocks (Ricci equation, Codazzi, Gauss)
                //   Psi_4 = 1/2 R_ninj mbar^i mbar^j - R_nikj mbar^i e_r^k mbar^j + 1/2 R_kilj e_r^k mbar^i e_r^l mbar^j,
                //   R_ninj = (d_t K_ij - L_beta K_ij + D_i D_j alpha)/alpha + K_ik K^k_j,
                //   R_nikj = D_k K_ij - D_j K_ik,  R_kilj = S_kilj (the Gauss block).
                const double x = extra->xyz[0], y = extra->xyz[1], z = extra->xyz[2];
                double pr = 0.0, pim = 0.0;
                if (x * x + y * y != 0.0) {
                    double e[3][3] = {{x, y, z}, {x * z, y * z, -(x * x + y * y)}, {-y, x, 0.0}};
                    auto dotg = [&](const double* a, const double* b) {
                        double d = 0.0;
#pragma unroll
                        for (int i = 0; i < 3; ++i)
#pragma unroll
                            for (int j = 0; j < 3; ++j) d = fma(gd[sidx(i, j)] * a[i], b[j], d);
                        return d;
                    };
#pragma unroll
                    for (int a = 0; a < 3; ++a) {
#pragma unroll
                        for (int b = 0; b < a; ++b) {
                            const double d = dotg(e[a], e[b]);
#pragma unroll
                            for (int i = 0; i < 3; ++i) e[a][i] -= d * e[b][i];
                        }
                        const double inv = 1.0 / sqrt(dotg(e[a], e[a]));
#pragma unroll
                        for (int i = 0; i < 3; ++i) e[a][i] *= inv;
                    }
                    // symmetric forms on (e_theta, e_phi) give Q(mbar, mbar) = (Q_tt - Q_pp - 2i Q_tp)/2
                    auto form = [&](const double* S6, const double* a, const double* b) {
                        double q = 0.0;
#pragma unroll
                        for (int i = 0; i < 3; ++i)
#pragma unroll
                            for (int j = 0; j < 3; ++j) q = fma(S6[sidx(i, j)] * a[i], b[j], q);
                        return q;
                    };
                    const double E1r = 0.5 * (form(C, e[1], e[1]) - form(C, e[2], e[2]));
                    const double E1i = -form(C, e[1], e[2]);
                    // S_kilj e_r^k e_r^l on (e_theta, e_phi) is S_ij there up to a multiple of the metric
                    const double E3r = 0.5 * (form(S, e[1], e[1]) - form(S, e[2], e[2]));
                    const double E3i = -form(S, e[1], e[2]);
                    // E2 = sum_i mbar^i W_i, W_i = sum_{k != j} R_nikj e_r^k mbar^j, mbar = (e_t - i e_p)/sqrt2
                    double E2r = 0.0, E2i = 0.0;
#pragma unroll
                    for (int i = 0; i < 3; ++i) {
                        double wr = 0.0, wi = 0.0;
#pragma unroll
                        for (int k = 0; k < 3; ++k)
#pragma unroll
                            for (int j = 0; j < 3; ++j)
                                if (k != j) {
                                    const double Rnikj = BC(i, k, j);
                                    wr = fma(Rnikj * e[0][k], e[1][j], wr);
                                    wi = fma(-Rnikj * e[0][k], e[2][j], wi);
                                }
                        // mbar^i W_i with both factors carrying 1/sqrt2
                        E2r += 0.5 * (e[1][i] * wr + e[2][i] * wi);
                        E2i += 0.5 * (e[1][i] * wi - e[2][i] * wr);
                    }
                    pr = 0.5 * E1r - E2r + 0.5 * E3r;
                    pim = 0.5 * E1i - E2i + 0.5 * E3i;
                }
                extra->psi4[0] = pr;
                extra->psi4[1] = pim;
            }
        }
    }
#undef BC
#undef BCFMA
#undef DH
#undef DH1
#undef D1
#undef D2
#undef ADV
}

}  // namespace grf
