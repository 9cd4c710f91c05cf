"""Rounding errors of the pointwise right-hand side (csrc/grf_point.cuh on the host, double against long
double on the same point data) near a puncture, where the curvature's large terms cancel.

BOUND holds, for each field, the root-mean-square error over that of the field's right-hand side that the plain
formulation has on this data: the Ricci tensor and D_i Z_j term by term, S_ij formed from the solution of the
system for (d_t K_ij, d_t Pi), products and sums fused. The present one has to be as accurate, with a margin of
a tenth for the differences in how two sums of the same terms round.
"""
import ctypes as C
import os
import subprocess

import numpy as np
import pytest

from test_kernel_formulas import D1_FIELDS, D2_FIELDS

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))
SRC = """
#include <math.h>
#include "grf_point.cuh"
#include "grf.h"
template <typename T>
static void eval(const grf_params* p, const double* v, const double* d1, const double* d2, T* rhs, int n) {
    grf::CoeffsT<T> c;
    c.kappa1 = p->kappa1; c.kappa2 = p->kappa2; c.kappa3 = p->kappa3; c.shift_F = p->shift_F; c.eta = p->eta;
    c.lam = p->lambda; c.g2 = p->g2; c.g3 = p->g3;
    c.inv_1pa = 1.0 / (1.0 + p->a0); c.a_1pa = p->a0 / (1.0 + p->a0);
    c.bK = 3.0 * p->b0 / (4.0 * (1.0 + p->b0)); c.bTh = 1.0 / (2.0 * (1.0 + p->b0));
    c.beta_kind = p->beta_kind; c.beta_kappa = p->beta_kappa; c.decoupled = p->decoupled; c.advection = 0;
    for (; n > 0; --n, v += 27, d1 += 72, d2 += 72, rhs += 27) {
        grf::PointInT<T> in;
        for (int f = 0; f < 27; ++f) in.v[f] = v[f];
        for (int m = 0; m < 72; ++m) { in.d1[m / 3][m % 3] = d1[m]; in.d2[m / 6][m % 6] = d2[m]; }
        bool ok = true;
        grf::point_rhs<T, T>(c, in, rhs, nullptr, ok);
    }
}
extern "C" void eval_double(const grf_params* p, const double* v, const double* d1, const double* d2, double* r, int n) {
    eval<double>(p, v, d1, d2, r, n);
}
extern "C" void eval_long(const grf_params* p, const double* v, const double* d1, const double* d2, long double* r, int n) {
    eval<long double>(p, v, d1, d2, r, n);
}
"""
NAMES = (["chi"] + ["h%d" % m for m in range(6)] + ["K"] + ["A%d" % m for m in range(6)] + ["Theta"] +
         ["Gamma%d" % m for m in range(3)] + ["lapse"] + ["shift%d" % m for m in range(3)] + ["B%d" % m for m in range(3)] +
         ["phi", "Pi"])
BOUND = {
    (0, 0.0): [9.46e-17, 1.67e-16, 1.27e-16, 1.30e-16, 1.58e-16, 1.07e-16, 1.23e-16, 2.37e-15, 5.98e-16, 4.07e-16, 4.14e-16,
               5.21e-16, 3.89e-16, 5.58e-16, 9.61e-15, 2.62e-16, 2.44e-16, 2.52e-16, 8.74e-17, 1.66e-16, 1.66e-16, 1.60e-16,
               2.41e-16, 2.42e-16, 2.42e-16, 4.76e-17, 2.45e-16],
    (1, 0.0): [9.46e-17, 1.67e-16, 1.27e-16, 1.30e-16, 1.58e-16, 1.07e-16, 1.23e-16, 2.37e-15, 6.01e-16, 4.01e-16, 4.11e-16,
               5.21e-16, 3.86e-16, 5.52e-16, 9.61e-15, 2.54e-16, 2.38e-16, 2.44e-16, 8.74e-17, 1.66e-16, 1.66e-16, 1.60e-16,
               2.36e-16, 2.37e-16, 2.35e-16, 4.76e-17, 2.19e-16],
    (0, 0.02): [9.46e-17, 1.67e-16, 1.27e-16, 1.30e-16, 1.58e-16, 1.07e-16, 1.23e-16, 2.37e-15, 6.05e-16, 4.08e-16, 4.11e-16,
                5.24e-16, 3.85e-16, 5.58e-16, 9.60e-15, 2.58e-16, 2.39e-16, 2.49e-16, 8.74e-17, 1.66e-16, 1.66e-16, 1.60e-16,
                2.38e-16, 2.37e-16, 2.38e-16, 4.76e-17, 2.53e-16],
}


@pytest.fixture(scope="module")
def lib(tmp_path_factory):
    if np.finfo(np.longdouble).nmant < 60:
        pytest.skip("long double is no wider than needed here")
    d = tmp_path_factory.mktemp("pointwise")
    (d / "e.cpp").write_text(SRC)
    subprocess.check_call(["g++", "-std=c++17", "-O2", "-ffp-contract=off", "-w", "-shared", "-fPIC",
                           "-I" + os.path.join(ROOT, "include"), "-I" + os.path.join(ROOT, "paper_2309_06225_gb300", "csrc"),
                           str(d / "e.cpp"), "-o", str(d / "e.so")])
    return C.CDLL(str(d / "e.so"))


def field_values(x, y, z):
    """Two punctures and a scalar bump, with small smooth perturbations of every field."""
    rng = np.random.default_rng(7)
    psi = 1.0 + sum(0.5 * m / np.sqrt((x - 0.03) ** 2 + (y + 0.03) ** 2 + (z - c) ** 2) for m, c in ((0.55, 3.04), (0.45, -2.96)))
    u = np.zeros((27,) + x.shape)
    u[0], u[18] = psi ** -4, psi ** -2
    u[[1, 4, 6]] = 1.0
    u[25] = 8e-3 * np.exp(-(x ** 2 + (y - 0.5) ** 2 + (z - 2.0) ** 2) / 4.0)
    for f in range(27):
        k, ph = rng.uniform(0.3, 0.9, 3), rng.uniform(0.0, 6.0, 3)
        u[f] += (1e-4 if f in (0, 18) else 2e-3) * rng.uniform(-1, 1) * (
            np.sin(k[0] * x + ph[0]) * np.cos(k[1] * y + ph[1]) * np.sin(k[2] * z + ph[2]))
    return u


def point_data(n=3000, h=0.125):
    """Values and 4th-order differences at n grid points within 2.5 of the upper puncture."""
    rng = np.random.default_rng(1)
    r, t, a = 2.5 * rng.random(n) ** (1 / 3), np.arccos(rng.uniform(-1, 1, n)), rng.uniform(0, 2 * np.pi, n)
    o = np.round(np.stack([r * np.sin(t) * np.cos(a), r * np.sin(t) * np.sin(a), 3.0 + r * np.cos(t)]) / h) * h

    def at(*s):
        return field_values(*(o[d] + h * s[d] for d in range(3)))
    w = {-2: 1.0, -1: -8.0, 1: 8.0, 2: -1.0}
    e = np.eye(3, dtype=int)
    v, d1, d2 = at(0, 0, 0), np.zeros((27, 3, n)), np.zeros((27, 6, n))
    for d in range(3):
        line = {k: at(*(k * e[d])) for k in w}
        d1[:, d] = sum(w[k] * line[k] for k in w) / (12 * h)
        d2[:, (0, 3, 5)[d]] = (16 * (line[1] + line[-1]) - line[2] - line[-2] - 30 * v) / (12 * h * h)
    for m, (a, b) in zip((1, 2, 4), ((0, 1), (0, 2), (1, 2))):
        d2[:, m] = sum(w[k] * w[l] * at(*(k * e[a] + l * e[b])) for k in w for l in w) / (144 * h * h)
    return [np.ascontiguousarray(np.moveaxis(q, -1, 0).reshape(n, -1)) for q in (v, d1[D1_FIELDS], d2[D2_FIELDS])]


def errors(lib, decoupled, g3):
    import paper_2309_06225_gb300 as grf
    v, d1, d2 = point_data()
    n = len(v)
    p = grf.grf_params(0.1, 0.0, 1.0, 0.75, 1.0, 0.2, 0.4, 0.05, 0.01, 0.3, 1e-4, 1e-4, 1, 1, decoupled, 0, 1.0, g3)
    got, ref = np.zeros((n, 27)), np.zeros((n, 27), dtype=np.longdouble)
    ptr = [q.ctypes.data_as(C.c_void_p) for q in (v, d1, d2)]
    lib.eval_double(C.byref(p), *ptr, got.ctypes.data_as(C.c_void_p), n)
    lib.eval_long(C.byref(p), *ptr, ref.ctypes.data_as(C.c_void_p), n)
    return np.sqrt(((got - ref) ** 2).sum(0) / (ref ** 2).sum(0)).astype(float)


@pytest.mark.parametrize("decoupled,g3", [(0, 0.0), (1, 0.0), (0, 0.02)])
def test_right_hand_side_rounds_as_the_plain_formulation(lib, decoupled, g3):
    err = errors(lib, decoupled, g3)
    for f in range(27):
        assert err[f] <= 1.1 * BOUND[decoupled, g3][f], (NAMES[f], err[f], BOUND[decoupled, g3][f])
