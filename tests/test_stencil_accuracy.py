"""Differences and dissipation sums in block fixed point (csrc/grf_diffs.cuh, host build) against exact rational
arithmetic, beside the FP64 sums of the same stencils (fused as in the kernels' FP64 fallback): on every kind of
field, smooth, steep, in a Gaussian's tail or rough, the fixed-point result has to be at least as near."""
import ctypes as C
from fractions import Fraction as F

import numpy as np
import pytest

H = 0.25                                     # a power of two: the spacing factors round alike on both sides
SYM = ((0, 0), (0, 1), (0, 2), (1, 1), (1, 2), (2, 2))


@pytest.fixture(scope="module")
def host():
    from paper_2309_06225_gb300 import build
    L = C.CDLL(build.build_flops())
    P = C.POINTER(C.c_double)
    L.grf_host_diffs.argtypes = [C.c_int, C.c_double, C.c_int, P, P, P, P]

    def diffs(ng, axes, planes, beta, outer=1, dx=H):
        out = np.full(13, np.nan)
        a = [np.ascontiguousarray(q, dtype=np.float64) for q in (axes, planes, beta)]
        st = L.grf_host_diffs(ng, dx, outer, *[q.ctypes.data_as(P) for q in a], out.ctypes.data_as(P))
        return None if st else out
    return diffs


def fma(a, b, c):
    return float(F(a) * F(b) + F(c))         # one rounding


def fields(rng):
    x0, y0, z0 = rng.uniform(-4, 4, 3)
    p, k = rng.uniform(-3, 3, 3), rng.uniform(0.2, 0.9, 3)
    n = rng.normal(size=3)
    o = n / np.linalg.norm(n) * rng.uniform(4, 8)
    noise = rng.uniform(-1, 1, (9, 9, 9))
    s, c, e = np.sin, np.cos, np.exp
    return {
        "smooth": lambda i, j, l: 1 + 0.3 * s(k[0] * (x0 + i * H) + p[0]) * c(k[1] * (y0 + j * H) + p[1]) * s(k[2] * (z0 + l * H) + p[2]),
        "perturbation": lambda i, j, l: 2e-3 * s(k[0] * (x0 + i * H) + p[0]) * c(k[1] * (y0 + j * H) + p[1]) * s(z0 + l * H + p[2]),
        "puncture": lambda i, j, l: (1 + 0.5 / np.sqrt(((x0 + i * H) ** 2 + (y0 + j * H) ** 2 + (z0 + l * H) ** 2) / 9)) ** -4,
        "tail": lambda i, j, l: 1e-2 * e(-((o[0] + i / 2) ** 2 + (o[1] + j / 2) ** 2 + (o[2] + l / 2) ** 2)),
        "zero": lambda i, j, l: 2e-3 * s(k[0] * i * H + 0.1 * p[0]) * c(k[1] * (y0 + j * H) + p[1]) * c(z0 + l * H),
        "steep": lambda i, j, l: e(-2 * (x0 + 4 + i * H) ** 2) * (1 + 1e-3 * s(k[1] * j * H + p[1]) + 1e-3 * c(z0 + l * H)),
        "rough": lambda i, j, l: noise[i + 4, j + 4, l + 4],
    }


def stencil(f, ng):
    line = [[[float(f(*(sg * (k + 1) * (d == q) for q in range(3)))) for k in range(ng)] for sg in (-1, 1)] for d in range(3)]
    off = [o for o in range(1 - ng, ng) if o]
    planes = [[[float(f(*(o * (a == q) + m * (b == q) for q in range(3)))) for m in off] for o in off]
              for a, b in ((0, 1), (0, 2), (1, 2))]
    return float(f(0, 0, 0)), line, planes


def sums(c, line, planes, beta, ng, fp64):
    """The 13 results: rational (fp64 = False), or in FP64."""
    one = fma if fp64 else (lambda a, b, x: a * b + x)
    if not fp64:
        q = lambda t: [q(y) for y in t] if isinstance(t, list) else F(t)
        c, line, planes = F(c), q(line), q(planes)
    h = H if fp64 else F(H)
    i1, i2 = (1 / (12 * h), 1 / (12 * h * h)) if ng == 3 else (1 / (60 * h), 1 / (180 * h * h))

    def first(a):                            # values at -w .. -1, 1 .. w
        if ng == 3:
            return one(8, a[2] - a[1], a[0] - a[3])
        return one(45, a[3] - a[2], one(-9, a[4] - a[1], a[5] - a[0]))
    out, t, up = [], [0] * ng, []
    w = ng - 1
    for d in range(3):
        out.append(first(line[d][0][:w][::-1] + line[d][1][:w]) * i1)
    d2 = {}
    for d in range(3):
        m, p = line[d]
        pr = [p[k] + m[k] for k in range(ng)]
        x = one(-30, c, one(16, pr[0], -pr[1])) if ng == 3 else one(270, pr[0], one(-27, pr[1], one(2, pr[2], -490 * c)))
        d2[d, d] = x * i2
        a, b = (p, m) if beta[d] >= 0 else (m, p)
        if ng == 3:
            x = one(18, a[0], one(-6, a[1], a[2])) - one(3, b[0], 10 * c)
        else:
            x = one(80, a[0], one(-30, a[1], one(8, a[2], -a[3]))) + one(2, b[1], one(-24, b[0], -35 * c))
        up.append(x * i1)
    for (a, b), x in zip(((0, 1), (0, 2), (1, 2)), planes):
        r = [first(y) * i1 for y in x]
        d2[a, b] = first(r) * i1
    for k in range(ng):
        t[k] = (line[0][0][k] + line[0][1][k]) + (line[1][0][k] + line[1][1][k]) + (line[2][0][k] + line[2][1][k])
    if ng == 3:
        ko = one(-60, c, one(15, t[0], one(-6, t[1], t[2])))
    else:
        ko = one(210, c, one(-56, t[0], one(28, t[1], one(-8, t[2], t[3]))))
    return out + [d2[s] for s in SYM] + [ko] + up


KIND = ["first"] * 3 + ["second" if a == b else "mixed" for a, b in SYM] + ["dissipation"] + ["lopsided"] * 3


@pytest.mark.parametrize("ng", [3, 4])
@pytest.mark.parametrize("family", list(fields(np.random.default_rng(0))))
def test_no_further_off_than_fp64(host, family, ng):
    rng = np.random.default_rng(17)
    err = {k: np.zeros((2, 2)) for k in set(KIND)}         # [fixed, FP64] x [relative, relative to the values]
    for _ in range(120):
        c, line, planes = stencil(fields(rng)[family], ng)
        beta = rng.uniform(-1, 1, 3)
        axes = [c] + [x for d in range(3) for s in range(2) for x in line[d][s]]
        exact = sums(c, line, planes, beta, ng, False)
        got, ref = host(ng, axes, planes, beta), sums(c, line, planes, beta, ng, True)
        top = F(max(abs(x) for x in axes))
        for m, k in enumerate(KIND):
            if exact[m] == 0:
                continue
            for s, x in enumerate((got[m], ref[m])):
                e = abs(F(float(x)) - exact[m])
                err[k][s] += min(1e-3, float(e / abs(exact[m]))), float(e / top) ** 2
    for k, ((rel, ab), (rel64, ab64)) in err.items():
        assert rel <= 1.1 * rel64 and ab <= 1.1 ** 2 * ab64, (family, k, rel, rel64, ab, ab64)


@pytest.mark.parametrize("ng", [3, 4])
@pytest.mark.parametrize("garbage", [1e3, 1e12, 1e30, 1e300, np.inf, np.nan])
def test_derivatives_keep_clear_of_the_outermost_points(host, ng, garbage):
    """The points at +-ng enter the dissipation and lopsided sums alone: whatever stands there, the centred
    derivatives have the bits of a stencil without them."""
    rng = np.random.default_rng(3)
    for name, f in fields(rng).items():
        c, line, planes = stencil(f, ng)
        axes = np.array([c] + [x for d in range(3) for s in range(2) for x in line[d][s]])
        want = host(ng, axes, planes, np.ones(3), outer=0)
        axes[ng::ng] = garbage
        assert np.array_equal(host(ng, axes, planes, np.ones(3), outer=0)[:9], want[:9])
        got = host(ng, axes, planes, np.ones(3))
        if got is not None:                  # (None: the point takes the FP64 sums)
            assert np.array_equal(got[:9], want[:9]), (name, ng, garbage)
        else:
            assert not abs(garbage) < 1e300


@pytest.mark.parametrize("ng", [3, 4])
def test_spacings_whose_factors_are_not_normal_take_fp64(host, ng):
    """1 / dx^2 beyond the doubles, or below the normal ones: the FP64 sums give what their division gives."""
    c, line, planes = stencil(fields(np.random.default_rng(2))["smooth"], ng)
    axes = [c] + [x for d in range(3) for s in range(2) for x in line[d][s]]
    for dx in (1e-160, 1e-200, 1e153, 1e160, 1e300):
        assert host(ng, axes, planes, np.ones(3), dx=dx) is None
    for dx in (1e-100, 1.0, 1e100):
        assert np.all(np.isfinite(host(ng, axes, planes, np.ones(3), dx=dx)))
