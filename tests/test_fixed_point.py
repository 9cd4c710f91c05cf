"""Block fixed point (csrc/grf_fixed.cuh, host build): stencil sums against exact rational arithmetic.

(The kernels take blocks outside its range in FP64: test_ko_of_extreme_values below, on a GPU.)

Bound, from the representation: each value is kept to one unit of 2^-(52 + guard) of the largest one's
leading bit (exactly, when it is within 2^guard of the largest), the integer sum is exact, and the result is
rounded once (the scaled one after a product kept to 63 bits).
"""
import ctypes as C
from fractions import Fraction

import numpy as np
import pytest

KO6 = [1, -6, 15, -20, 15, -6, 1]
MIXED = [a * b for a in (1, -8, 8, -1) for b in (1, -8, 8, -1)]


@pytest.fixture(scope="module")
def fixed_sum():
    from paper_2309_06225_gb300 import build
    L = C.CDLL(build.build_flops())
    L.grf_host_fixed_sum.restype = C.c_double
    L.grf_host_fixed_sum.argtypes = [C.POINTER(C.c_double), C.POINTER(C.c_int), C.c_int, C.c_int, C.c_double]

    def f(x, w, guard, c=0.0):
        x, w = np.ascontiguousarray(x, dtype=np.float64), np.ascontiguousarray(w, dtype=np.int32)
        return L.grf_host_fixed_sum(x.ctypes.data_as(C.POINTER(C.c_double)), w.ctypes.data_as(C.POINTER(C.c_int)),
                                    len(x), guard, c)
    return f


@pytest.mark.parametrize("spread", [0, 2, 12, 70, 400])
@pytest.mark.parametrize("weights,guard", [(KO6 * 3, 2), (MIXED, 1), ([1, -1], 2), ([1], 2)])
def test_sums_against_exact(fixed_sum, weights, guard, spread):
    rng = np.random.default_rng(spread + len(weights))
    for t in range(300):
        n = len(weights)
        x = rng.uniform(1.0, 2.0, n) * rng.choice([-1.0, 1.0], n) * 2.0 ** rng.integers(-spread, 1, n)
        if t % 3 == 0:
            x[rng.integers(n)] = rng.choice([0.0, -0.0])
        if t % 7 == 0:
            x[:] = x[0] * (1.0 + 2.0 ** -52 * rng.integers(0, 3, n))  # nearly equal: massive cancellation
        x *= 2.0 ** int(rng.integers(-300, 300))
        top = Fraction(2) ** (int(np.frexp(np.max(np.abs(x)))[1]) - 1)
        unit = top / 2 ** (52 + guard)
        for c in (0.0, 1.0 / 12.0, 7.3e5, 3.1e-9):
            exact = sum(Fraction(int(w)) * Fraction(float(v)) for w, v in zip(weights, x)) * (Fraction(c) if c else 1)
            got = Fraction(fixed_sum(x, weights, guard, c))
            small = [abs(int(w)) for w, v in zip(weights, x) if v != 0 and abs(Fraction(float(v))) * 2 ** guard < top]
            bound = sum(small) * unit * (Fraction(c) if c else 1)
            bound += abs(exact) * Fraction(1, 2 ** 53) * (1 + Fraction(1, 2 ** 8)) + bound / 2 ** 52
            assert abs(got - exact) <= bound, (x, c, float(got), float(exact))


@pytest.mark.parametrize("rough", [0.0, 1e-12, 1e-3, 1.0])
def test_sixth_order_second_difference_against_exact(rough):
    """The sums whose weights exceed the room above the values: exact while the second differences are small,
    else with them cut to 53 bits (a unit of 2^-53 of the largest one, times the weights 299, at most)."""
    from paper_2309_06225_gb300 import build
    L = C.CDLL(build.build_flops())
    L.grf_host_fixed_second6.restype = C.c_double
    L.grf_host_fixed_second6.argtypes = [C.POINTER(C.c_double)]
    w = [2, -27, 270, -490, 270, -27, 2]
    rng = np.random.default_rng(3)
    for t in range(2000):
        x = (1.0 + rough * rng.uniform(-1, 1, 7)) * 2.0 ** int(rng.integers(-100, 100)) * rng.choice([-1.0, 1.0])
        if rough == 1.0:
            x *= rng.choice([-1.0, 1.0], 7)             # alternating signs: the largest second differences
        f = [Fraction(float(v)) for v in x]
        exact = sum(a * b for a, b in zip(w, f))
        top = Fraction(2) ** (int(np.frexp(np.max(np.abs(x)))[1]) - 1)
        second = max(abs(f[3 + r] + f[3 - r] - 2 * f[3]) for r in (1, 2, 3))
        bound = 299 * (second / 2 ** 53 if second > top / 2 ** 2 else 0) + 1098 * top / 2 ** 54 * any(
            v != 0 and abs(v) * 4 < top for v in f) + abs(exact) * Fraction(1, 2 ** 53)
        got = Fraction(L.grf_host_fixed_second6(x.ctypes.data_as(C.POINTER(C.c_double))))
        assert abs(got - exact) <= bound, (list(x), float(got), float(exact))


@pytest.mark.parametrize("guard", [1, 2])
def test_special_values(fixed_sum, guard):
    w = MIXED
    assert fixed_sum(np.zeros(16), w, guard) == 0.0 and fixed_sum(-np.zeros(16), w, guard, 0.25) == 0.0
    assert fixed_sum(np.full(16, -0.1), w, guard, 12.5) == 0.0          # weights sum to zero
    assert fixed_sum(np.full(16, 1e-310), w, guard) == 0.0              # below the representation's floor
    for bad in (np.nan, np.inf, -np.inf):
        x = np.ones(16)
        x[3] = bad
        assert np.isnan(fixed_sum(x, w, guard)) and np.isnan(fixed_sum(x, w, guard, 2.0))
        assert np.isnan(fixed_sum(np.full(16, bad), w, guard, 1e-30))
    big = np.zeros(16)
    big[5] = 1e308                                                      # beyond the range: the FP64 sums'
    assert np.isnan(fixed_sum(big, w, guard))
    assert fixed_sum(big * 2.0 ** -20, w, guard) == 64 * (1e308 * 2.0 ** -20)


@pytest.mark.gpu
@pytest.mark.parametrize("kind", ["ordinary", "tiny", "huge", "special"])
def test_ko_of_extreme_values(fixed_sum, kind):
    """grf_ko_dissipation on fields of any magnitude: the kernel gives the bits of the host build of the sums
    (checked against exact arithmetic above) or, for a stencil whose largest value is out of the fixed-point
    range, the FP64 sum, whose non-finite values it keeps."""
    torch = pytest.importorskip("torch")
    assert torch.cuda.is_available()
    import paper_2309_06225_gb300 as g
    rng = np.random.default_rng(5)
    dx = 1.0 / 12.0                                     # the spacing constants are 1, 12, 1
    assert (64.0 / 12.0) / (64.0 * dx) == 1.0
    box = g.make_box(11, 7, 5, dx, bc=g.GRF_BC_FROZEN)
    u = rng.normal(size=(27, 11, 13, 17))
    if kind == "tiny":
        u *= 10.0 ** rng.uniform(-320, -200, u.shape)
    elif kind == "huge":
        u *= 10.0 ** rng.uniform(290, 305, (27, 1, 1, 1))
    elif kind == "special":
        u[rng.random(u.shape) < 0.01] = np.nan
        u[rng.random(u.shape) < 0.01] = np.inf
        u[rng.random(u.shape) < 0.05] = 0.0
    t, out = g.to_device(u, box), g.alloc_state(box)
    g.grf_ko_dissipation(box, 64.0 / 12.0, t, out)
    got = g.to_host(out, box)[:, 3:-3, 3:-3, 3:-3]
    st = [(1, 0, 0), (0, 1, 0), (0, 0, 1)]
    weights = [-60] + [w for _ in st for w in (15, 15, -6, -6, 1, 1)]
    top = 2046 - 13 - 3                                 # biased exponents above this take the FP64 sum
    fixed = 0
    for f in range(27):
        for k, j, i in np.ndindex(got.shape[1:]):
            at = lambda d, r: u[f, k + 3 + r * d[2], j + 3 + r * d[1], i + 3 + r * d[0]]
            x = [u[f, k + 3, j + 3, i + 3]] + [at(d, s * r) for d in st for r in (1, 2, 3) for s in (-1, 1)]
            e = int(np.max(np.array(x).view(np.int64) >> 52 & 2047))
            if e <= top:
                fixed += 1
                assert got[f, k, j, i] == fixed_sum(x, weights, 2), (f, k, j, i)
            else:
                with np.errstate(invalid="ignore", over="ignore"):
                    ref = sum(np.longdouble(w) * v for w, v in zip(weights, x))
                assert np.isfinite(ref) or not np.isfinite(got[f, k, j, i])
    assert fixed > 0
