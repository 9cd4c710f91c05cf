"""Points whose fields leave the fixed-point range (grf_fixed.cuh) take their differences in FP64: the values, against
the oracle, in every kernel that gathers; and non-finite values reach the outputs that read them, and no others."""
import numpy as np
import pytest

import grf_inputs as gi
from parity import describe, field_errors

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def g():
    torch = pytest.importorskip("torch")
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_2309_06225_gb300 import build
    build.build()
    import paper_2309_06225_gb300 as grf
    grf.lib()
    return grf


def state_for(box, seed, eps=2e-2):
    mirror = box.bc in (gi.BC_REFLECT_LOW, gi.BC_REFLECT_LOW_SOMMERFELD)
    base = gi.mirror_symmetric_state(box) if mirror else gi.single_puncture(box, amp=0.05)
    return gi.random_perturbed_state(box, seed, base=base, eps=eps)


ROUTES = {
    # name: (extents, ghost layers, other parameters): team of 4, team of 2, one lane a point; lopsided; 6th order
    "team4": ((12, 11, 10), 3, {}),
    "team4_lopsided": ((12, 11, 10), 3, dict(advection=1)),
    "team2": ((19, 18, 17), 3, {}),
    "team2_lopsided": ((19, 18, 17), 3, dict(advection=1)),
    "one_lane": ((27, 22, 19), 3, {}),
    "one_lane_lopsided": ((27, 22, 19), 3, dict(advection=1)),
    "one_lane_cubic": ((27, 22, 19), 3, dict(g3=0.3)),
    "sixth": ((13, 11, 10), 4, {}),
    "sixth_lopsided": ((13, 11, 10), 4, dict(advection=1)),
}


def setup(route):
    """A state whose B^i, which only dissipation changes here (shift_F = eta = 0), is beyond the fixed-point range:
    2^1011 at this spacing."""
    n, ng, extra = ROUTES[route]
    box = gi.Box(*n, 0.3, -0.15 * n[0] + 0.04, -0.15 * n[1] + 0.03, -0.15 * n[2] + 0.02, bc=gi.BC_FROZEN, ng=ng)
    s = state_for(box, 101)
    s[22:25] = 5e304 * (1.0 + 0.1 * np.random.default_rng(1).uniform(-1, 1, s[22:25].shape))
    assert s[22:25].min() > 2.0 ** 1011
    return box, gi.Params(lam=0.3, g2=0.2, beta_kind=1, shift_F=0.0, eta=0.0, **extra), s


@pytest.mark.parametrize("route", sorted(ROUTES))
def test_step_of_fields_beyond_the_range(g, orc, route):
    """One step <= 1e-11 of each field's maximum, as for ordinary fields."""
    box, params, s = setup(route)
    cpu, b = s.copy(), g.box_like(box)
    orc.rk4(box, params, cpu, 0.25 * box.dx, 1)
    t = g.to_device(s, b)
    g.grf_rk4_step(b, g.params_like(params), t, 0.25 * box.dx, 1)
    assert g.grf_check_status() == 0
    errs = field_errors(g.to_host(t, b), cpu, box)
    assert np.all(np.isfinite(cpu)) and np.max(errs) < 1e-11, describe(errs)


@pytest.mark.parametrize("route", ["one_lane", "one_lane_lopsided", "sixth", "sixth_lopsided"])
def test_rhs_and_dissipation_of_fields_beyond_the_range(g, orc, route):
    box, params, s = setup(route)
    b = g.box_like(box)
    t, out = g.to_device(s, b), g.alloc_state(b)
    g.grf_rhs(b, g.params_like(params), t, out)
    errs = field_errors(g.to_host(out, b), orc.rhs(box, params, s), box, state=s, sigma=params.sigma_ko)
    assert np.max(errs) < 1e-11, describe(errs)
    out.zero_()
    g.grf_ko_dissipation(b, 0.3, t, out)
    errs = field_errors(g.to_host(out, b), orc.ko(box, 0.3, s), box, state=s, sigma=0.3)
    assert np.max(errs) < 1e-11, describe(errs)


@pytest.mark.parametrize("bad", [np.nan, np.inf, -np.inf])
@pytest.mark.parametrize("ng", [3, 4])
def test_non_finite_values_reach_their_stencils_only(g, ng, bad):
    """phi at one point: the right-hand sides are non-finite wherever the dissipation reads that point, and points
    whose stencils do not have the bits of the clean state."""
    box = gi.Box(17, 16, 15, 0.3, -2.36, -2.2, -2.07, bc=gi.BC_FROZEN, ng=ng)
    b, params = g.box_like(box), g.params_like(gi.Params(lam=0.3, g2=0.2, beta_kind=1))
    s = state_for(box, 103)
    out = []
    at = np.array([ng + 7, ng + 8, ng + 8])               # z, y, x
    for dirty in (False, True):
        if dirty:
            s[(25,) + tuple(at)] = bad
        t, o = g.to_device(s, b), g.alloc_state(b)
        g.grf_rhs(b, params, t, o)
        out.append(box.interior(g.to_host(o, b)))
    g.grf_check_status()
    d = np.abs(np.indices(out[0].shape[1:]) + ng - at[:, None, None, None])
    line = (np.sort(d, axis=0)[:2].sum(axis=0) == 0) & (d.max(axis=0) <= ng)     # on an axis through the point
    plane = (d.min(axis=0) == 0) & (d.max(axis=0) < ng)                          # on a coordinate plane, near
    assert not np.isfinite(out[1][25][line]).any()
    assert np.array_equal(out[1][:, ~(line | plane)], out[0][:, ~(line | plane)]) and np.isfinite(out[0]).all()
