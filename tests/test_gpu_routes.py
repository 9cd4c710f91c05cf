"""RK4 stage kernels by the size of the box: teams of 4 lanes a point up to 4,864 points, of 2 up to 9,728, one lane
a point above, with an instantiation for each scheme. The larger boxes here reach the one-lane instantiations."""
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


def gpu_rk4(g, box, params, s, dt, n=1):
    b = g.box_like(box)
    t = g.to_device(s, b)
    g.grf_rk4_step(b, g.params_like(params), t, dt, n)
    assert g.grf_check_status() == 0
    return g.to_host(t, b)


def batched_rk4(g, box, params, s, dt, n=1):
    """The same step by the batched kernels, which always take one lane a point."""
    import torch
    b, stream = g.box_like(box), torch.cuda.Stream()
    gp = g.params_array([g.params_like(params)])
    with torch.cuda.stream(stream):
        dev = [g.to_device(s, b)]
        items = g.batch_items([b], dev, [0], [dt])
        cfg = g.batch_config(g.GRF_BATCH_GRAPH, (32, 4, 1))
        g.grf_batched_rk4(items, gp, n, cfg, ws=g.alloc_workspace(g.grf_batched_workspace_bytes(items, cfg)), stream=stream)
    stream.synchronize()
    return g.to_host(dev[0], b)


SCHEMES = {
    "default": dict(beta_kind=1),
    "linear": dict(beta_kind=0),
    "decoupled": dict(beta_kind=1, decoupled=1),
    "exponential": dict(beta_kind=2),
    "exponential_decoupled": dict(beta_kind=2, decoupled=1),
    "cubic": dict(beta_kind=1, g3=0.3),
    "cubic_decoupled": dict(beta_kind=1, g3=0.3, decoupled=1),
    "lopsided": dict(beta_kind=1, advection=1),
    "lopsided_cubic": dict(beta_kind=1, advection=1, g3=0.3),
    "lopsided_decoupled": dict(beta_kind=1, advection=1, decoupled=1),
}
FROZEN, MIRROR = (27, 22, 19, 0.3, -4.0, -3.2, -2.8), (27, 22, 19, 0.3, 0.15, 0.15, 0.15)   # 11,286 points


@pytest.mark.parametrize("scheme", sorted(SCHEMES))
@pytest.mark.parametrize("bc", [gi.BC_PERIODIC, gi.BC_FROZEN, gi.BC_REFLECT_LOW])
def test_one_lane_kernels_against_the_oracle(g, orc, bc, scheme):
    """Tolerance as in test_gpu_parity.py: one step <= 1e-11 of each field's maximum."""
    box = gi.Box(*(MIRROR if bc == gi.BC_REFLECT_LOW else FROZEN), bc=bc)
    params = gi.Params(lam=0.3, g2=0.2, **SCHEMES[scheme])
    s0, dt = state_for(box, 91), 0.25 * box.dx
    cpu = s0.copy()
    orc.rk4(box, params, cpu, dt, 1)
    gpu = gpu_rk4(g, box, params, s0, dt)
    errs = field_errors(gpu, cpu, box)
    assert np.max(errs) < 1e-11, describe(errs)
    if bc != gi.BC_REFLECT_LOW and params.beta_kind != 2 and params.g3 == 0.0:
        # the batched kernels (general instantiation, cubic code included) give the same bits
        assert np.array_equal(box.interior(batched_rk4(g, box, params, s0, dt)), box.interior(gpu))


@pytest.mark.parametrize("bc", [gi.BC_SOMMERFELD, gi.BC_EXTRAPOLATE, gi.BC_REFLECT_LOW_SOMMERFELD])
def test_one_lane_kernels_with_outer_boundaries(g, orc, bc):
    box = gi.Box(*(MIRROR if bc == gi.BC_REFLECT_LOW_SOMMERFELD else FROZEN), bc=bc)
    params = gi.Params(lam=0.3, g2=0.2, beta_kind=1)
    s0, dt = state_for(box, 93), 0.25 * box.dx
    cpu = s0.copy()
    orc.rk4(box, params, cpu, dt, 1)
    errs = field_errors(gpu_rk4(g, box, params, s0, dt), cpu, box)
    assert np.max(errs) < 1e-11, describe(errs)


@pytest.mark.parametrize("advection", [0, 1])
@pytest.mark.parametrize("decoupled", [0, 1])
@pytest.mark.parametrize("size", [(1, 1, 1), (16, 16, 19), (17, 13, 22), (32, 19, 16), (23, 18, 24), (152, 64, 1), (139, 7, 10)])
def test_teams_give_the_bits_of_one_lane(g, size, decoupled, advection):
    """4,864 points are the last for teams of 4 (16 x 16 x 19), 9,728 for teams of 2 (32 x 19 x 16, 152 x 64 x 1)."""
    box = gi.Box(*size, 0.3, 0.4, -0.5 * 0.3 * size[1], -1.1, bc=gi.BC_FROZEN)
    params = gi.Params(lam=0.3, g2=0.2, beta_kind=1, decoupled=decoupled, advection=advection)
    s0, dt = state_for(box, 97), 0.25 * box.dx
    assert np.array_equal(gpu_rk4(g, box, params, s0, dt, 2), batched_rk4(g, box, params, s0, dt, 2))
