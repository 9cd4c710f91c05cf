"""grf_rk4_step_host on boxes that run as several slabs: the bits of grf_rk4_step for frozen, mirror and periodic
ghosts, a last slab of one plane, 16 slabs, several steps, lopsided advection, pageable buffers and queued in-place
calls. A slab holds at least 291,840 points and 4 planes, so the boxes are wide in x and y."""
import numpy as np
import pytest

import grf_inputs as gi

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


SLAB_POINTS = 5 * 152 * 12 * 32


def slabs(box):
    """The library's rule (grf_api.cu): planes per slab, slabs, planes of the last one."""
    q = min(max(box.nz, 4), max(4, -(-box.nz // 16), -(-SLAB_POINTS // (box.nx * box.ny))))
    s = -(-box.nz // q)
    return q, s, box.nz - q * (s - 1)


def box_of(nz, bc, nx=301, ny=250):
    if bc == gi.BC_REFLECT_LOW:
        return gi.Box(nx, ny, nz, 0.1, 0.05, 0.05, 0.05, bc=bc)
    return gi.Box(nx, ny, nz, 0.1, -0.05 * nx + 0.013, -0.05 * ny + 0.02, -0.05 * nz + 0.03, bc=bc)


def device_state(g, box, seed, poison):
    """A smooth state in the padded layout; a periodic box's ghosts are NaN on request (they must not be read)."""
    import torch
    gen = torch.Generator(device="cuda")
    gen.manual_seed(seed)
    t = g.alloc_state(g.box_like(box))
    ax = [torch.arange(n + 6, dtype=torch.float64, device="cuda") for n in (box.nx, box.ny, box.nz)]
    u = torch.rand((27, 7), generator=gen, dtype=torch.float64, device="cuda").tolist()
    v = t[..., :box.nx + 6]
    for f in range(27):
        a = u[f]
        v[f] = 0.02 * (a[0] - 0.5) * (torch.sin(0.2 * (0.5 + a[1]) * ax[0] + 6 * a[2])[None, None, :] *
                                      torch.cos(0.2 * (0.5 + a[3]) * ax[1] + 6 * a[4])[None, :, None] *
                                      torch.sin(0.3 * (0.5 + a[5]) * ax[2] + 6 * a[6])[:, None, None])
    for f, x in ((0, 0.8), (1, 1.0), (4, 1.0), (6, 1.0), (18, 0.9)):
        v[f] += x
    if poison:
        nan = float("nan")
        v[:, :3], v[..., :3, :], v[..., :3] = nan, nan, nan
        v[:, -3:], v[..., -3:, :], v[..., -3:] = nan, nan, nan
    return t


CASES = {
    # name: (planes, boundary, steps, other parameters, slabs, planes of the last slab)
    "periodic": (13, gi.BC_PERIODIC, 1, {}, 4, 1),
    "frozen_3_steps": (13, gi.BC_FROZEN, 3, {}, 4, 1),
    "mirror_2_steps": (14, gi.BC_REFLECT_LOW, 2, {}, 4, 2),
    "periodic_lopsided_2_steps": (15, gi.BC_PERIODIC, 2, dict(advection=1), 4, 3),
    "frozen_decoupled": (8, gi.BC_FROZEN, 1, dict(decoupled=1), 2, 4),
    "mirror_cubic": (9, gi.BC_REFLECT_LOW, 1, dict(g3=0.1), 3, 1),
    "frozen_16_slabs": (61, gi.BC_FROZEN, 1, {}, 16, 1),
}


def run(g, case):
    nz, bc, nsteps, extra, want, last = CASES[case]
    box = box_of(nz, bc)
    assert slabs(box)[1:] == (want, last)
    b, params = g.box_like(box), g.params_like(gi.Params(lam=0.2, g2=0.1, beta_kind=1, **extra))
    s = device_state(g, box, 5, bc == gi.BC_PERIODIC)
    hin = s.cpu()
    g.grf_rk4_step(b, params, s, 0.25 * box.dx, nsteps)
    return box, b, params, nsteps, hin, s.cpu()[..., :box.nx + 6]


@pytest.mark.parametrize("case", sorted(CASES))
def test_several_slabs_give_the_bits_of_the_device_step(g, case):
    import torch
    box, b, params, nsteps, hin, ref = run(g, case)
    assert torch.isfinite(ref).all()
    hin, hout = hin.pin_memory(), torch.full_like(hin, float("nan")).pin_memory()
    state = torch.full(g.state_shape(b), float("nan"), dtype=torch.float64, device="cuda")
    g.grf_rk4_step_host(b, params, hin, hout, state, 0.25 * box.dx, nsteps)
    torch.cuda.synchronize()
    assert torch.equal(hout[..., :box.nx + 6], ref) and torch.equal(state.cpu()[..., :box.nx + 6], ref)
    assert g.grf_check_status() == 0


@pytest.mark.parametrize("pinned_in,pinned_out", [(False, False), (True, False), (False, True)])
def test_several_slabs_with_pageable_buffers(g, pinned_in, pinned_out):
    import torch
    box, b, params, nsteps, hin, ref = run(g, "frozen_3_steps")
    hout = torch.full_like(hin, float("nan"))
    hin, hout = hin.pin_memory() if pinned_in else hin, hout.pin_memory() if pinned_out else hout
    g.grf_rk4_step_host(b, params, hin if pinned_in else hin.numpy(), hout if pinned_out else hout.numpy(),
                        g.alloc_state(b), 0.25 * box.dx, nsteps)
    torch.cuda.synchronize()
    assert torch.equal(hout[..., :box.nx + 6], ref)


def test_several_slabs_in_place_back_to_back(g):
    """Two calls queued without a synchronisation, host_in == host_out, on a side stream: the second call's copies
    see the first one's result."""
    import torch
    box = box_of(13, gi.BC_FROZEN)
    assert slabs(box)[1] == 4
    b, params = g.box_like(box), g.params_like(gi.Params(lam=0.3, g2=0.05))
    s = device_state(g, box, 9, False)
    h = s.cpu().pin_memory()
    g.grf_rk4_step(b, params, s, 0.25 * box.dx, 2)
    state, ws, side = g.alloc_state(b), g.alloc_workspace(g.grf_workspace_bytes(b, g.GRF_OP_RK4)), torch.cuda.Stream()
    torch.cuda.synchronize()
    for _ in range(2):
        g.grf_rk4_step_host(b, params, h, h, state, 0.25 * box.dx, 1, ws=ws, stream=side)
    side.synchronize()
    assert torch.equal(h[..., :box.nx + 6], s.cpu()[..., :box.nx + 6])
