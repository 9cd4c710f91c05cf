"""Calls that discard the dissipation sums, or scale them by zero, do not depend on the outermost ghost layer: the
derivatives read two (6th order: three) points to each side."""
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


def state_for(box, seed, eps=2e-2):
    mirror = box.bc in (gi.BC_REFLECT_LOW, gi.BC_REFLECT_LOW_SOMMERFELD)
    base = gi.mirror_symmetric_state(box) if mirror else gi.single_puncture(box, amp=0.05)
    return gi.random_perturbed_state(box, seed, base=base, eps=eps)


@pytest.mark.parametrize("garbage", [1e3, 1e12, 1e30])
@pytest.mark.parametrize("ng", [3, 4])
def test_outermost_ghosts_of_a_frozen_box_do_not_count(g, ng, garbage):
    import torch
    box = gi.Box(13, 11, 10, 0.3, -1.9, -1.6, -1.5, bc=gi.BC_FROZEN, ng=ng)
    b, params = g.box_like(box), g.params_like(gi.Params(lam=0.3, g2=0.2, beta_kind=1, sigma_ko=0.0))
    clean = state_for(box, 83)
    dirty = np.full_like(clean, garbage)
    dirty[:, 1:-1, 1:-1, 1:-1] = clean[:, 1:-1, 1:-1, 1:-1]
    calls = {"rhs": (27, g.grf_rhs), "constraints": (4, g.grf_constraints), "psi4": (2, g.grf_weyl_psi4),
             "densities": (3, g.grf_energy_densities), "hyperbolicity": (4, g.grf_hyperbolicity)}
    for name, (n, call) in calls.items():
        out = []
        for s in (clean, dirty):
            o = g.alloc_state(b, n)
            call(b, params, g.to_device(s, b), o)
            out.append(o.cpu()[:, ng:-ng, ng:-ng, ng:ng + box.nx].contiguous())
        # (bits: where the perturbed chi is negative, next to the puncture, Psi_4's triad is not a number)
        assert torch.isfinite(out[0]).float().mean() > 0.99 and torch.equal(out[0].view(torch.int64), out[1].view(torch.int64)), name
