"""The batched launch's tuner (autotune.py): its candidates differ in what reaches the kernels, and its cache does not
return configurations that were timed on other kernels."""
import numpy as np
import pytest

import grf_inputs as gi


def test_candidates_are_different_launches():
    from paper_2309_06225_gb300 import autotune
    launches = [(v, t[0] * t[1] * t[2]) for v, t in autotune.CANDIDATES]
    assert len(set(launches)) == len(launches)
    assert all(32 <= n <= 128 and n % 32 == 0 for _, n in launches)


def test_cache_key_names_the_kernels():
    import paper_2309_06225_gb300 as g
    from paper_2309_06225_gb300 import autotune
    boxes = [g.box_like(b) for b in gi.amr_like_boxes(4)]
    sig = autotune.signature(boxes)
    key = autotune.cache_key("GPU", boxes)
    assert key.startswith("GPU|") and key.endswith(sig) and autotune.KERNELS in key
    assert key != f"GPU|{sig}"                 # an entry of the kernels with tile shapes


@pytest.mark.gpu
@pytest.mark.parametrize("variant", [1, 2, 3])
@pytest.mark.parametrize("tile", [(32, 2, 1), (32, 1, 1), (8, 4, 2), (37, 1, 2)])
def test_small_tiles_give_the_bits_of_the_single_box_path(variant, tile):
    torch = pytest.importorskip("torch")
    import paper_2309_06225_gb300 as g
    boxes = [gi.Box(13, 9, 7, 0.25, -1.6, -1.1, -0.9, bc=gi.BC_FROZEN), gi.Box(8, 8, 8, 0.3, -1.05, -1.05, -1.05),
             gi.Box(1, 1, 1, 0.1, 1.1, 0.7, 0.9, bc=gi.BC_FROZEN)]
    states = [gi.random_perturbed_state(b, 40 + i, base=gi.single_puncture(b, amp=0.05), eps=2e-2) for i, b in enumerate(boxes)]
    gb, gp = [g.box_like(b) for b in boxes], g.params_array([g.params_like(gi.Params(lam=0.3, g2=0.1, beta_kind=1))])
    ref, dts = [], [0.25 * b.dx for b in boxes]
    for b, s, dt in zip(gb, states, dts):
        t = g.to_device(s, b)
        g.grf_rk4_step(b, gp[0], t, dt, 2)
        ref.append(g.to_host(t, b))
    stream = torch.cuda.Stream()
    with torch.cuda.stream(stream):
        dev = [g.to_device(s, b) for s, b in zip(states, gb)]
        items, cfg = g.batch_items(gb, dev, [0, 0, 0], dts), g.batch_config(variant, tile)
        g.grf_batched_rk4(items, gp, 2, cfg, ws=g.alloc_workspace(g.grf_batched_workspace_bytes(items, cfg)), stream=stream)
    stream.synchronize()
    for b, t, r in zip(gb, dev, ref):
        assert np.array_equal(g.to_host(t, b), r)
