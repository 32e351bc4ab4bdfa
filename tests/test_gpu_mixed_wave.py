"""Propagation whose last wave goes to whole CTAs while the waves before it go
to single warps: the same planes, choices and energies as with every superpixel
in a CTA and with every superpixel in a warp."""
import numpy as np
import pytest
import torch

from paper_1812_06856_gb300 import synth

pytestmark = pytest.mark.gpu


def _single_warps(S, sms):
    """Superpixels that single warps take: whole waves of 7 CTAs of 4 warps per SM, unless the rest fills most of one."""
    slots = 7 * 4 * sms
    waves, rest = divmod(S, slots)
    return S if waves >= 4 or 4 * rest >= 3 * slots else waves * slots


# superpixel pitches with one, two and three whole waves and a part of one on 152 SMs
@pytest.mark.parametrize("pitch", [14, 11.4, 9.6])
@pytest.mark.parametrize("rig", ["arc", "grid"])
def test_warps_and_ctas_of_one_launch_agree_with_either(pitch, rig):
    from paper_1812_06856_gb300 import lfd
    W, H, V = 640, 480, 4
    r = synth.arc_rig(V, 30.0, 5.0, 600.0, W, H) if rig == "arc" else synth.grid_rig(2, 2, 0.08, 600.0, W, H)
    scene = synth._random_scene(np.random.default_rng(4), 4, 1, 1, float(r.K[0, 0, 0]), 2.0, 8.0, 1.8)
    views = synth.quantize_rgba8(synth.render(r, scene, "cuda")[0])
    maps = [synth.grid_labels_fast(W, H, pitch, True, seed=v, device="cuda") for v in range(V)]
    labels, (GW, GH) = torch.stack([m[0] for m in maps]).contiguous(), maps[0][1:]
    S = V * GW * GH
    sms = torch.cuda.get_device_properties(0).multi_processor_count
    if sms == 152:
        assert 0 < _single_warps(S, sms) < S
    item = dict(views=views, labels=labels, K=r.K, R=r.R, t=r.t, GW=GW, GH=GH,
                params=synth.method_params(synth.make_config(1, scale=0.3, views=V), num_labels=32, iterations=3))
    out = []
    for opt in (dict(), dict(prop_coop=1), dict(prop_persistent=0)):
        ctx = lfd.Context(0)
        planes, depths = ctx.estimate_batch([item], options=opt)
        ctx.synchronize()
        out.append((planes.clone(), depths[0].clone(), ctx.counters()))
        ctx.close()
    for planes, depth, counters in out[1:]:
        assert torch.equal(planes, out[0][0]) and torch.equal(depth, out[0][1]) and counters == out[0][2]
