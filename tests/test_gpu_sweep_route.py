"""Which sweep a light field takes follows from its own sizes and label count:
one that needs the full sweep does not take it for the others of the call, and
the results are those of each light field by itself."""
import numpy as np
import pytest
import torch

from paper_1812_06856_gb300 import synth

pytestmark = pytest.mark.gpu


def _item(lf_index, pitch, labels, rig="grid", W=320, H=240, V=4):
    r = synth.arc_rig(V, 30.0, 5.0, 300.0, W, H) if rig == "arc" else synth.grid_rig(2, 2, 0.08, 300.0, W, H)
    scene = synth._random_scene(np.random.default_rng(lf_index + 1), 4, 1, 1, 300.0, 2.0, 8.0, 1.8)
    views = synth.quantize_rgba8(synth.render(r, scene, "cuda")[0])
    maps = [synth.grid_labels_fast(W, H, pitch, True, seed=v, device="cuda") for v in range(V)]
    lab, (GW, GH) = torch.stack([m[0] for m in maps]).contiguous(), maps[0][1:]
    return dict(views=views, labels=lab, K=r.K, R=r.R, t=r.t, GW=GW, GH=GH,
                params=dict(d_min=2.0, d_max=8.0, num_labels=labels, iterations=0, lf_index=lf_index))


def _full(item):
    V, H, W = item["views"].shape[:3]
    return item["params"]["num_labels"] * V * H * W * (V - 1)


def test_a_light_field_of_many_labels_leaves_the_others_bounded():
    from paper_1812_06856_gb300 import lfd
    small, large = _item(0, 16, 64), _item(1, 16, 257)
    ctx = lfd.Context(0)
    planes, _ = ctx.estimate_batch([small, large], want_depth=False)
    ctx.synchronize()
    taken = ctx.samples_taken()[0]
    assert _full(large) < taken < _full(large) + 0.9 * _full(small)
    alone = []
    for item in (small, large):
        p, _ = ctx.estimate_batch([item], want_depth=False)
        ctx.synchronize()
        alone.append(p.clone())
    assert torch.equal(planes, torch.cat(alone))
    ctx.close()


# (rig, pitch, labels, full): each side of the rule's lines
@pytest.mark.parametrize("rig,pitch,labels,full", [("grid", 4, 64, True), ("grid", 5, 64, False), ("arc", 6, 40, True),
                                                   ("arc", 6, 96, False), ("arc", 8, 40, False), ("arc", 40, 129, True),
                                                   ("arc", 40, 128, False), ("grid", 40, 200, False),
                                                   ("grid", 48, 200, True)])
def test_both_sides_of_the_rule_pick_the_full_sweeps_labels(rig, pitch, labels, full):
    from paper_1812_06856_gb300 import lfd
    item = _item(0, pitch, labels, rig)
    ctx = lfd.Context(0)
    ctx.set_input(*[item[k] for k in ("views", "labels", "K", "R", "t", "GW", "GH", "params")])
    planes, lab, _ = ctx.plane_sweep(want_labels=True)
    taken = ctx.samples_taken()[0]
    want, want_lab, _ = ctx.plane_sweep(want_labels=True, want_costs=True)
    ctx.synchronize()
    assert torch.equal(planes, want) and torch.equal(lab, want_lab)
    assert (taken == _full(item)) == full
    ctx.close()
