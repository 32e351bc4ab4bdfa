"""Fusion over view counts: every width of the candidate registers, the
many-views form and more references than one group holds, against the FP64
fusion oracle, and again on the same context (the z-buffers are left clear)."""
import numpy as np
import pytest
import torch

from oracle import oracle as orc
from paper_1812_06856_gb300 import synth

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def lfd():
    from paper_1812_06856_gb300 import lfd as mod
    mod.load()
    return mod


def _bound(lfd, V, W, H):
    rig = synth.line_rig(V, 0.02, 0.9 * W, W, H)
    lab, GW, GH = synth.grid_labels(W, H, 8)
    views = torch.zeros((V, H, W, 4), dtype=torch.uint8, device="cuda")
    labels = torch.from_numpy(np.stack([lab] * V)).cuda()
    ctx = lfd.Context(0)
    ctx.set_input(views, labels, rig.K, rig.R, rig.t, GW, GH, dict(d_min=1.0, d_max=5.0, num_labels=8))
    return rig, ctx


def _depth(V, W, H, seed):
    rng = np.random.default_rng(seed)
    y, x = np.mgrid[0:H, 0:W]
    base = np.where((x // 11 + y // 9) % 2 == 0, 1.7, 3.1)
    d = base[None] * (1.0 + 0.006 * rng.standard_normal((V, H, W)))
    d = np.where(rng.random(d.shape) < 0.06, rng.uniform(1.0, 5.0, d.shape), d)
    d = np.where(rng.random(d.shape) < 0.05, 0.0, d).astype(np.float32)
    d[0, 0, :4] = [np.nan, np.inf, -1.0, 1e-30]
    return torch.from_numpy(d).cuda()


@pytest.mark.parametrize("V,W,H", [(2, 64, 48), (3, 33, 21), (5, 61, 47), (6, 40, 40), (9, 67, 35), (10, 65, 33),
                                   (16, 40, 23), (17, 40, 23), (32, 31, 17), (33, 31, 17), (40, 19, 11)])
def test_fusion_matches_the_oracle_for_every_view_count(lfd, V, W, H):
    rig, ctx = _bound(lfd, V, W, H)
    for seed in (1, 2):
        d = _depth(V, W, H, seed)
        g = ctx.fuse(d)
        ctx.synchronize()
        g = g.cpu().numpy().astype(np.float64)
        clean = torch.where(torch.isfinite(d), d, torch.zeros_like(d)).cpu().numpy().astype(np.float64)
        ref, flags = orc.fuse(rig.K, rig.R, rig.t, [clean[v] for v in range(V)], tau=0.01)
        for v in range(V):
            ok = (flags[v] == 0)
            assert ok.any()
            assert np.all(np.abs(g[v] - ref[v])[ok] <= 2e-5 * np.abs(ref[v])[ok])


def test_fusion_after_a_larger_and_a_smaller_light_field(lfd):
    rig, ctx = _bound(lfd, 4, 40, 30)
    d = _depth(4, 40, 30, 3)
    first = ctx.fuse(d).clone()
    ctx.synchronize()
    rig2, ctx2 = _bound(lfd, 4, 40, 30)
    lab, GW, GH = synth.grid_labels(90, 70, 8)
    big = synth.line_rig(7, 0.02, 80.0, 90, 70)
    ctx2.set_input(torch.zeros((7, 70, 90, 4), dtype=torch.uint8, device="cuda"),
                   torch.from_numpy(np.stack([lab] * 7)).cuda(), big.K, big.R, big.t, GW, GH,
                   dict(d_min=1.0, d_max=5.0, num_labels=8))
    ctx2.fuse(_depth(7, 90, 70, 4))
    lab, GW, GH = synth.grid_labels(40, 30, 8)
    ctx2.set_input(torch.zeros((4, 30, 40, 4), dtype=torch.uint8, device="cuda"),
                   torch.from_numpy(np.stack([lab] * 4)).cuda(), rig2.K, rig2.R, rig2.t, GW, GH,
                   dict(d_min=1.0, d_max=5.0, num_labels=8))
    again = ctx2.fuse(d)
    ctx2.synchronize()
    assert torch.equal(first, again)
