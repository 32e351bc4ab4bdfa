"""Refinement on a rig whose neighbours' principal planes cut the depth range, so
that the anchor pixels of current planes lie anywhere up to far outside the
neighbour views: the scan's energy of every chosen plane is the scorer's, which
tests every sample."""
import math

import numpy as np
import pytest
import torch

from paper_1812_06856_gb300 import synth
import parity as PT

pytestmark = pytest.mark.gpu

# the scan takes the chosen plane in FP32 form from its source, the scorer from the rounded output: each energy is
# within the per-hypothesis tolerance of the exact one
REL, ABS = 2 * PT.REL, PT.ABS


def _rig(W, H, deg):
    f = 0.9 * W
    K = np.array([[f, 0, (W - 1) / 2], [0, f, (H - 1) / 2], [0, 0, 1.0]])
    R, t = [np.eye(3)], [np.zeros(3)]
    for side in (-1.0, 1.0):
        a = math.radians(deg)
        z = np.array([-side * math.sin(a), 0.0, math.cos(a)])          # looks across the first camera's axis
        x = np.cross([0.0, 1.0, 0.0], z)
        x /= np.linalg.norm(x)
        r = np.stack([x, np.cross(z, x), z])
        c = np.array([side * 2.5, 0.1 * side, 3.5])
        R.append(r)
        t.append(-r @ c)
    return synth.Rig(np.stack([K] * 3), np.stack(R), np.stack(t), W, H)


@pytest.mark.parametrize("deg", [45, 73, 85])
@pytest.mark.parametrize("pitch", [6, 11, 15])
def test_the_scans_energies_are_the_scorers(deg, pitch):
    from paper_1812_06856_gb300 import lfd
    W, H, V = 480, 270, 3
    r = _rig(W, H, deg)
    g = torch.Generator().manual_seed(deg)
    img = torch.rand((V, H // 6 + 1, W // 6 + 1, 4), generator=g).repeat_interleave(6, 1).repeat_interleave(6, 2)
    views = (img[:, :H, :W] * 255).to(torch.uint8).cuda().contiguous()
    lab, GW, GH = synth.grid_labels_fast(W, H, pitch, False, seed=1, device="cuda")
    labels = torch.stack([lab] * V).contiguous()
    params = dict(d_min=1.0, d_max=8.0, num_labels=32, iterations=1, xy_eps=0.0, eta=0.5, alpha=0.5, sigma=0.05)
    ctx = lfd.Context(0)
    ctx.set_input(views, labels, r.K, r.R, r.t, GW, GH, params)
    S = GW * GH
    rng = np.random.default_rng(deg + pitch)
    n = rng.standard_normal((V * S, 3)) * 0.3
    n[:, 2] -= 1.0
    state = np.concatenate([rng.uniform(1.2, 7.5, (V * S, 1)), n / np.linalg.norm(n, axis=1, keepdims=True)], 1)
    state = torch.from_numpy(state.astype(np.float32)).cuda()
    out, choice, energy = ctx.iterate(1, state, want_choice=True)
    ctx.synchronize()
    o, e = out.cpu().numpy(), energy.cpu().numpy()
    # homogeneous coordinate of the current planes' anchors: some near and behind the neighbours' principal planes
    cen = np.stack([(np.arange(S) % GW + 0.5) * W / GW, (np.arange(S) // GW + 0.5) * H / GH, np.ones(S)], 1)
    X = state[:S, :1].cpu().numpy() * (cen @ np.linalg.inv(r.K[0]).T)
    w = (X @ r.R[1].T + r.t[1])[:, 2]
    assert (w < 0).any() and (w > 0).any() and (np.abs(w) < 0.02).any()
    pick = np.nonzero(e[:, 1] > 0)[0]
    pick = rng.choice(pick, min(600, len(pick)), replace=False)
    E = ctx.score(state, [(int(i) // S, int(i) % S, *[float(v) for v in o[i]]) for i in pick])[:, 0].astype(np.float64)
    far = np.abs(E - e[pick, 1]) > REL * np.abs(E) + ABS
    # a pixel on a rounding boundary of its position or depth split may fall either way in the two forms of a plane
    assert far.mean() <= 0.02, (far.sum(), np.abs(E - e[pick, 1]).max())
    ctx.close()
