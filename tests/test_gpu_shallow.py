"""Superpixels of one to five pixel slots per lane, whose samples inside a
neighbour view take bodies of their own: the refinement's best energy against
every candidate summed in full by the per-hypothesis scorer."""
import numpy as np
import pytest
import torch

from paper_1812_06856_gb300 import synth
import parity as PT

pytestmark = pytest.mark.gpu

# scorer and scan take the same candidate through planes that differ by FP32
# rounding; each energy is within the per-hypothesis tolerance of the exact one
REL, ABS = 2 * PT.REL, PT.ABS


# uneven cells around 9, 32, 64, 96, 128 and 144 pixels
@pytest.mark.parametrize("pitch", [3, 5.7, 8, 9.8, 11.3, 12])
@pytest.mark.parametrize("rig", ["arc", "grid"])
def test_shallow_superpixels_keep_the_best_of_all_candidates(pitch, rig):
    from paper_1812_06856_gb300 import lfd
    W, H, V = 160, 120, 4
    r = synth.arc_rig(V, 10.0, 5.0, 150.0, W, H) if rig == "arc" else synth.grid_rig(2, 2, 0.08, 150.0, W, H)
    scene = synth._random_scene(np.random.default_rng(2), 4, 1, 1, float(r.K[0, 0, 0]), 2.0, 8.0, 1.8)
    views = synth.quantize_rgba8(synth.render(r, scene, "cuda")[0])
    maps = [synth.grid_labels_fast(W, H, pitch, True, seed=v, device="cuda") for v in range(V)]
    labels, (GW, GH) = torch.stack([m[0] for m in maps]).contiguous(), maps[0][1:]
    params = synth.method_params(synth.make_config(1, scale=0.3, views=V), num_labels=32, xy_eps=0.0)
    ctx = lfd.Context(0)
    ctx.set_input(views, labels, r.K, r.R, r.t, GW, GH, params)
    planes, _, _ = ctx.plane_sweep()
    # depths of their own: no plane of one view coincides with one of another
    gen = torch.Generator().manual_seed(3)
    state = planes.clone().reshape(-1, 4)
    state[:, 0] *= torch.exp(0.05 * torch.randn(V * GW * GH, generator=gen)).to(state.device)
    _, choice, energy = ctx.iterate(2, state.reshape(planes.shape), want_choice=True)
    ctx.synchronize()
    st, choice, energy = state.cpu().numpy(), choice.cpu().numpy(), energy.cpu().numpy()
    size = int(min(W, H) / np.sqrt(W * H / (GW * GH)))
    offs = lfd.kernel_offsets(size, int(np.floor(size / 5.0 + 0.5)), 2)
    S = GW * GH
    Ki = np.linalg.inv(r.K[0])
    cen = [ctx.get_superpixels(v)["stats"][:, :2].astype(np.float64) for v in range(V)]
    ray = lambda c: Ki @ np.array([c[0], c[1], 1.0])
    for gs in np.random.default_rng(5).choice(V * S, 16, replace=False):
        v, s = divmod(int(gs), S)
        q, ms = [], []
        for m, (dx, dy) in enumerate(offs):
            x, y = s % GW + dx, s // GW + dy
            if not (0 <= x < GW and 0 <= y < GH):
                continue
            j = v * S + y * GW + x
            d, n = float(st[j, 0]), st[j, 1:].astype(np.float64)
            dep = d * (n @ ray(cen[v][y * GW + x])) / (n @ ray(cen[v][s])) if m else d
            if m and (not (params["d_min"] <= dep <= params["d_max"])
                      or abs(n @ ray(cen[v][s])) < 0.1 * np.linalg.norm(ray(cen[v][s]))):
                continue
            q.append((v, s, dep, *n))
            ms.append(m)
        E = ctx.score(state.reshape(planes.shape), q)[:, 0].astype(np.float64)
        best = E.max()
        tol = REL * abs(best) + ABS
        assert abs(energy[gs, 0] - best) <= tol, (gs, energy[gs, 0], best)
        assert E[ms.index(int(choice[gs, 0]))] >= best - tol
    ctx.close()
