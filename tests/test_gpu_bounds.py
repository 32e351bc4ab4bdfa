"""The bounded scans (hypotheses dropped once they can no longer win) choose
what full sums choose: the refinement against every candidate summed in full
by the per-hypothesis scorer, for each set of energy terms, and against the
cooperative form, which meets the candidates in another order."""
import numpy as np
import pytest
import torch

from paper_1812_06856_gb300 import synth
import parity as PT

pytestmark = pytest.mark.gpu

# scorer and scan take the same candidate through planes that differ by FP32
# rounding; each energy is within the per-hypothesis tolerance of the exact
# one.  xy_eps keeps Eq. 10's split off the tie of a plane with itself.
REL, ABS = 2 * PT.REL, PT.ABS


@pytest.fixture(scope="module")
def lfd():
    from paper_1812_06856_gb300 import lfd as mod
    mod.load()
    return mod


def _bound(lfd, views=4, **over):
    lf = synth.make_config(1, scale=0.3, views=views)
    v, labels, _ = PT.gpu_inputs(lf, "rgba8")
    params = synth.method_params(lf, **dict(dict(num_labels=48, xy_eps=1e-3), **over))
    ctx = lfd.Context(0)
    ctx.set_input(v, labels, lf.rig.K, lf.rig.R, lf.rig.t, lf.GW, lf.GH, params)
    return lf, ctx, (v, labels, params)


@pytest.mark.parametrize("over", [dict(), dict(term_mask=1), dict(term_mask=2), dict(term_mask=3), dict(term_mask=6),
                                  dict(eta=0.0), dict(eta=20.0), dict(depth_domain=1), dict(xy_eps=0.02)])
@pytest.mark.parametrize("views", [2, 4])
def test_iteration_keeps_the_best_of_all_candidates(lfd, over, views):
    lf, ctx, (_, _, params) = _bound(lfd, views, **over)
    planes, _, _ = ctx.plane_sweep()
    state, _, _ = ctx.iterate(1, planes)
    _, choice, energy = ctx.iterate(2, state, want_choice=True)
    st, choice, energy = state.cpu().numpy(), choice.cpu().numpy(), energy.cpu().numpy()
    pitch = np.sqrt(lf.rig.W * lf.rig.H / (lf.GW * lf.GH))
    size = int(min(lf.rig.W, lf.rig.H) / pitch)
    offs = lfd.kernel_offsets(size, int(np.floor(size / 5.0 + 0.5)), 2)
    S, GW, GH = lf.GW * lf.GH, lf.GW, lf.GH
    rng = np.random.default_rng(5)
    Ki = np.linalg.inv(lf.rig.K[0])
    cen = [ctx.get_superpixels(v)["stats"][:, :2].astype(np.float64) for v in range(views)]
    for gs in rng.choice(views * S, 24, replace=False):
        v, s = divmod(int(gs), S)
        gx, gy = s % GW, s // GW
        q, ms = [], []
        for m, (dx, dy) in enumerate(offs):
            x, y = gx + dx, gy + dy
            if not (0 <= x < GW and 0 <= y < GH):
                continue
            j = v * S + y * GW + x
            d, n = float(st[j, 0]), st[j, 1:].astype(np.float64)
            ray = lambda c: Ki @ np.array([c[0], c[1], 1.0])
            dep = d * (n @ ray(cen[v][y * GW + x])) / (n @ ray(cen[v][s])) if m else d
            if m and not (params["d_min"] <= dep <= params["d_max"]):
                continue
            if m and abs(n @ ray(cen[v][s])) < 0.1 * np.linalg.norm(ray(cen[v][s])):
                continue
            q.append((v, s, dep, *n))
            ms.append(m)
        E = ctx.score(state, q)[:, 0].astype(np.float64)
        best = E.max()
        tol = REL * abs(best) + ABS
        assert abs(energy[gs, 0] - best) <= tol, (gs, energy[gs, 0], best)
        assert E[ms.index(int(choice[gs, 0]))] >= best - tol
        assert energy[gs, 1] >= energy[gs, 0]


@pytest.mark.parametrize("colour", [None, float("nan"), float("inf")])
def test_scan_order_does_not_change_the_choice(lfd, colour):
    lf, _, _ = _bound(lfd, 4)
    v, labels, _ = PT.gpu_inputs(lf, "rgba_f32") if colour is not None else PT.gpu_inputs(lf, "rgba8")
    if colour is not None:
        v[1, 10:20, 15:40, 1] = colour
    item = dict(views=v, labels=labels, K=lf.rig.K, R=lf.rig.R, t=lf.rig.t, GW=lf.GW, GH=lf.GH,
                params=synth.method_params(lf, num_labels=48, iterations=3, perturb_samples=6))
    out = []
    for opt in (dict(), dict(prop_coop=1), dict(prop_batch=16), dict(prop_persistent=0)):
        ctx = lfd.Context(0)
        planes, depths = ctx.estimate_batch([item], options=opt)
        ctx.synchronize()
        hyp, samples = ctx.counters()
        sweep, refine = ctx.samples_taken()
        assert 0 < sweep and 0 < refine and sweep + refine <= samples
        out.append((planes.clone(), depths[0].clone(), hyp, samples))
    for planes, depth, hyp, samples in out[1:]:
        assert torch.equal(planes, out[0][0]) and torch.equal(depth, out[0][1])
        assert (hyp, samples) == out[0][2:]


def _views(kind, rig, fmt):
    H, W, V = rig.H, rig.W, rig.V
    if kind == "rendered":
        scene = synth._random_scene(np.random.default_rng(2), 4, 1, 1, float(rig.K[0, 0, 0]), 2.0, 8.0, 1.8)
        rgb, _, _ = synth.render(rig, scene, "cuda")
    else:                      # "flat": every label costs the same; "steps": many labels tie, few differ
        rgb = torch.full((V, H, W, 3), 0.25, dtype=torch.float64, device="cuda")
        if kind == "steps":
            rgb[:, :, W // 2:] = 0.75
    if fmt == "rgba8":
        return synth.quantize_rgba8(rgb)
    dt = {"rgba_f16": torch.float16, "rgba_bf16": torch.bfloat16, "rgba_f32": torch.float32}[fmt]
    v = synth.to_rgba_float(rgb, dt)
    if kind == "rendered":     # a few texels without a finite colour
        v[0, H // 2, W // 3, 0] = float("nan")
        v[1, H // 3, W // 2, 1] = float("inf")
    return v


# label counts around a pass (32), the lane stage (48) and the bounded sweep's limit (256); pitches with
# superpixels below a warp, around one chunk of 128 pixels, of several chunks, and above 4096 pixels
@pytest.mark.parametrize("rig,fmt,form,L,pitch,kind", [
    ("grid", "rgba_f16", 2, 256, 16, "rendered"), ("grid", "rgba8", 2, 255, 5, "rendered"),
    ("grid", "rgba8", 1, 33, 11, "rendered"), ("arc", "rgba8", 0, 256, 14, "rendered"),
    ("arc", "rgba_bf16", 0, 49, 23, "rendered"), ("arc", "rgba_f32", 0, 100, 12, "rendered"),
    ("grid", "rgba_f32", 2, 64, 9, "rendered"), ("grid", "rgba_f32", 1, 48, 30, "rendered"),
    ("pair", "rgba8", 2, 32, 8, "rendered"), ("pair", "rgba_f16", 2, 1, 16, "rendered"),
    ("pair", "rgba_f16", 0, 2, 16, "rendered"), ("grid", "rgba8", 2, 257, 16, "rendered"),
    ("grid", "rgba8", 2, 256, 16, "flat"), ("arc", "rgba8", 0, 200, 16, "flat"),
    ("grid", "rgba8", 2, 256, 16, "steps"), ("arc", "rgba_f16", 0, 256, 20, "steps"),
    ("grid", "rgba8", 2, 70, 90, "rendered"), ("arc", "rgba8", 0, 70, 300, "rendered"),
])
@pytest.mark.parametrize("T", [0.04, 1e-6, float("inf")])
def test_bounded_sweep_picks_the_full_sweeps_label(lfd, rig, fmt, form, L, pitch, kind, T):
    W, H = 301, 203
    f = 300.0 * W / 320.0
    r = {"grid": lambda: synth.grid_rig(2, 2, 0.08, f, W, H), "arc": lambda: synth.arc_rig(5, 30.0, 5.0, f, W, H),
         "pair": lambda: synth.line_rig(2, 0.1, f, W, H)}[rig]()
    views = _views(kind, r, fmt)
    maps = [synth.grid_labels_fast(W, H, pitch, True, seed=v, device="cuda") for v in range(r.V)]
    labels, (GW, GH) = torch.stack([m[0] for m in maps]).contiguous(), maps[0][1:]
    ctx = lfd.Context(0)
    ctx.set_pair_forms(form)
    ctx.set_input(views, labels, r.K, r.R, r.t, GW, GH, dict(d_min=2.0, d_max=8.0, num_labels=L, T=T))
    assert ctx.pair_form() == form
    full_planes, full_labels, _ = ctx.plane_sweep(want_labels=True, want_costs=True)
    taken_full = ctx.samples_taken()[0]
    planes, lab, _ = ctx.plane_sweep(want_labels=True)
    ctx.synchronize()
    assert torch.equal(lab, full_labels)
    assert torch.equal(planes, full_planes)
    assert taken_full == L * r.V * W * H * (r.V - 1)
    if kind == "rendered" and 64 <= L <= 256 and T == 0.04 and pitch < 60:
        assert ctx.samples_taken()[0] - taken_full < 0.9 * taken_full      # labels were excluded
