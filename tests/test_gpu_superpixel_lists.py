"""Superpixel lists and statistics (and the allocation-free statistics) on
label maps at the edges of their kernels: strips of 32 x 32 pixels, boxes below
a warp's step and above the limit that a whole CTA takes, scattered labels,
empty labels, and every pixel format."""
import numpy as np
import pytest
import torch

from paper_1812_06856_gb300 import synth

pytestmark = pytest.mark.gpu

DT = {"rgba8": torch.uint8, "rgba_f16": torch.float16, "rgba_bf16": torch.bfloat16, "rgba_f32": torch.float32}


@pytest.fixture(scope="module")
def lfd():
    from paper_1812_06856_gb300 import lfd as mod
    mod.load()
    return mod


def _labels(kind, W, H, rng):
    if kind == "grid":
        return synth.grid_labels(W, H, 7, True, seed=3)
    if kind == "scattered":          # every label anywhere: boxes are the whole image
        GW, GH = 5, 4
        return rng.integers(0, GW * GH, (H, W)).astype(np.int32), GW, GH
    if kind == "big":                # one label almost everywhere, one single pixel, the others empty
        lab = np.full((H, W), 2, np.int32)
        lab[H // 2, W // 2] = 5
        return lab, 3, 3
    assert kind == "pixels"          # one pixel per label
    return np.arange(W * H, dtype=np.int32).reshape(H, W), W, H


@pytest.mark.parametrize("kind,W,H", [("grid", 97, 65), ("grid", 32, 32), ("grid", 31, 33), ("scattered", 40, 25),
                                      ("scattered", 130, 70), ("big", 64, 64), ("big", 65, 63), ("big", 129, 97),
                                      ("pixels", 33, 32), ("pixels", 1, 1)])
@pytest.mark.parametrize("fmt", list(DT))
def test_lists_and_statistics(lfd, kind, W, H, fmt):
    rng = np.random.default_rng(W * 1000 + H)
    lab, GW, GH = _labels(kind, W, H, rng)
    img = torch.from_numpy(rng.random((2, H, W, 4)))
    if fmt == "rgba8":
        v = (img * 255).to(torch.uint8)
    else:
        img[1] *= 3e3                # halves beyond the integer range of their fast sums
        v = img.to(DT[fmt])
    v, labels = v.cuda().contiguous(), torch.from_numpy(np.stack([lab, lab])).cuda()
    K = np.array([[50.0, 0, W / 2], [0, 50.0, H / 2], [0, 0, 1]])
    ctx = lfd.Context(0)
    ctx.set_input(v, labels, np.stack([K, K]), np.stack([np.eye(3)] * 2), np.array([[0.0, 0, 0], [-0.1, 0, 0]]), GW, GH,
                  dict(d_min=1.0, d_max=5.0, num_labels=4, alpha=0.3))
    ctx.synchronize()
    S = GW * GH
    y, x = np.mgrid[0:H, 0:W]
    for view in range(2):
        got = ctx.get_superpixels(view)
        order = np.argsort(lab.reshape(-1), kind="stable")
        cnt = np.bincount(lab.reshape(-1), minlength=S)
        assert np.array_equal(got["off"], np.concatenate([[0], np.cumsum(cnt)]))
        assert np.array_equal(got["pix"], order)
        col = v[view, ..., :3].double().cpu().numpy() / (255.0 if fmt == "rgba8" else 1.0)
        n = np.maximum(cnt, 1)
        want = [np.bincount(lab.reshape(-1), weights=w.reshape(-1), minlength=S) / n
                for w in (x.astype(float), y.astype(float), col[..., 0], col[..., 1], col[..., 2])]
        st = got["stats"].astype(np.float64)
        for k in range(5):           # FP64 sums rounded to FP32 once
            assert np.all(np.abs(st[:, k] - want[k]) <= 2.0 ** -23 * np.abs(want[k]) + 1e-12)
        assert np.array_equal(st[:, 6], cnt)
        stats = torch.full((S, 8), -1.0, device="cuda")
        lfd.superpixel_stats_noalloc(labels[view], v[view], GW, GH, 0.3, stats)
        torch.cuda.synchronize()
        keep = [0, 1, 2, 3, 4, 6, 7]     # slot 5: alpha's factor is FP64 here, FP32 in the view records
        assert np.array_equal(stats.cpu().numpy()[:, keep], got["stats"][:, keep])


@pytest.mark.parametrize("W,H,pitch", [(256, 256, 8), (264, 248, 8), (320, 240, 5), (40, 30, 30)])
def test_work_orders_of_one_and_several_tiles(lfd, W, H, pitch):
    # 1024 superpixels are one tile; the orders only permute the work, so the planes cannot depend on the bands
    lab, GW, GH = synth.grid_labels(W, H, pitch, True, seed=1)
    rig = synth.line_rig(2, 0.1, 0.9 * W, W, H)
    g = torch.Generator().manual_seed(1)
    v = torch.randint(0, 256, (2, H, W, 4), generator=g, dtype=torch.uint8).cuda()
    item = dict(views=v, labels=torch.from_numpy(np.stack([lab, lab])).cuda(), K=rig.K, R=rig.R, t=rig.t, GW=GW, GH=GH,
                params=dict(d_min=1.0, d_max=5.0, num_labels=16, iterations=2))
    out = []
    for opt in (dict(), dict(order_bands=1), dict(prop_persistent=0, sweep_persistent=0)):
        ctx = lfd.Context(0)
        planes, depth = ctx.estimate_batch([item], options=opt)
        ctx.synchronize()
        out.append((planes.clone(), depth[0].clone()))
    for p, d in out[1:]:
        assert torch.equal(p, out[0][0]) and torch.equal(d, out[0][1])
