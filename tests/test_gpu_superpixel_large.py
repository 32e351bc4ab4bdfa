"""Superpixel lists and statistics where superpixels are large and few, so that a
CTA takes from one to seven of them."""
import numpy as np
import pytest
import torch

from paper_1812_06856_gb300 import synth

pytestmark = pytest.mark.gpu


def _per_cta(S, px):
    return 8 if px < 2500 * S else max(1, min(8, -(-S // (152 * 8))))


# (W, H, pitch or None: 24 labels scattered over the image, superpixels per CTA for two views and for one)
@pytest.mark.parametrize("W,H,pitch,per", [(320, 240, None, (1, 1)), (301, 203, 70, (1, 1)), (1600, 1200, 52, (2, 1)),
                                           (2561, 2049, 51, (4, 2))])
def test_lists_and_statistics_of_large_superpixels(W, H, pitch, per):
    from paper_1812_06856_gb300 import lfd
    rng = np.random.default_rng(W)
    if pitch is None:
        GW, GH = 6, 4
        lab = rng.integers(0, GW * GH, (H, W)).astype(np.int32)
    else:
        m, GW, GH = synth.grid_labels_fast(W, H, pitch, True, seed=2, device="cuda")
        lab = m.cpu().numpy()
    S = GW * GH
    assert (_per_cta(2 * S, 2 * W * H), _per_cta(S, W * H)) == per
    v = torch.from_numpy(rng.integers(0, 256, (2, H, W, 4)).astype(np.uint8)).cuda()
    labels = torch.from_numpy(np.stack([lab, lab])).cuda()
    K = np.array([[500.0, 0, W / 2], [0, 500.0, H / 2], [0, 0, 1]])
    ctx = lfd.Context(0)
    ctx.set_input(v, labels, np.stack([K, K]), np.stack([np.eye(3)] * 2), np.array([[0.0, 0, 0], [-0.1, 0, 0]]), GW, GH,
                  dict(d_min=1.0, d_max=5.0, num_labels=4, alpha=0.3))
    ctx.synchronize()
    flat = lab.reshape(-1)
    cnt = np.bincount(flat, minlength=S)
    n = np.maximum(cnt, 1)
    y, x = np.divmod(np.arange(W * H), W)
    for view in range(2):
        got = ctx.get_superpixels(view)
        assert np.array_equal(got["pix"], np.argsort(flat, kind="stable"))
        col = v[view, ..., :3].reshape(-1, 3).cpu().numpy().astype(np.float64)
        want = [np.bincount(flat, weights=w, minlength=S) / n for w in (x, y, col[:, 0] / 255, col[:, 1] / 255,
                                                                        col[:, 2] / 255)]
        st = got["stats"].astype(np.float64)
        for k in range(5):           # exact or FP64 sums rounded to FP32 once
            assert np.all(np.abs(st[:, k] - want[k]) <= 2.0 ** -23 * np.abs(want[k]) + 1e-12)
        stats = torch.full((S, 8), -1.0, device="cuda")
        lfd.superpixel_stats_noalloc(labels[view], v[view], GW, GH, 0.3, stats)
        torch.cuda.synchronize()
        keep = [0, 1, 2, 3, 4, 6, 7]
        assert np.array_equal(stats.cpu().numpy()[:, keep], got["stats"][:, keep])
    ctx.close()
