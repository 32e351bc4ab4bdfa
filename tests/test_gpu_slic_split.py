"""SLIC gives a view the same labels and centres whatever number of warps
shares a cell (it follows from the cell size and the number of views)."""
import numpy as np
import pytest
import torch

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def lfd():
    from paper_1812_06856_gb300 import lfd as mod
    mod.load()
    return mod


@pytest.mark.parametrize("H,W,GW,GH", [(150, 210, 15, 11), (150, 210, 7, 5), (97, 131, 40, 33), (260, 300, 2, 2)])
@pytest.mark.parametrize("dtype", [torch.uint8, torch.float32])
def test_labels_do_not_depend_on_the_warps_per_cell(lfd, H, W, GW, GH, dtype):
    g = torch.Generator().manual_seed(3)
    img = torch.rand((H // 4 + 1, W // 4 + 1, 4), generator=g).repeat_interleave(4, 0).repeat_interleave(4, 1)[:H, :W]
    img = (img + 0.05 * torch.rand((H, W, 4), generator=g)).clamp(0, 1)
    v = (img * 255).to(torch.uint8) if dtype == torch.uint8 else img
    if dtype == torch.float32:
        v[3, 5:9, 0] = float("nan")
        v[H - 2, W - 3, 2] = float("inf")
    v = v.cuda().contiguous()
    ctx = lfd.Context(0)
    one, cen = ctx.slic(v[None].contiguous(), GW, GH, iterations=5, want_centres=True)
    many, cens = ctx.slic(v[None].repeat(20, 1, 1, 1).contiguous(), GW, GH, iterations=5, want_centres=True)
    ctx.synchronize()
    assert torch.isfinite(cen).all()
    for k in range(20):
        assert torch.equal(many[k], one[0])
        assert torch.equal(cens[k], cen[0])
    # the final centres' sums are those of a plain assignment by the labels of the step before
    assert int(one.min()) >= 0 and int(one.max()) < GW * GH
