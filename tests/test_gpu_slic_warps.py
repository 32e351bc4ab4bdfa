"""SLIC gives a view the same labels and centres with one and with several
warps per cell: shapes whose cells a single view splits between warps and a
batch does not."""
import pytest
import torch

pytestmark = pytest.mark.gpu


def _warps_per_cell(W, H, GW, GH, n):
    """The launch's rule: more warps for few or large cells while each keeps a step of 128 pixels."""
    stride = -(-(-(-W // GW) * -(-H // GH)) // 4) * 4
    wpc = 1
    while wpc < 8 and stride > 128 * wpc and (stride > 1024 * wpc or GW * GH * n * wpc < 152 * 32):
        wpc *= 2
    return wpc


@pytest.mark.parametrize("W,H,GW,GH,warps", [(476, 420, 34, 30, (2, 1)), (601, 597, 20, 20, (8, 1)),
                                             (487, 503, 25, 26, (4, 1)), (700, 350, 14, 7, (8, 4))])
@pytest.mark.parametrize("dtype", [torch.uint8, torch.float16])
def test_warps_per_cell_do_not_change_the_result(W, H, GW, GH, warps, dtype):
    from paper_1812_06856_gb300 import lfd
    n = 16
    assert (_warps_per_cell(W, H, GW, GH, 1), _warps_per_cell(W, H, GW, GH, n)) == warps
    g = torch.Generator().manual_seed(7)
    img = torch.rand((n, H // 5 + 1, W // 5 + 1, 4), generator=g).repeat_interleave(5, 1).repeat_interleave(5, 2)[:, :H, :W]
    img = (img + 0.1 * torch.rand((n, H, W, 4), generator=g)).clamp(0, 1)
    v = ((img * 255).to(torch.uint8) if dtype == torch.uint8 else img.to(dtype)).cuda().contiguous()
    ctx = lfd.Context(0)
    many, cens = ctx.slic(v, GW, GH, iterations=4, want_centres=True)
    for k in (0, 7, 15):
        one, cen = ctx.slic(v[k:k + 1].contiguous(), GW, GH, iterations=4, want_centres=True)
        torch.cuda.synchronize()
        assert torch.equal(one[0], many[k]) and torch.equal(cen[0], cens[k])
    ctx.close()
