"""SLIC takes its views in groups whose scratch is bounded; the groups do not
show in the labels or centres."""
import pytest
import torch

pytestmark = pytest.mark.gpu


def test_scratch_is_bounded_and_views_are_independent():
    from paper_1812_06856_gb300 import lfd
    H, W, n = 1024, 1024, 7          # a cell per pixel: 0.55 GB of scratch a view
    g = torch.Generator().manual_seed(5)
    v = torch.randint(0, 256, (n, H, W, 4), generator=g, dtype=torch.uint8).cuda()
    ctx = lfd.Context(0)
    ctx.slic(v[:1, :64, :64].contiguous(), 8, 8, iterations=1)
    torch.cuda.synchronize()
    before = torch.cuda.mem_get_info()[0] + torch.cuda.memory_reserved()
    many, cen = ctx.slic(v, W, H, iterations=1, want_centres=True)
    torch.cuda.synchronize()
    after = torch.cuda.mem_get_info()[0] + torch.cuda.memory_reserved()
    assert before - after <= (2 << 30) + (64 << 20)
    for k in (0, 2, 3, 6):           # the first and last views of groups
        one, c = ctx.slic(v[k:k + 1].contiguous(), W, H, iterations=1, want_centres=True)
        torch.cuda.synchronize()
        assert torch.equal(one[0], many[k]) and torch.equal(c[0], cen[k])
    ctx.close()
