"""Plane, choice and energy buffers that a kernel cannot take word by word (an
odd byte offset, pinned host memory) are copied all the same."""
import ctypes as C

import numpy as np
import pytest
import torch

from paper_1812_06856_gb300 import synth
import parity as PT

pytestmark = pytest.mark.gpu


def _shifted(nbytes, offset, where):
    buf = torch.zeros(nbytes + 16, dtype=torch.uint8, device="cuda") if where == "device" else \
        torch.zeros(nbytes + 16, dtype=torch.uint8).pin_memory()
    return buf[offset:offset + nbytes]


@pytest.mark.parametrize("offset,where", [(0, "device"), (4, "device"), (1, "device"), (2, "device"), (0, "host"),
                                          (4, "host")])
def test_iterate_takes_any_buffer_the_copies_take(offset, where):
    from paper_1812_06856_gb300 import lfd
    lf = synth.make_config(1, scale=0.25)
    v, labels, _ = PT.gpu_inputs(lf, "rgba8")
    ctx = lfd.Context(0)
    ctx.set_input(v, labels, lf.rig.K, lf.rig.R, lf.rig.t, lf.GW, lf.GH, synth.method_params(lf, num_labels=32))
    planes, _, _ = ctx.plane_sweep()
    want, choice, energy = ctx.iterate(1, planes, want_choice=True)
    ctx.synchronize()
    S, V = lf.GW * lf.GH, lf.rig.V
    bufs = {k: _shifted(V * S * b, offset, where) for k, b in (("in", 16), ("out", 16), ("choice", 8), ("energy", 8))}
    bufs["in"].copy_(planes.contiguous().view(torch.uint8).reshape(-1))
    torch.cuda.synchronize()
    ptrs = {k: (C.c_void_p * V)(*[bufs[k].data_ptr() + u * S * b for u in range(V)])
            for k, b in (("in", 16), ("out", 16), ("choice", 8), ("energy", 8))}
    assert ctx.lib.lfd_iterate(ctx.h, 1, ptrs["in"], ptrs["out"], ptrs["choice"], ptrs["energy"], None) == 0
    ctx.synchronize()
    for k, w in (("out", want), ("choice", choice), ("energy", energy)):
        assert np.array_equal(bufs[k].cpu().numpy(), w.contiguous().view(torch.uint8).reshape(-1).cpu().numpy()), k
    ctx.close()
