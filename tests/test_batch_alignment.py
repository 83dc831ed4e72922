"""batch->dz is written as 16-byte vectors: a pointer that does not allow it is refused on the host."""
import ctypes

import pytest

import paper_2206_14735_gb300 as gs
import scenegen as sg
from paper_2206_14735_gb300 import _lib
from paper_2206_14735_gb300 import build as gbuild

GS_ERR_ALIGN = 3


def test_noalloc_refuses_a_misaligned_dz_before_it_needs_a_device():
    """No GPU is touched: the pointers are never followed (made up here), and a call that passed the
    argument checks would report the missing device instead."""
    gbuild.build()
    L = _lib.lib()
    cfg = gs.make_config(sg.WORKLOADS["cube-1024x64"])
    b = gs.GsBatch(8, cfg.n_strat + cfg.n_guided, 0, *([0x1000] * 7), None, None, None, 0x1000, None, 0x1004, None)
    p = ctypes.c_void_p(0x1000)
    assert L.gs_forward_backward_noalloc(ctypes.byref(cfg), p, ctypes.byref(b), None, p, p, None) == GS_ERR_ALIGN
    assert b"dz" in L.gs_last_error(None)


@pytest.mark.gpu
@pytest.mark.parametrize("arch", ["compact", "paper"])
def test_backward_passes_refuse_a_misaligned_dz(arch):
    import torch

    w = sg.WORKLOADS["cube-1024x64"].with_(name="align", rays=8, n_smooth=0, arch=arch)
    fr = sg.make_frames(w)
    ctx = gs.Context(w, max_smooth=1)
    b = gs.Batch.allocate(8, w.n_samples, 0)
    ctx.sample_rays(gs.DeviceFrames(fr.rgb, fr.depth, fr.c2w, fr.fx, fr.fy, fr.cx, fr.cy), 1, 1, b)
    width = 32 if arch == "paper" else 16
    b.dz = torch.zeros(8 * w.n_samples * width + 4, device="cuda")[1:]
    theta = torch.from_numpy(sg.init_params(w)).cuda()
    loss, grad = torch.zeros(6, device="cuda"), torch.zeros_like(theta)
    with pytest.raises(gs.GoSurfError, match="dz"):
        ctx.forward_backward(theta, b, None, loss, grad)
    with pytest.raises(gs.GoSurfError, match="dz"):
        ctx.backward(theta, b, None, grad)
    torch.cuda.synchronize()
    assert float(grad.abs().max()) == 0.0
