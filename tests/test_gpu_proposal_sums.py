"""Proposal training over many rays: the decoder gradients are summed per ray first.

All rays of the batch are the same ray, so every ray contributes the same vector v, and a per-ray sum
followed by a sum over the rays only ever adds numbers of one sign to an entry.  An addition errs by at
most 2^-24 of the running sum, which is half the final one on average: K rays a warp err by K / 2 times
2^-24, relatively, the rows of warps and blocks likewise.  Twice that is allowed.  A single chain over all
bins of all rays has 32 times as many additions, and its bins' terms cancel.
"""
import numpy as np
import pytest
import torch

import oracle as oc
import paper_2206_14735_gb300 as gs
import scenegen as sg
from helpers import CUBE

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("precision", ["bf16", "fp32"])
def test_gradient_of_many_equal_rays(precision):
    per_warp, blocks = 512, 2 * torch.cuda.get_device_properties(0).multi_processor_count
    R = 4 * blocks * per_warp
    w = CUBE.with_(name="sums", precision=precision, n_strat=2, n_guided=0, prop_samples=2, prop_guided=0, rays=R,
                   n_smooth=0)
    ctx = gs.Context(w, max_smooth=1)
    rng = np.random.default_rng(7)
    theta = torch.from_numpy((sg.init_params(w) + rng.normal(0, 0.2, w.layout()[2])).astype(np.float32)).cuda()
    prop = torch.from_numpy(rng.normal(0, 0.3, oc.PROP_PARAMS).astype(np.float32)).cuda()
    grads = []
    for n in (1, R):
        b = gs.Batch.allocate(n, 2, 0, weights=True)
        b.origin.copy_(torch.tensor([-0.9, 0.2, 0.1], device="cuda").expand(n, 3))
        b.dir.copy_(torch.tensor([0.9, -0.1, 0.3], device="cuda").expand(n, 3))
        b.rgb.zero_(), b.depth.fill_(1.0), b.cls.zero_()
        b.t.copy_(torch.tensor([0.7, 1.3], device="cuda").expand(n, 2))
        b.w.copy_(torch.tensor([0.2, 0.7], device="cuda").expand(n, 2))
        grad, ce = torch.zeros(oc.PROP_PARAMS, device="cuda"), torch.zeros(2, device="cuda")
        ctx.proposal_backward(theta, prop, b, grad, ce)
        ctx.sync_status()
        assert int(ce[1]) == n
        grads.append(grad.cpu().numpy().astype(np.float64))
    one, all_ = grads
    bound = (per_warp / 2 + 4 + blocks / 2) * 2.0 ** -23
    err = np.abs(all_ - one) / np.maximum(np.abs(one), 1e-30)
    assert np.abs(one).max() > 1e-3
    assert err.max() <= bound, (err.max(), bound, int(err.argmax()))
