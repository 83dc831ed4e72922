"""Every form of the render kernels at sample and ray counts that fill no chunk and no tile.

A ray whose depths are continued with copies of its last one renders the same: two equal SDF values give
no opacity, and the copies belong to no loss term.  So a batch of N samples a ray and the same batch
filled up to whole chunks of 32 have the same losses, outputs and gradients up to the order of the
sums, in each precision and architecture, without a reference of the other's rounding."""
import numpy as np
import pytest
import torch

import paper_2206_14735_gb300 as gs
import scenegen as sg
from gpu_common import GRAD_TOL, LOSS_RTOL, Problem
from helpers import CUBE, paper_parity_params, sdf_parity_params

pytestmark = pytest.mark.gpu

FORMS = {"fp32": {}, "bf16": dict(precision="bf16"), "paper": dict(arch="paper")}


def _workload(form, rays, n):
    return CUBE.with_(name=f"forms-{form}", rays=rays, n_strat=n - n // 3, n_guided=n // 3, n_smooth=0, **FORMS[form])


def _params(form, w, p):
    theta = (paper_parity_params if form == "paper" else sdf_parity_params)(w, sg.cube_scene(), seed=21)
    th = torch.from_numpy(theta).cuda()
    return th, th[:p.n_grid].to(torch.bfloat16).view(torch.int16).contiguous() if form == "bf16" else None


def _padded(b, n):
    q = gs.Batch.allocate(b.R, n, 0, weights=True)
    for k in ("pix", "origin", "dir", "rgb", "depth", "counts"):
        getattr(q, k).copy_(getattr(b, k))
    q.t.copy_(torch.cat([b.t, b.t[:, -1:].expand(-1, n - b.N)], 1))
    q.cls.zero_()
    q.cls[:, :b.N] = b.cls
    return q


def _outputs(ctx, th, mirror, b, split):
    out = dict(loss=torch.empty(6, device="cuda"), grad=torch.zeros_like(th), rgb=torch.zeros(b.R, 3, device="cuda"),
               d=torch.zeros(b.R, device="cuda"), wsum=torch.zeros(b.R, device="cuda"))
    if split:
        ctx.forward(th, b, out["loss"], out["rgb"], out["d"], out["wsum"], theta_bf16=mirror)
        ctx.backward(th, b, None, out["grad"], theta_bf16=mirror)
    else:
        ctx.forward_backward(th, b, None, out["loss"], out["grad"], theta_bf16=mirror)
    ctx.sync_status()
    return {k: v.cpu().numpy().astype(np.float64) for k, v in out.items()} | {"w": b.w.cpu().numpy()}


@pytest.mark.parametrize("form", FORMS)
@pytest.mark.parametrize("rays,n", [(1, 2), (5, 31), (4, 33), (7, 65), (9, 99), (301, 131)])
def test_ragged_rays_render_as_whole_chunks(form, rays, n):
    w = _workload(form, rays, n)
    full = _workload(form, rays, (n + 31) // 32 * 32)
    p = Problem(w)
    th, mirror = _params(form, w, p)
    b = p.gpu_sample(3, 5)
    b.w = torch.zeros_like(b.t)
    for store in (False, True):
        ctx, ctx_full = (gs.Context(x, max_smooth=1, store_activations=store) for x in (w, full))
        for split in (True, False):
            got = _outputs(ctx, th, mirror, b, split)
            ref = _outputs(ctx_full, th, mirror, _padded(b, full.n_samples), split)
            np.testing.assert_allclose(got["loss"], ref["loss"], rtol=LOSS_RTOL, atol=1e-9)
            np.testing.assert_allclose(got["w"], ref["w"][:, :n], rtol=0, atol=2e-6)
            np.testing.assert_allclose(got["rgb"], ref["rgb"], rtol=0, atol=2e-6)
            np.testing.assert_allclose(got["d"], ref["d"], rtol=0, atol=2e-5)
            np.testing.assert_allclose(got["wsum"], ref["wsum"], rtol=0, atol=2e-6)
            A, B = p.split_grad(got["grad"]), p.split_grad(ref["grad"])
            for k in A:
                assert np.abs(A[k] - B[k]).max() <= GRAD_TOL * np.abs(B[k]).max() + 1e-12, (store, split, k)


@pytest.mark.parametrize("form", FORMS)
@pytest.mark.parametrize("n", [5, 33])
def test_forward_of_more_rays_than_one_round(form, n):
    """Each tile group of the forward-only kernel takes several ray-quads here; in pieces of 1200 rays
    it takes at most one, and from two chunks on the compact kernel has two groups for three then.  A
    ray's outputs are the same bits."""
    R, piece = 8 * 4 * torch.cuda.get_device_properties(0).multi_processor_count + 3, 1200
    w = _workload(form, R, n)
    p = Problem(w)
    th, mirror = _params(form, w, p)
    b = p.gpu_sample(3, 5)
    loss = torch.empty(6, device="cuda")

    def outputs(batch):
        o = torch.zeros(batch.R, 3, device="cuda"), torch.zeros(batch.R, device="cuda"), torch.zeros(batch.R, device="cuda")
        p.ctx.forward(th, batch, loss, *o, theta_bf16=mirror)
        p.ctx.sync_status()
        return [x.clone() for x in o]

    whole = outputs(b)
    for i in range(0, R, piece):
        m = min(piece, R - i)
        q = gs.Batch.allocate(m, n, 0)
        for k in ("pix", "origin", "dir", "rgb", "depth", "t", "cls"):
            getattr(q, k).copy_(getattr(b, k)[i:i + m])
        q.counts.copy_(b.counts)
        for x, y in zip(outputs(q), whole):
            assert torch.equal(x, y[i:i + m])
