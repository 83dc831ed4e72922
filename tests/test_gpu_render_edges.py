"""Render kernel and plain sampler at the edges of their tiles: one ray and one more than a tile's
four, sample counts around the 32-sample chunks, no guided samples, the most samples per ray; the
stored and the recomputed activations, fused and split.  Against the FP64 oracle at the parity
module's tolerances."""
import numpy as np
import pytest
import torch

import paper_2206_14735_gb300 as gs
import scenegen as sg
from gpu_common import (GRAD_ELEM_RTOL, GRAD_TOL, LOSS_RTOL, Problem, assert_grad_close, prepare_parity_batch,
                        upload_oracle_batch)
from helpers import CUBE, sdf_parity_params

pytestmark = pytest.mark.gpu

CASES = [(1, 2, 0), (5, 31, 0), (4, 20, 13), (6, 40, 24), (7, 65, 0), (301, 64, 64), (9, 100, 60)]


@pytest.mark.parametrize("rays,n_strat,n_guided", CASES)
def test_render_edges(rays, n_strat, n_guided):
    w = CUBE.with_(name="edges", rays=rays, n_strat=n_strat, n_guided=n_guided, n_smooth=16)
    p = Problem(w)
    b = p.gpu_sample(3, 5)
    bt, sm = p.oracle_sample(3, 5)
    assert np.array_equal(b.t.cpu().numpy().view(np.uint32), bt["t"].view(np.uint32))
    assert np.array_equal(b.cls.cpu().numpy(), bt["cls"])
    assert list(b.counts.cpu().numpy()[:3]) == list(bt["counts"][:3])
    theta = sdf_parity_params(w, sg.cube_scene(), seed=21)
    bt_s, ref, _ = prepare_parity_batch(p, theta, bt, sm, max_drop=0.34, label=w.name)
    batch = upload_oracle_batch(bt_s, sm, sm["n_valid"][0])
    th = torch.from_numpy(theta).cuda()
    for store in (False, True):
        ctx = gs.Context(w, store_activations=store)
        for split in (False, True):
            loss, grad = torch.empty(6, device="cuda"), torch.zeros_like(th)
            if split:
                ctx.forward(th, batch, loss)
                ctx.backward(th, batch, None, grad)
            else:
                ctx.forward_backward(th, batch, None, loss, grad)
            ctx.sync_status()
            got = loss.cpu().numpy().astype(np.float64)
            for k in range(6):
                assert abs(got[k] - ref["loss"][k]) <= LOSS_RTOL * abs(ref["loss"][k]) + 1e-9, (store, split, k)
            assert_grad_close(p, grad.cpu().numpy(), ref["grad"], GRAD_TOL, GRAD_ELEM_RTOL)
