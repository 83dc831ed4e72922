"""The work a user of this framework has it do, as cases that can be timed and compared.

A case is one call, or the few calls of one optimisation step, through the Python entry points
(``Context``, ``GoSurfStep``, ``SdfGrad``) on data a training run has in hand: posed RGB-D
frames of a room or a cube, a feature grid that carries the scene's SDF in one feature and
O(0.1) values elsewhere, decoders whose hidden units switch from sample to sample, and ray
batches drawn as the method draws them.  Everything is made on the GPU from the seed alone.

``exact`` restates each path in 64 bits with plain torch (no code of this repository).
"""
from __future__ import annotations

import math
from types import SimpleNamespace

import numpy as np
import torch

import paper_2206_14735_gb300 as gs

DEV = "cuda"
F64 = torch.float64

# the two scenes of the repository's workloads: extents, voxel edges (coarse to fine), camera
SCENES = {
    "room": dict(lo=(0.0, 0.0, 0.0), hi=(8.0, 6.0, 3.0), voxels=(0.96, 0.24, 0.06, 0.02), near=0.1, far=6.0,
                 frames=40, height=480, width=640, f=525.0),
    "cube": dict(lo=(-1.28, -1.28, -1.28), hi=(1.28, 1.28, 1.28), voxels=(0.64, 0.32, 0.16, 0.08), near=0.1, far=4.0,
                 frames=1, height=120, width=160, f=130.0),
}
LAMBDAS = (10.0, 1.0, 10.0, 1.0, 1.0)
TRUNC, GUIDE, KAPPA_FS, DELTA_S = 0.10, 0.10, 5.0, 0.004

_RENDER = dict(scene="room", arch="compact", precision="fp32", store=True, rays=8192, strat=64, guided=32, points=4096)


def listed():
    return [
        # a whole training step of the smallest scene: sampling, fused forward + backward, with
        # the activations recomputed (the context's default)
        dict(_RENDER, name="step-cube-1024x64", kind="step", scene="cube", store=False, rays=1024, strat=48, guided=16),
        # a small odd batch (the last rays of a pass, a preview): latency counts
        dict(_RENDER, name="grad-cube-333x33", kind="grad", scene="cube", store=False, rays=333, strat=22, guided=11,
             points=37),
        # the default training batch: losses and gradients in one pass, stored activations
        dict(_RENDER, name="grad-room-8192x96", kind="grad"),
        # the step as a differentiable function of the parameters, large batch (the largest case)
        dict(_RENDER, name="autograd-room-65536x96", kind="autograd", rays=65536),
        # the BF16 form: gathers from the bfloat16 copy, bfloat16 decoders
        dict(_RENDER, name="grad-room-bf16-32768x96", kind="grad", precision="bf16", rays=32768),
        # the paper's architecture: colour grid, view direction, two hidden layers in each decoder
        dict(_RENDER, name="grad-paper-8192x96", kind="grad", arch="paper"),
        # the paper's whole method in one step: importance sampler, Eikonal term, poses
        dict(_RENDER, name="method-room-8192x132", kind="method", arch="paper", coarse=96, steps=3, per_step=12),
        # rendering held-out rays with the importance sampler's sample count: forward only
        dict(_RENDER, name="eval-room-8192x132", kind="eval", strat=96, guided=36, points=0, store=False),
        # the learned proposal: sampling from it and its own training step (BF16 network)
        dict(_RENDER, name="proposal-bf16-65536x32", kind="proposal", precision="bf16", rays=65536, prop=32,
             prop_guided=24, points=0, store=False),
        # SDF and its gradient at points, and the double backward to the parameters
        dict(name="query-room-4096", kind="query", scene="room", arch="compact", points=4096),
        # mesh extraction of the whole room (2 cm lattice): 18 M SDF values and the isosurface
        dict(name="mesh-room-2cm", kind="mesh", scene="room", arch="compact", step=0.02),
        # the dense optimiser update of every grid and decoder parameter
        dict(name="adam-room", kind="adam", scene="room", arch="compact", mirror=False),
    ]


def draw(rng):
    """One more case of the same ranges; no costlier than the largest listed one."""

    def log_int(lo, hi):
        return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))

    kind = rng.choice(["step", "grad", "grad", "grad", "grad", "autograd", "method", "eval", "proposal", "query",
                       "mesh"])
    if kind == "query":
        return dict(kind=kind, scene=rng.choice(["room", "cube"]), arch=rng.choice(["compact", "paper"]),
                    points=log_int(100, 300000))
    if kind == "mesh":
        scene = rng.choice(["room", "cube"])
        return dict(kind=kind, scene=scene, arch="compact",
                    step=rng.uniform(0.02, 0.1) if scene == "room" else rng.uniform(0.008, 0.08))
    c = dict(_RENDER, kind=kind, scene=rng.choice(["room", "room", "cube"]), store=rng.random() < 0.6)
    n = rng.randint(12, 132)
    c["guided"] = int(n * rng.uniform(0.15, 0.5))
    c["strat"] = n - c["guided"]
    c["points"] = log_int(30, 4096)
    c["rays"] = log_int(60, 50000 if n <= 96 else 30000)
    if kind == "proposal":
        c.update(precision=rng.choice(["bf16", "fp32"]), prop=rng.randint(12, 32), points=0, store=False)
        c["prop_guided"] = rng.randint(0, c["prop"] // 2)
        c["strat"], c["guided"] = 64, 32
        c["rays"] = log_int(100, 40000)
    elif kind == "method":
        c.update(arch=rng.choice(["paper", "compact"]), coarse=rng.randint(32, 112), steps=rng.randint(1, 3),
                 per_step=rng.randint(4, 12), rays=log_int(60, 9000))
    elif kind == "eval":
        c.update(points=0, store=False, arch=rng.choice(["compact", "paper"]))
        c["rays"] = min(c["rays"], 20000)
    else:
        form = rng.choice(["fp32", "fp32", "bf16", "paper"])
        if form == "bf16":
            c["precision"] = "bf16"
        elif form == "paper":
            c["arch"] = "paper"
            c["rays"] = min(c["rays"], 16000)
    return c


# ---- scene, frames and parameters ----------------------------------------------------------


def _generator(seed):
    g = torch.Generator(device=DEV)
    g.manual_seed(int(seed) * 2654435761 % (1 << 62) + 17)
    return g


def _workload(c):
    """The attributes gs.Context reads of a workload, and the grid's layout."""
    s = SCENES[c["scene"]]
    w = SimpleNamespace(**s)
    w.extent_min = s["lo"]
    w.dims = [tuple(int(math.ceil((h - l) / v - 1e-6)) + 1 for l, h in zip(s["lo"], s["hi"])) for v in s["voxels"]]
    w.rays, w.n_smooth = c.get("rays", 1), c.get("points", 0) if c["kind"] not in ("query", "mesh") else 0
    w.n_strat, w.n_guided = c.get("strat", 64), c.get("guided", 32)
    w.guide_half, w.trunc, w.kappa_fs, w.lambdas, w.delta_s = GUIDE, TRUNC, KAPPA_FS, LAMBDAS, DELTA_S
    w.precision, w.arch = c.get("precision", "fp32"), c.get("arch", "compact")
    w.prop_samples, w.prop_guided = c.get("prop", 0), c.get("prop_guided", 0)
    w.imp_coarse, w.imp_steps, w.imp_per_step = c.get("coarse", 0), c.get("steps", 0), c.get("per_step", 0)
    if c["kind"] != "method":
        w.imp_coarse = 0
    w.N = w.imp_coarse + w.imp_steps * w.imp_per_step if w.imp_coarse else w.n_strat + w.n_guided
    w.counts = [d[0] * d[1] * d[2] for d in w.dims]
    w.offs = [4 * sum(w.counts[:l]) for l in range(4)]
    w.n_geo = 4 * sum(w.counts)
    w.n_grid = w.n_geo + ((6 * w.counts[3] + 3) // 4 * 4 if w.arch == "paper" else 0)
    w.shapes = ([("gW1", (32, 16)), ("gb1", (32,)), ("gW2", (32, 32)), ("gb2", (32,)), ("gw3", (1, 32)), ("gb3", (1,)),
                 ("cW1", (32, 9)), ("cb1", (32,)), ("cW2", (32, 32)), ("cb2", (32,)), ("cW3", (3, 32)), ("cb3", (3,)),
                 ("kappa", (1,))] if w.arch == "paper" else
                [("W1", (32, 16)), ("b1", (32,)), ("W2", (16, 32)), ("b2", (16,)), ("W3", (32, 15)), ("b3", (32,)),
                 ("W4", (3, 32)), ("b4", (3,)), ("kappa", (1,))])
    w.n = w.n_grid + sum(math.prod(s) for _, s in w.shapes)
    w.n_pad = (w.n + 3) // 4 * 4  # the optimiser works on whole vectors of four
    return w


def _primitives(c, rng):
    """Spheres (centre, radius) and boxes (centre, half extents) standing in the scene."""
    if c["scene"] == "cube":
        return [((-0.4, 0.0, 0.0), 0.5 + rng.uniform(-0.03, 0.03))], [((0.55, 0.0, 0.0), (0.3, 0.3, 0.3))]
    sph, box = [], []
    for _ in range(8):
        r = rng.uniform(0.15, 0.5)
        a, k = rng.uniform(0, 2 * math.pi), rng.uniform(0.0, 0.4)
        sph.append(((4 + 3 * k * math.cos(a), 3 + 2 * k * math.sin(a), r), r))
    for _ in range(10):
        h = tuple(rng.uniform(0.1, 0.6) for _ in range(3))
        x = rng.choice([h[0], 8 - h[0]])
        box.append(((x, rng.uniform(h[1], 6 - h[1]), h[2]), h))
    return sph, box


def _sdf(c, prims, x):
    """Signed distance of the scene at x [..., 3]."""
    sph, box = prims
    d = None
    if c["scene"] == "room":
        lo, hi = (torch.tensor(SCENES["room"][k], device=x.device, dtype=x.dtype) for k in ("lo", "hi"))
        d = torch.minimum(x - lo, hi - x).amin(-1)
    for o, r in sph:
        e = (x - torch.tensor(o, device=x.device, dtype=x.dtype)).norm(dim=-1) - r
        d = e if d is None else torch.minimum(d, e)
    for o, h in box:
        q = (x - torch.tensor(o, device=x.device, dtype=x.dtype)).abs() - torch.tensor(h, device=x.device, dtype=x.dtype)
        d = torch.minimum(d, q.clamp(min=0).norm(dim=-1) + q.amax(-1).clamp(max=0))
    return d


def _hit(c, prims, o, r):
    """First hit along o + t r (0 where nothing is hit)."""
    inf = torch.full(r.shape[:-1], math.inf, device=r.device)
    t = inf
    inv = 1.0 / torch.where(r.abs() < 1e-9, torch.full_like(r, 1e-9), r)
    if c["scene"] == "room":
        lo, hi = (torch.tensor(SCENES["room"][k], device=r.device) for k in ("lo", "hi"))
        t = torch.maximum((lo - o) * inv, (hi - o) * inv).amin(-1)
    for p, rad in prims[0]:
        d = o - torch.tensor(p, device=r.device)
        a, b, q = (r * r).sum(-1), (d * r).sum(-1), (d * d).sum(-1) - rad * rad
        disc = b * b - a * q
        s = (-b - disc.clamp(min=0).sqrt()) / a
        t = torch.where((disc > 0) & (s > 0), torch.minimum(t, s), t)
    for p, h in prims[1]:
        d, hh = o - torch.tensor(p, device=r.device), torch.tensor(h, device=r.device)
        t0, t1 = torch.minimum((-hh - d) * inv, (hh - d) * inv).amax(-1), torch.maximum((-hh - d) * inv, (hh - d) * inv).amin(-1)
        t = torch.where((t1 > t0) & (t0 > 0), torch.minimum(t, t0), t)
    return torch.where(torch.isfinite(t), t, torch.zeros_like(t))


def _poses(c, w, rng):
    out = []
    ph = rng.uniform(0, 2 * math.pi)
    for k in range(w.frames):
        if c["scene"] == "cube":
            v = np.array([rng.gauss(0, 1) for _ in range(3)])
            p, tgt = 1.1 * v / np.linalg.norm(v), np.zeros(3)
        else:
            a = 2 * math.pi * k / w.frames + ph
            p = np.array([4 + 3 * math.cos(a), 3 + 2 * math.sin(a), 1.55 + 0.15 * math.sin(3 * a)])
            tgt = np.array([4 + 1.2 * math.cos(2 * a), 3 + 0.8 * math.sin(2 * a), 0.8 + 0.2 * math.sin(a)])
        fwd = (tgt - p) / np.linalg.norm(tgt - p)
        right = np.cross(fwd, (0.0, 0.0, 1.0) if abs(fwd[2]) < 0.95 else (0.0, 1.0, 0.0))
        right /= np.linalg.norm(right)
        out.append(np.concatenate([np.stack([right, np.cross(fwd, right), fwd], 1), p[:, None]], 1))
    return torch.tensor(np.stack(out), device=DEV, dtype=torch.float32)


def _frames(c, w, prims, rng, g):
    """Posed colour and depth images: exact hits, 1 mm z^2 noise, 5 % of the depths missing."""
    c2w = _poses(c, w, rng)
    v, u = torch.meshgrid(torch.arange(w.height, device=DEV) + 0.5, torch.arange(w.width, device=DEV) + 0.5,
                          indexing="ij")
    d = torch.stack([(u - w.width / 2) / w.f, (v - w.height / 2) / w.f, torch.ones_like(u)], -1)
    depth = torch.empty(w.frames, w.height, w.width, device=DEV)
    rgb = torch.empty(w.frames, w.height, w.width, 3, device=DEV, dtype=torch.uint8)
    k = torch.tensor([3.0, 5.0, 7.0], device=DEV)
    for i in range(w.frames):
        r, o = d @ c2w[i, :, :3].T, c2w[i, :, 3]
        t = _hit(c, prims, o, r)
        x = o + t[..., None] * r
        rgb[i] = ((0.5 + 0.5 * torch.sin(k * x + torch.tensor([0.0, 1.0, 2.0], device=DEV))) * 255).to(torch.uint8)
        noise = 0.001 * t * t * torch.randn(t.shape, device=DEV, generator=g)
        keep = torch.rand(t.shape, device=DEV, generator=g) >= 0.05
        depth[i] = torch.where(keep & (t > 0), t + noise, torch.zeros_like(t))
    return rgb, depth, c2w


def _theta(c, w, prims, g):
    """Parameters of a scene in training: the SDF (3 cm off) in feature 0 of the finest level through
    pass-through units, features and the other units' weights at random, biases near zero."""
    th = torch.zeros(w.n_pad, device=DEV)
    th[:w.n_grid].normal_(0.0, 0.1, generator=g)
    if w.arch == "paper":
        th[w.n_geo + 6 * w.counts[3]:w.n_grid] = 0.0
    nx, ny, nz = w.dims[3]
    ax = [torch.arange(n, device=DEV) * w.voxels[3] + w.lo[k] for k, n in enumerate((nx, ny, nz))]
    lev = th[w.offs[3]:w.offs[3] + 4 * w.counts[3]].view(nz, ny, nx, 4)
    for z0 in range(0, nz, 16):
        zz, yy, xx = torch.meshgrid(ax[2][z0:z0 + 16], ax[1], ax[0], indexing="ij")
        lev[z0:z0 + 16, ..., 0] = _sdf(c, prims, torch.stack([xx, yy, zz], -1))
    m = _decoder(th, w)

    def uni(t, a):
        t.copy_((torch.rand(t.shape, device=DEV, generator=g) * 2 - 1) * a)

    if w.arch == "paper":
        uni(m["gW1"], 0.25), uni(m["gb1"], 0.02), uni(m["gW2"], 0.3), uni(m["gb2"], 0.004), uni(m["gw3"], 0.1)
        m["gW1"][:, 12] = 0.0
        m["gW1"][:2] = 0.0
        m["gW1"][0, 12], m["gW1"][1, 12] = 1.0, -1.0
        m["gb1"][:2] = 0.0
        m["gW2"][:, :2] = 0.0
        m["gW2"][:2] = 0.0
        m["gW2"][0, 0], m["gW2"][0, 1], m["gW2"][1, 0], m["gW2"][1, 1] = 1.0, -1.0, -1.0, 1.0
        m["gb2"][:2] = 0.0
        m["gw3"][0, 0], m["gw3"][0, 1] = 1.0, -1.0
        m["gb3"][0] = 0.03
        uni(m["cW1"], 0.5), uni(m["cb1"], 0.02), uni(m["cW2"], 0.3), uni(m["cb2"], 0.004), uni(m["cW3"], 1.0)
        uni(m["cb3"], 0.2)
    else:
        uni(m["W1"], 0.25), uni(m["b1"], 0.02), uni(m["W2"], 0.25), uni(m["b2"], 0.02), uni(m["W3"], 0.25)
        uni(m["b3"], 0.004), uni(m["W4"], 1.0), uni(m["b4"], 0.2)
        m["W1"][:, 12] = 0.0
        m["W1"][:2] = 0.0
        m["W1"][0, 12], m["W1"][1, 12] = 1.0, -1.0
        m["b1"][:2] = 0.0
        m["W2"][0] *= 0.4
        m["W2"][1:, :2] = 0.0
        m["W2"][0, 0], m["W2"][0, 1] = 1.0, -1.0
        m["b2"][0] = 0.03
    m["kappa"][0] = math.log(20.0)
    return th


def _decoder(th, w):
    out, o = {}, w.n_grid
    for name, shape in w.shapes:
        n = math.prod(shape)
        out[name] = th[o:o + n].view(shape)
        o += n
    return out


def _rays(c, w, frames, R, g):
    """R random pixels and their samples: strata of [near, far] and of [D - g, D + g], sorted."""
    rgb, depth, c2w = frames
    F, H, W = depth.shape
    pix = torch.randint(0, F * H * W, (R,), device=DEV, generator=g)
    f, v, u = pix // (H * W), pix // W % H, pix % W
    d = torch.stack([(u + 0.5 - W / 2) / w.f, (v + 0.5 - H / 2) / w.f, torch.ones(R, device=DEV)], -1).float()
    o, r = c2w[f, :, 3].contiguous(), torch.einsum("rab,rb->ra", c2w[f, :, :3], d).contiguous()
    D = depth.view(-1)[pix]
    N = w.n_strat + w.n_guided

    def strata(n, lo, span):
        k = torch.arange(n, device=DEV) + torch.rand(R, n, device=DEV, generator=g)
        return lo + k * (span / n)

    t = torch.cat([strata(w.n_strat, w.near, w.far - w.near), strata(w.n_guided, D[:, None] - GUIDE, 2 * GUIDE)], 1)
    t = torch.where(D[:, None] > 0, t, strata(N, w.near, w.far - w.near)).sort(1).values
    b = D[:, None] - t
    cls = torch.where(b.abs() <= TRUNC, 1, torch.where(b > TRUNC, 2, 0)) * (D[:, None] > 0)
    return dict(pix=pix, origin=o, dir=r, rgb=rgb.view(-1, 3)[pix].float() / 255.0, depth=D, t=t,
                cls=cls.to(torch.uint8))


def _points(c, w, frames, P, g, jitter=TRUNC):
    """P points near the observed surface."""
    q = _rays(c, w, frames, P, g)
    D = torch.where(q["depth"] > 0, q["depth"], torch.full_like(q["depth"], 1.5))
    return (q["origin"] + D[:, None] * q["dir"] + (torch.rand(P, 3, device=DEV, generator=g) * 2 - 1) * jitter), q


def _batch(c, w, frames, g, R=None, weights=False):
    """A device batch holding rays and smoothness points (what the sampler would have written)."""
    R, P = w.rays if R is None else R, w.n_smooth
    b = gs.Batch.allocate(R, w.n_strat + w.n_guided, P, weights=weights)
    q = _rays(c, w, frames, R, g)
    for k, v in q.items():
        getattr(b, k).copy_(v)
    nv = 0
    if P:
        x, s = _points(c, w, frames, P, g)
        e = torch.randn(P, 3, device=DEV, generator=g)
        b.xs.copy_(x)
        b.eps.copy_(DELTA_S * e / e.norm(dim=1, keepdim=True))
        b.valid.copy_(s["depth"] > 0)
        nv = int(b.valid.sum())
    b.counts.copy_(torch.tensor([int((b.depth > 0).sum()), int((b.cls == 1).sum()), int((b.cls == 2).sum()), nv]))
    return b


def _inputs(c, seed):
    """Everything made from the seed: workload, frames, parameters and the generator to go on with."""
    import random
    rng, g = random.Random(int(seed) * 7919 + 1), _generator(seed)
    w = _workload(c)
    prims = _primitives(c, rng)
    frames = _frames(c, w, prims, rng, g) if c["kind"] not in ("mesh", "adam") else None
    th = _theta(c, w, prims, g) if c["kind"] != "adam" else None
    return w, frames, th, g


def _adam_inputs(w, g):
    """Parameters, moments and a gradient of which an eighth of the vertices were touched."""
    n = w.n_pad
    th = torch.randn(n, device=DEV, generator=g) * 0.1
    touched = (torch.rand(n // 4, device=DEV, generator=g) < 0.125).repeat_interleave(4)
    grad = torch.where(touched, torch.randn(n, device=DEV, generator=g) * 1e-4, torch.zeros(n, device=DEV))
    m = torch.randn(n, device=DEV, generator=g) * 1e-5
    v = torch.rand(n, device=DEV, generator=g) * 1e-9
    return th, grad, m, v


def _prop_params(g):
    q = torch.zeros(1476, device=DEV)
    q[:1473] = torch.randn(1473, device=DEV, generator=g) * 0.1
    return q


def prepare(case, seed):
    c, kind = case, case["kind"]
    w, frames, th, g = _inputs(c, seed)
    s = dict(kind=kind, w=w, seed=int(seed) & 0xFFFFFFFF)
    ctx = gs.Context(w, max_smooth=max(w.n_smooth, 1), store_activations=bool(c.get("store", False)))
    s["ctx"] = ctx
    if kind == "adam":
        s["theta"], s["grad"], s["m"], s["v"] = _adam_inputs(w, g)
        s["mirror"] = torch.zeros(w.n_grid, device=DEV, dtype=torch.bfloat16) if c["mirror"] else None
        s["t"] = 100
        return s
    s["theta"] = th
    if kind == "mesh":
        s["lattice"] = _lattice(c, w)
        nx, ny, nz = s["lattice"]
        s["phi"] = torch.empty(nz, ny, nx, device=DEV)
        return s
    if kind == "query":
        s["x"], _ = _points(c, w, frames, c["points"], g, jitter=0.3)
        s["gs"], s["gg"] = torch.randn(c["points"], device=DEV, generator=g), torch.randn(c["points"], 3, device=DEV, generator=g)
        s["theta"].requires_grad_(True)
        return s
    s["mirror"] = th[:w.n_grid].to(torch.bfloat16) if w.precision == "bf16" else None
    if kind in ("step", "method", "proposal"):
        s["frames"] = gs.DeviceFrames(*frames, w.f, w.f, w.width / 2, w.height / 2)
    if kind == "proposal":
        s["q"] = _prop_params(g)
        s["gq"], s["ce"] = torch.zeros_like(s["q"]), torch.zeros(2, device=DEV)
        s["pdf"] = torch.empty(w.rays, 32, device=DEV)
        s["drawn"] = gs.Batch.allocate(w.rays, w.prop_samples, 0)
        R = min(w.rays, 16384)  # the proposal trains on the first rays of the main model's batch
        s["batch"] = _batch(c, w, frames, g, R=R, weights=True)
        s["batch"].w.copy_(_target_weights(s["batch"].t, s["batch"].depth))
        return s
    if kind in ("step", "method"):
        s["batch"] = gs.Batch.allocate(w.rays, w.N, w.n_smooth, dz=kind == "method",
                                       dz_width=32 if w.arch == "paper" else 16, eik=kind == "method")
    else:
        s["batch"] = _batch(c, w, frames, g)
    s["loss"] = torch.zeros(6, device=DEV)
    if kind == "eval":
        s["rgb"], s["d"], s["wsum"] = (torch.empty(w.rays, 3, device=DEV), torch.empty(w.rays, device=DEV),
                                       torch.empty(w.rays, device=DEV))
    elif kind == "autograd":
        s["theta"].requires_grad_(True)
    else:
        s["grad"] = torch.zeros_like(th)
    if kind == "method":
        n = w.frames
        s["xi"] = torch.randn(n, 6, device=DEV, generator=g) * 2e-3
        s["c2w"] = torch.empty_like(s["frames"].c2w)
        s["posed"] = s["frames"].with_poses(s["c2w"])
        s["pose_grad"], s["eik"] = torch.zeros(n, 6, device=DEV), torch.zeros(1, device=DEV)
    return s


def _target_weights(t, D):
    """Rendering weights peaked at the observed depth (2 m where none was observed)."""
    D = torch.where(D > 0, D, torch.full_like(D, 2.0))
    p = torch.exp(-0.5 * ((t - D[:, None]) / 0.1) ** 2)
    return 0.9 * p / p.sum(1, keepdim=True).clamp(min=1e-6)


def _lattice(c, w):
    return tuple(max(2, int((h - l) / c["step"])) for l, h in zip(w.lo, w.hi))


def run(s):
    kind, ctx, th = s["kind"], s["ctx"], s["theta"]
    if kind == "adam":
        s["t"] += 1
        ctx.adam_step(th, s["grad"], s["m"], s["v"], s["t"], 1e-2, 1e-3, theta_bf16=s["mirror"])
        return {"theta": th, "m": s["m"], "v": s["v"], "grad": s["grad"]} | (
            {} if s["mirror"] is None else {"mirror": s["mirror"]})
    if kind == "mesh":
        w = s["w"]
        _, total = ctx.extract_mesh(th, w.lo, _spacing(w, s["lattice"]), s["lattice"], phi=s["phi"])
        return {"phi": s["phi"], "triangles": total}  # the triangles come in no fixed order
    if kind == "query":
        th.grad = None
        sdf, g = gs.SdfGrad.apply(th, ctx, s["x"])
        torch.autograd.backward((sdf, g), (s["gs"], s["gg"]))
        return {"sdf": sdf.detach(), "grad_x": g.detach(), "grad": th.grad}
    if kind == "proposal":
        b = s["drawn"]
        ctx.proposal_sample(s["frames"], s["seed"], 5, b, theta=th, prop=s["q"], pdf_out=s["pdf"])
        ctx.proposal_backward(th, s["q"], s["batch"], s["gq"], s["ce"])
        return {"pdf": s["pdf"], "t": b.t, "cls": b.cls, "pix": b.pix, "counts": b.counts, "grad": s["gq"],
                "ce": s["ce"]}
    b = s["batch"]
    if kind == "eval":
        ctx.forward(th, b, s["loss"], rgb_hat=s["rgb"], d_hat=s["d"], wsum=s["wsum"], theta_bf16=s["mirror"])
        return {"loss": s["loss"], "rgb": s["rgb"], "depth": s["d"], "wsum": s["wsum"]}
    if kind == "autograd":
        th.grad = None
        losses = gs.GoSurfStep.apply(th, ctx, b, s["mirror"])
        losses[5].backward()
        return {"loss": losses.detach(), "grad": th.grad}
    if kind == "step":
        ctx.sample_rays(s["frames"], s["seed"], 7, b)
    elif kind == "method":
        ctx.pose_apply(s["frames"].c2w, s["xi"], s["c2w"])
        ctx.sample_importance(s["posed"], th, s["seed"], 7, b)
        ctx.eikonal(th, b, loss=s["eik"], grad=s["grad"])  # its grid part rides on the next call's scatter
    # gradients accumulate, as over the several batches of one update
    ctx.forward_backward(th, b, None, s["loss"], s["grad"], theta_bf16=s["mirror"])
    out = {"loss": s["loss"], "grad": s["grad"]}
    if kind == "method":
        ctx.pose_backward(th, s["posed"], s["xi"], b, s["pose_grad"])
        ctx.eikonal_pose_backward(th, s["posed"], s["xi"], b, s["pose_grad"])
        out |= {"eik": s["eik"], "pose_grad": s["pose_grad"]}
    if kind != "grad":
        out |= {"t": b.t, "cls": b.cls, "counts": b.counts}
    return out


def _spacing(w, lattice):
    """The mesh lattice's spacing (the same on every axis)."""
    return (w.hi[0] - w.lo[0]) / lattice[0]


# ---- the work that cannot be avoided -----------------------------------------------------


def work(case):
    c, w = case, _workload(case)
    kind = c["kind"]
    if kind == "adam":
        return {"bytes": float(w.n_pad * 28 + w.n_pad * 0.125 * 4 + (2 * w.n_grid if c["mirror"] else 0)), "flops": 12.0 * w.n_pad}
    if kind == "mesh":
        nx, ny, nz = _lattice(c, w)
        return {"bytes": float(16 * sum(w.counts) + 4 * nx * ny * nz), "flops": nx * ny * nz * 1400.0}
    gb = 2 if w.precision == "bf16" else 4

    def touched(n, per, levels=range(4)):  # a level's vertices are read (or updated) at most once each
        return sum(min(n * 8, w.counts[l]) * per for l in levels)

    if kind == "query":
        n = c["points"]
        return {"bytes": float(touched(n, 16) * 3 + 4 * w.n_pad + n * 56), "flops": n * 9000.0}
    R, N = w.rays, w.N
    S = R * N
    batch = R * 52 + S * 5
    flop = 2 * (3000 if w.arch == "paper" else 1600) + 4 * 80
    colour = min(8 * S, w.counts[3]) * 24 if w.arch == "paper" else 0
    if kind == "eval":
        return {"bytes": float(touched(S, 4 * gb) + colour + batch + R * 20), "flops": float(S * flop)}
    if kind == "proposal":
        T = min(R, 16384)
        return {"bytes": float(touched(R * 32, 16, (0, 1)) + R * (w.prop_samples * 5 + 128 + 60) + T * 96 * 8),
                "flops": 32.0 * (R * 2900 + T * 8700)}
    grad = 2 * touched(S, 16) + 2 * colour
    pts = w.n_smooth * 25 + 3 * touched(2 * w.n_smooth, 16)
    total = touched(S, 4 * gb) + colour + grad + batch + pts
    fl = S * 3 * flop + w.n_smooth * 2 * 9000.0
    if kind == "autograd":
        total += 4 * w.n_pad  # the gradient vector is new on every call
    if kind == "step":
        total += S * 5 + R * 68
    if kind == "method":
        total += 2 * S * 5 + R * 68
        fl += S * (flop + 9000.0)
    return {"bytes": float(total), "flops": float(fl)}


# ---- the same in 64 bits -------------------------------------------------------------------


def _cell(w, l, x):
    """Base vertex, fractions and clamp mask of the cells holding x [P][3] (binary32 decisions)."""
    d = w.dims[l]
    v = torch.tensor(w.voxels[l], device=DEV, dtype=torch.float32)
    u = (x - torch.tensor(w.lo, device=DEV, dtype=torch.float32)) / v
    top = torch.tensor([n - 1 for n in d], device=DEV, dtype=torch.float32)
    clamped = (u < 0) | (u > top)
    u = torch.minimum(u.clamp(min=0), top)
    i = torch.minimum(u.floor().long(), torch.tensor([n - 2 for n in d], device=DEV))
    return (i[:, 2] * d[1] + i[:, 1]) * d[0] + i[:, 0], (u - i.float()).to(F64), clamped


def _corners(w, l, f, clamped):
    """Vertex offset, weight and weight gradient (per metre) of a cell's 8 corners."""
    nx, ny, _ = w.dims[l]
    iv = 1.0 / float(np.float32(w.voxels[l]))
    for k in range(8):
        bits = (k & 1, (k >> 1) & 1, k >> 2)
        a = [f[:, q] if bits[q] else 1 - f[:, q] for q in range(3)]
        sg = [1.0 if b else -1.0 for b in bits]
        dw = torch.stack([sg[0] * a[1] * a[2], a[0] * sg[1] * a[2], a[0] * a[1] * sg[2]], 1) * iv
        yield bits[0] + nx * (bits[1] + ny * bits[2]), a[0] * a[1] * a[2], torch.where(clamped, torch.zeros_like(dw), dw)


def _features(w, grid, x, jac=False):
    """z [P][16] (and dz/dx [P][16][3]) at x from the geometry levels."""
    z, J = [], []
    for l in range(4):
        lev = grid[w.offs[l]:w.offs[l] + 4 * w.counts[l]].view(-1, 4)
        base, f, cl = _cell(w, l, x)
        zl, Jl = 0.0, 0.0
        for off, wt, dw in _corners(w, l, f, cl):
            v = lev[base + off].to(F64)
            zl = zl + wt[:, None] * v
            if jac:
                Jl = Jl + v[:, :, None] * dw[:, None, :]
        z.append(zl)
        J.append(Jl)
    return torch.cat(z, 1), torch.cat(J, 1) if jac else None


def _scatter(w, grad, x, dz=None, dJ=None):
    """Adjoint of _features, added to grad (64 bits)."""
    for l in range(4):
        lev = grad[w.offs[l]:w.offs[l] + 4 * w.counts[l]].view(-1, 4)
        base, f, cl = _cell(w, l, x)
        for off, wt, dw in _corners(w, l, f, cl):
            v = 0.0
            if dz is not None:
                v = v + wt[:, None] * dz[:, 4 * l:4 * l + 4]
            if dJ is not None:
                v = v + (dJ[:, 4 * l:4 * l + 4] * dw[:, None, :]).sum(2)
            lev.index_add_(0, base + off, v)


def _phi(m, w, z):
    """SDF (and the colour decoder's geometry features) from z."""
    if w.arch == "paper":
        a = torch.relu(torch.relu(z @ m["gW1"].T + m["gb1"]) @ m["gW2"].T + m["gb2"])
        return (a @ m["gw3"].T + m["gb3"])[..., 0], None
    y = torch.relu(z @ m["W1"].T + m["b1"]) @ m["W2"].T + m["b2"]
    return y[..., 0], y[..., 1:]


def _colour(m, w, h, cf, d):
    if w.arch == "paper":
        u = torch.cat([cf, d], -1)
        a = torch.relu(torch.relu(u @ m["cW1"].T + m["cb1"]) @ m["cW2"].T + m["cb2"])
        return torch.sigmoid(a @ m["cW3"].T + m["cb3"])
    return torch.sigmoid(torch.relu(h @ m["W3"].T + m["b3"]) @ m["W4"].T + m["b4"])


def _exact_render(c, seed):
    w, frames, th, g = _inputs(c, seed)
    kind = c["kind"]
    b = _batch(c, w, frames, g)
    back = kind != "eval"
    grid = th[:w.n_grid].to(torch.bfloat16) if w.precision == "bf16" else th[:w.n_grid]
    m = {k: v.to(F64).requires_grad_(back) for k, v in _decoder(th, w).items()}
    grad = torch.zeros(w.n_pad if back else 1, device=DEV, dtype=F64)
    n = b.counts.tolist()
    R, N = b.t.shape
    loss = torch.zeros(6, device=DEV, dtype=F64)
    outs = [[], [], []]
    step = max(1, 400000 // N)
    for r0 in range(0, R, step):
        sl = slice(r0, min(R, r0 + step))
        t, o, r, D = b.t[sl], b.origin[sl], b.dir[sl], b.depth[sl]
        x = (o[:, None, :] + t[..., None] * r[:, None, :]).view(-1, 3)
        z = _features(w, grid, x)[0].requires_grad_(back)
        cf = d = None
        if w.arch == "paper":
            lev = grid[w.n_geo:w.n_geo + 6 * w.counts[3]].view(-1, 6)
            base, f, cl = _cell(w, 3, x)
            cf = sum(wt[:, None] * lev[base + off].to(F64) for off, wt, _ in _corners(w, 3, f, cl)).requires_grad_(back)
            d = (r.to(F64) / r.to(F64).norm(dim=1, keepdim=True))[:, None, :].expand(-1, N, 3).reshape(-1, 3)
        with torch.set_grad_enabled(back):
            phi, h = _phi(m, w, z)
            col = _colour(m, w, h, cf, d).view(-1, N, 3)
            phi = phi.view(-1, N)
            P = torch.sigmoid(torch.exp(m["kappa"][0]) * phi)
            al = ((P[:, :-1] - P[:, 1:]) / P[:, :-1].clamp(min=1e-6)).clamp(min=0)
            T = torch.cumprod(torch.cat([torch.ones_like(al[:, :1]), 1 - al], 1), 1)[:, :-1]
            wt = torch.cat([T * al, torch.zeros_like(al[:, :1])], 1)
            ch, dh = (wt[..., None] * col).sum(1), (wt * t.to(F64)).sum(1)
            bb = (D[:, None] - t).to(F64)
            cls = b.cls[sl]
            l_rgb = ((b.rgb[sl].to(F64) - ch) ** 2).sum() / R
            l_d = (D.to(F64) - dh)[D > 0].abs().sum() / max(n[0], 1)
            l_sdf = (phi - bb)[cls == 1].abs().sum() / max(n[1], 1)
            pf, bf = phi[cls == 2], bb[cls == 2]
            l_fs = torch.maximum((torch.exp(-KAPPA_FS * pf) - 1).clamp(min=0), pf - bf).sum() / max(n[2], 1)
            terms = torch.stack([l_rgb, l_d, l_sdf, l_fs])
            if back:
                (terms * torch.tensor(LAMBDAS[:4], device=DEV, dtype=F64)).sum().backward()
        loss[:4] += terms.detach()
        for k, v in enumerate((ch, dh, wt.sum(1))):
            outs[k].append(v.detach())
        if back:
            _scatter(w, grad, x, z.grad)
            if cf is not None:
                lev = grad[w.n_geo:w.n_geo + 6 * w.counts[3]].view(-1, 6)
                base, f, cl = _cell(w, 3, x)
                for off, q, _ in _corners(w, 3, f, cl):
                    lev.index_add_(0, base + off, q[:, None] * cf.grad)
    if w.n_smooth and n[3]:  # the smoothness term reads the FP32 grid in every form
        ok = b.valid.bool()
        pts = (b.xs[ok], (b.xs + b.eps)[ok])
        gr = []
        for x in pts:
            z, J = _features(w, th, x, jac=True)
            z.requires_grad_(True), J.requires_grad_(True)
            p = torch.autograd.grad(_phi(m, w, z)[0].sum(), z, create_graph=back)[0]
            gr.append((J, (J * p[:, :, None]).sum(1)))
        l_sm = ((gr[0][1] - gr[1][1]) ** 2).sum() / n[3]
        loss[4] = l_sm.detach()
        if back:
            (LAMBDAS[4] * l_sm).backward()
            for x, (J, _) in zip(pts, gr):
                _scatter(w, grad, x, dJ=J.grad)
    loss[5] = sum(LAMBDAS[k] * loss[k] for k in range(5))
    if not back:
        return {"loss": loss, "rgb": torch.cat(outs[0]), "depth": torch.cat(outs[1]), "wsum": torch.cat(outs[2])}
    o = w.n_grid
    for name, shape in w.shapes:
        k = math.prod(shape)
        grad[o:o + k] += m[name].grad.reshape(-1)
        o += k
    return {"loss": loss, "grad": grad}


def _exact_query(c, seed):
    w, frames, th, g = _inputs(c, seed)
    x, _ = _points(c, w, frames, c["points"], g, jitter=0.3)
    s, gg = torch.randn(c["points"], device=DEV, generator=g), torch.randn(c["points"], 3, device=DEV, generator=g)
    m = {k: v.to(F64).requires_grad_(True) for k, v in _decoder(th, w).items()}
    z, J = _features(w, th, x, jac=True)
    z.requires_grad_(True), J.requires_grad_(True)
    phi = _phi(m, w, z)[0]
    p = torch.autograd.grad(phi.sum(), z, create_graph=True)[0]
    gx = (J * p[:, :, None]).sum(1)
    ((phi * s.to(F64)).sum() + (gx * gg.to(F64)).sum()).backward()
    grad = torch.zeros(w.n_pad, device=DEV, dtype=F64)
    _scatter(w, grad, x, z.grad, J.grad)
    o = w.n_grid
    for name, shape in w.shapes:
        k = math.prod(shape)
        if m[name].grad is not None:
            grad[o:o + k] += m[name].grad.reshape(-1)
        o += k
    return {"sdf": phi.detach(), "grad_x": gx.detach(), "grad": grad}


def _exact_mesh(c, seed):
    w, _, th, _ = _inputs(c, seed)
    nx, ny, nz = _lattice(c, w)
    m = {k: v.to(F64) for k, v in _decoder(th, w).items()}
    phi = torch.empty(nz, ny, nx, device=DEV, dtype=F64)
    st = torch.tensor(_spacing(w, (nx, ny, nz)), device=DEV, dtype=torch.float32)
    ax = [torch.arange(n, device=DEV, dtype=torch.float32) * st + w.lo[k] for k, n in enumerate((nx, ny, nz))]
    per = max(1, 1500000 // (nx * ny))
    for z0 in range(0, nz, per):
        zz, yy, xx = torch.meshgrid(ax[2][z0:z0 + per], ax[1], ax[0], indexing="ij")
        x = torch.stack([xx, yy, zz], -1).view(-1, 3)
        phi[z0:z0 + per] = _phi(m, w, _features(w, th, x)[0])[0].view(-1, ny, nx)
    return {"phi": phi, "triangles": None}


def _exact_adam(c, seed):
    w, _, _, g = _inputs(c, seed)
    th, grad, m, v = (x.to(F64) for x in _adam_inputs(w, g))
    t, b1, b2, eps = 101, 0.9, 0.999, 1e-8
    b1, b2, eps = (float(np.float32(x)) for x in (b1, b2, eps))
    m = b1 * m + (1 - b1) * grad
    v = b2 * v + (1 - b2) * grad * grad
    lr = torch.full((w.n_pad,), 1e-3, device=DEV, dtype=F64)
    lr[:w.n_grid] = 1e-2
    th = th - lr * (m / (1 - b1 ** t)) / ((v / (1 - b2 ** t)).sqrt() + eps)
    out = {"theta": th, "m": m, "v": v, "grad": torch.zeros_like(th)}
    return out | ({"mirror": None} if c["mirror"] else {})


def _exact_proposal(c, seed):
    """The training step; the draws themselves follow binary32 rules and have no 64-bit value."""
    w, frames, th, g = _inputs(c, seed)
    q = _prop_params(g)[:1473].to(F64).requires_grad_(True)
    b = _batch(c, w, frames, g, R=min(w.rays, 16384), weights=True)
    W1, b1, W2, b2, w3, b3 = q[:352].view(32, 11), q[352:384], q[384:1408].view(32, 32), q[1408:1440], q[1440:1472], q[1472]
    wts = _target_weights(b.t, b.depth)
    width = (w.far - w.near) / 32
    tc = (w.near + (torch.arange(32, device=DEV) + 0.5) * width).float()
    x = (b.origin[:, None, :] + tc[None, :, None] * b.dir[:, None, :]).view(-1, 3)
    z = _features(w, th, x)[0][:, :8]
    d = (b.dir.to(F64) / b.dir.to(F64).norm(dim=1, keepdim=True))[:, None, :].expand(-1, 32, 3).reshape(-1, 3)
    a = torch.relu(torch.relu(torch.cat([z, d], 1) @ W1.T + b1) @ W2.T + b2)
    logp = torch.log_softmax((a @ w3 + b3).view(-1, 32), 1)
    wd = torch.tensor(w.far, dtype=torch.float32) - torch.tensor(w.near, dtype=torch.float32)
    k = ((b.t - w.near) / (wd / 32).to(DEV)).floor().long().clamp(0, 31)
    hist = torch.zeros(b.R, 32, device=DEV, dtype=F64).scatter_add_(1, k, wts.to(F64))
    tot = hist.sum(1)
    use = tot >= 1e-3
    ce = -(hist[use] / tot[use, None] * logp[use]).sum() / use.sum()
    ce.backward()
    grad = torch.zeros(1476, device=DEV, dtype=F64)
    grad[:1473] = q.grad
    return {"pdf": None, "t": None, "cls": None, "pix": None, "counts": None, "grad": grad,
            "ce": torch.stack([ce.detach(), use.sum().to(F64)])}


def exact(case, seed):
    kind = case["kind"]
    if kind in ("grad", "autograd", "eval"):
        return _exact_render(case, seed)
    if kind == "query":
        return _exact_query(case, seed)
    if kind == "mesh":
        return _exact_mesh(case, seed)
    if kind == "adam":
        return _exact_adam(case, seed)
    if kind == "proposal":
        return _exact_proposal(case, seed)
    return None  # whole steps: their rays and depths are drawn by binary32 rules inside the call
