"""The work that users of this library have it do, as measurable cases.

A case is a dict of plain values; `prepare` makes its inputs and the objects a program keeps (model, contexts,
captured iterations) on the GPU, `run` is one pass through the public entry points, `work` what the pass cannot
do without, and `exact` the same results in 64 bits from plain torch (the method written out below, without the
library).  Scenes are the library's synthetic hand captures: a posed hand seen by a ring of pinhole cameras over
random plates, observations rendered from another pose plus sensor noise.
"""
import dataclasses
import functools
import math

import numpy as np
import torch
import torch.nn.functional as F

from paper_2107_05509_gb300 import binding as B
from paper_2107_05509_gb300 import inputs as I
from paper_2107_05509_gb300 import pipeline as P
from paper_2107_05509_gb300 import proposal

# Area of the hand in a view, in units of W^2 pixels (focal length 1.2 W at 0.6 m), averaged over a ring.
HAND_AREA = 0.03


def listed():
    return [
        # One refinement iteration of one hand (skinning, BVH, render, loss, backward, skinning adjoint) as a
        # captured step: a preview-size capture, where launches and latencies are all there is ...
        dict(name="step-tiny", kind="step", views=2, width=128, height=128, spp=4, edge_samples=1024),
        # ... and the paper's workload, the call that a refinement repeats hundreds of times.
        dict(name="step-paper", kind="step", views=8, width=512, height=384, spp=16, edge_samples=4096),
        # Forward and backward of the subdivided, textured hand at full resolution and 64 samples per pixel.
        dict(name="textured-scale", kind="textured", levels=2, texture=256, views=16, width=1024, height=1024, spp=64,
             edge_samples=32768),
        # The same for the heterogeneous batch: 64 hands with 4-16 views of 256^2 to 512^2 each.
        dict(name="batch-64", kind="batch", n=64, layout=2000),
        # Rendering training pairs for the proposal network: many small views at few samples per pixel.
        dict(name="pairs-128", kind="pairs", n=128, views=8, width=256, height=256, spp=4),
        # The masked photometric loss and its adjoint over a full-resolution capture.
        dict(name="loss-scale", kind="loss", views=16, width=1024, height=1024),
        # The paper's other objective terms: colour map, colour transforms, Canny edge term, with their adjoints.
        dict(name="objective-paper", kind="objective", views=8, width=512, height=384, texture=512),
        # One proposal for the 64 hands of a batch: residual inputs and the network's forward pass.
        dict(name="propose-64", kind="propose", n=64, views=8),
        # The network's share of a training step on 128 pairs: inputs, forward, parameter gradients.
        dict(name="train-128", kind="train", n=128, views=8),
        # The library's bf16 matrix product at the size its peak is quoted on.
        dict(name="gemm-8192", kind="gemm", m=8192, n=8192, k=8192, bias=False, relu=False, bf16=True, splits=1),
        # Geometry of a training batch: skinning, BVH, skinning adjoint for 128 hands.
        dict(name="geometry-128", kind="geometry", n=128),
        # Bringing captured views (plates and masks) to the proposal network's grid.
        dict(name="resample-96", kind="resample", views=96, width=512, height=384, out_w=256, out_h=256),
    ]


def draw(rng):
    def log(lo, hi):
        return min(hi, max(lo, round(math.exp(rng.uniform(math.log(lo), math.log(hi + 1)) - 0.5 / hi))))

    def size(lo, hi):   # sides are often, not always, multiples of 8
        x = log(lo, hi)
        return max(lo, x - x % 8) if rng.random() < 0.4 else x

    kind = rng.choice(["step", "step", "step", "textured", "textured", "batch", "batch", "pairs", "loss", "objective",
                       "propose", "train", "gemm", "geometry", "resample"])
    if kind == "step":
        return dict(kind=kind, views=rng.randint(1, 16), width=size(64, 512), height=size(64, 512), spp=log(1, 32),
                    edge_samples=log(256, 8192))
    if kind == "textured":
        return dict(kind=kind, levels=rng.randint(0, 2), texture=log(64, 512), views=rng.randint(1, 16),
                    width=size(96, 1024), height=size(96, 1024), spp=log(2, 64), edge_samples=log(256, 32768))
    if kind == "batch":
        return dict(kind=kind, n=log(2, 48), layout=rng.randint(3000, 9999))
    if kind == "pairs":
        return dict(kind=kind, n=log(1, 100), views=rng.randint(1, 8), width=size(64, 256), height=size(64, 256),
                    spp=log(1, 8))
    if kind == "loss":
        return dict(kind=kind, views=rng.randint(1, 16), width=size(64, 1024), height=size(64, 1024))
    if kind == "objective":
        return dict(kind=kind, views=rng.randint(1, 16), width=size(64, 640), height=size(64, 640),
                    texture=8 * log(8, 64))
    if kind in ("propose", "train"):
        return dict(kind=kind, n=4 * log(1, 24), views=rng.randint(1, 10))
    if kind == "gemm":
        bf16 = rng.random() < 0.5
        return dict(kind=kind, m=log(1, 8192), n=log(8, 8192), k=64 * log(1, 120), bias=rng.random() < 0.5,
                    relu=rng.random() < 0.5, bf16=bf16, splits=1 if bf16 else rng.choice([1, 1, 2, 5, 16]))
    if kind == "geometry":
        return dict(kind=kind, n=log(1, 256))
    return dict(kind=kind, views=log(1, 90), width=size(64, 1024), height=size(64, 512), out_w=log(64, 256),
                out_h=log(64, 256))


# --------------------------------------------------------------------------------------
# Inputs
# --------------------------------------------------------------------------------------

@functools.lru_cache(maxsize=None)
def _hand(levels):
    """The hand asset (subdivided `levels` times): read from disk once in a user's program."""
    hand = I.make_hand(0)
    return I.subdivide_hand(hand, levels) if levels else hand


def _gen(seed):
    return torch.Generator(device="cuda").manual_seed(seed)


def _config(views, width, height, spp, edge_samples):
    return I.SceneConfig("case", views=views, width=width, height=height, spp=spp, edge_samples=edge_samples,
                         elevation_deg=30.0, azimuths_deg=tuple(360.0 * k / views for k in range(views)))


def _cameras(cfgs):
    target = _hand(0).v_template.mean(0)
    return torch.as_tensor(np.concatenate([I.pack_cameras(I.make_cameras(c, target)) for c in cfgs]), device="cuda")


def _params(seed, n):
    gt = np.stack([I.gt_params(1000 * seed + i) for i in range(n)])
    est = np.stack([I.perturb_params(gt[i], 1000 * seed + i) for i in range(n)])
    return torch.as_tensor(gt, device="cuda"), torch.as_tensor(est, device="cuda")


def _noisy(image, gen):
    return image + 0.01 * torch.randn(image.shape, generator=gen, device="cuda")


def _mask(image, plate):
    """Pixels the hand covers, dilated by 8 pixels, of [N][H][W][3] images."""
    hit = (image != plate).any(-1, keepdim=True).permute(0, 3, 1, 2).float()
    return F.max_pool2d(hit, 17, 1, 8)[:, 0].to(torch.uint8)


def _options(cfg, seed, **kw):
    return P.opts_for(cfg, seed=7919 * seed + 17, **kw)


def _scene(cfg, levels, seed, texture=None):
    """One capture: model, views and parameters of the estimate."""
    gen = _gen(seed)
    model = B.Model(_hand(levels))
    cams = _cameras([cfg])
    gt, est = _params(seed, 1)
    ctx = B.Context(model.hand.V, model.hand.F, model.hand.E, cfg.views, cfg.width, cfg.height)
    shape = (cfg.views, cfg.height, cfg.width, 3)
    plate = torch.rand(shape, generator=gen, device="cuda")
    verts, clean = torch.empty((model.V, 3), device="cuda"), torch.empty(shape, device="cuda")
    B.hr_skin(ctx, model, gt[0], verts)
    B.hr_build_bvh(ctx, model, verts)
    B.hr_render_fwd(ctx, model, verts, cams, cfg.height, cfg.width, plate, _options(cfg, seed + 1, texture=texture), clean)
    views = P.Views(cams=cams, background=plate, observed=_noisy(clean, gen), mask=_mask(clean, plate),
                    H=cfg.height, W=cfg.width)
    return model, views, est[0].contiguous(), ctx


def _prepare_step(c, seed):
    cfg = _config(c["views"], c["width"], c["height"], c["spp"], c["edge_samples"])
    model, views, params, ctx = _scene(cfg, 0, seed)
    ref = P.Refiner(model, views, _options(cfg, seed), ctx=ctx)
    return dict(ref=ref, params=params, graph=ref.capture_step(params))


def _prepare_textured(c, seed):
    cfg = _config(c["views"], c["width"], c["height"], c["spp"], c["edge_samples"])
    tex = torch.as_tensor(I.texture(seed, c["texture"]), device="cuda")
    model, views, params, ctx = _scene(cfg, c["levels"], seed, texture=tex)
    d_tex = torch.zeros_like(tex)
    ref = P.Refiner(model, views, _options(cfg, seed, texture=tex, d_texture=d_tex), ctx=ctx)
    ref.forward(params)      # leaves the adjoint image that the timed backward takes
    return dict(ref=ref, params=params, tex=tex, d_tex=d_tex)


def _batch_configs(c):
    if c["kind"] == "batch":
        return I.batch_configs(c["n"], seed_base=c["layout"])
    return [_config(c["views"], c["width"], c["height"], c["spp"], 0)] * c["n"]


def _prepare_batch(c, seed):
    cfgs = _batch_configs(c)
    gen = _gen(seed)
    model = B.Model(_hand(0))
    bt = B.Batch(model.hand.V, model.hand.F, model.hand.E,
                 [(k.views, k.width, k.height, k.spp, k.edge_samples, i) for i, k in enumerate(cfgs)])
    gt, est = _params(seed, c["n"])
    # a batch usually shares few distinct camera rigs
    rigs = {k: _cameras([k]) for k in set(cfgs)}
    cams = torch.cat([rigs[k] for k in cfgs])
    plate = torch.rand((bt.total_pixels, 3), generator=gen, device="cuda")
    state = dict(model=model, bt=bt, cams=cams, plate=plate, params=est, gt=gt,
                 verts=torch.empty((c["n"], model.V, 3), device="cuda"), image=torch.empty_like(plate),
                 opts=_options(cfgs[0], seed))
    if c["kind"] == "pairs":
        return state
    _batch_forward(state, gt, _options(cfgs[0], seed + 1))
    mask = torch.empty(bt.total_pixels, dtype=torch.uint8, device="cuda")
    for i, k in enumerate(cfgs):
        sl = slice(int(bt.pixel_offsets[i]), int(bt.pixel_offsets[i + 1]))
        shape = (k.views, k.height, k.width, 3)
        mask[sl] = _mask(state["image"][sl].view(shape), plate[sl].view(shape)).reshape(-1)
    obs = _noisy(state["image"], gen)
    state.update(adjoint=torch.empty_like(plate), d_verts=torch.empty_like(state["verts"]),
                 d_params=torch.empty_like(est), loss=torch.empty(c["n"], device="cuda"))
    _batch_forward(state, est, state["opts"])
    B.hr_loss_batch(bt, state["image"], obs, mask, state["loss"], state["adjoint"])
    return state


def _batch_forward(s, params, opts):
    B.hr_skin_batch(s["bt"], s["model"], params, s["verts"])
    B.hr_build_bvh_batch(s["bt"], s["model"], s["verts"])
    B.hr_render_fwd_batch(s["bt"], s["model"], s["verts"], s["cams"], s["plate"], opts, s["image"])


def _shaded_images(c, seed):
    """Images with the statistics of a render over a noise plate and of its observation, without rendering:
    smooth blobs over random plates, and the mask of the blobs."""
    gen = _gen(seed)
    n, h, w = c["views"], c["height"], c["width"]
    rand = lambda *s: torch.rand(s, generator=gen, device="cuda")
    centre = rand(n, 6, 2) * 0.5 + 0.25
    radius = 0.05 + 0.12 * rand(n, 6)
    y = (torch.arange(h, device="cuda") + 0.5) / h
    x = (torch.arange(w, device="cuda") + 0.5) / w
    d = ((y[None, None, :, None] - centre[:, :, 0, None, None]) ** 2 +
         (x[None, None, None, :] - centre[:, :, 1, None, None]) ** 2).sqrt() / radius[:, :, None, None]
    near = d.amin(1)
    shade = (0.85 - 0.5 * near.clamp(0, 1) ** 2)[..., None] * (0.4 + 0.6 * rand(n, 1, 1, 3))
    plate = rand(n, h, w, 3)
    cover = ((1.0 - near) * 40.0).clamp(0, 1)[..., None]
    clean = cover * shade + (1 - cover) * plate
    image = (clean.roll((2, -1), (1, 2)) + clean) * 0.5
    mask = F.max_pool2d((near < 1.0)[:, None].float(), 17, 1, 8)[:, 0].to(torch.uint8)
    return image.contiguous(), _noisy(clean, gen), mask


def _prepare_loss(c, seed):
    image, observed, mask = _shaded_images(c, seed)
    hand = _hand(0)
    return dict(ctx=B.Context(hand.V, hand.F, hand.E, c["views"], c["width"], c["height"]), image=image,
                observed=observed, mask=mask, loss=torch.empty(1, device="cuda"), adjoint=torch.empty_like(image))


def _prepare_objective(c, seed):
    s = _prepare_loss(c, seed)
    gen = _gen(seed + 7)
    n, t = c["views"], c["texture"]
    s["T"] = torch.eye(3, device="cuda").reshape(1, 9) + 0.05 * torch.randn((n, 9), generator=gen, device="cuda")
    s["low"] = torch.rand((8, 8, 3), generator=gen, device="cuda")
    s["high"] = 0.05 * torch.randn((t, t, 3), generator=gen, device="cuda")
    s["d_tex"] = torch.randn((t, t, 3), generator=gen, device="cuda") * (torch.rand((t, t, 1), generator=gen, device="cuda") < 0.3)
    s["edges_obs"] = torch.empty(s["mask"].shape, device="cuda")
    B.hr_edges(s["ctx"], s["observed"], s["edges_obs"])
    s.update(dT=torch.empty((n, 9), device="cuda"), tex=torch.empty((t, t, 3), device="cuda"),
             d_low=torch.empty((8, 8, 3), device="cuda"), edge_loss=torch.empty(1, device="cuda"))
    return s


@functools.lru_cache(maxsize=None)
def _weights():
    return proposal.load_weights(proposal.WEIGHTS)[0]


def _prepare_net(c, seed):
    n, k = c["n"], c["views"]
    image, observed, _ = _shaded_images(dict(views=n * k, height=256, width=256), seed)
    cams = _cameras([_config(k, 256, 256, 16, 0)] * n)
    net = B.Net(n, k)
    gen = _gen(seed + 3)
    weights = torch.as_tensor(_weights(), device="cuda")
    net.set_params(weights)
    return dict(net=net, weights=weights, image=image, observed=observed, cams=cams, base=_params(seed, n)[1],
                out=torch.empty((n, 61), device="cuda"), d_out=torch.randn((n, 61), generator=gen, device="cuda") / n,
                grads=torch.empty(net.P, device="cuda"))


def _prepare_gemm(c, seed):
    gen = _gen(seed)
    m, n, k = c["m"], c["n"], c["k"]
    hand = _hand(0)
    rand = lambda r, q: torch.randn((r, q), generator=gen, device="cuda").to(torch.bfloat16)
    s = dict(ctx=B.Context(hand.V, hand.F, hand.E, 1, 64, 64), a=rand(m, k), b=rand(n, k), bias=None, buf=None,
             out=torch.empty((m, n), dtype=torch.bfloat16 if c["bf16"] else torch.float32, device="cuda"),
             relu=c["relu"], splits=c["splits"])
    if c["bias"]:
        s["bias"] = torch.randn(n, generator=gen, device="cuda")
    if c["splits"] > 1:
        s["buf"] = torch.empty((c["splits"], m, n), device="cuda")
    return s


def _prepare_geometry(c, seed):
    n = c["n"]
    model = B.Model(_hand(0))
    bt = B.Batch(model.hand.V, model.hand.F, model.hand.E, [(1, 64, 64, 1, 0, i) for i in range(n)])
    verts = torch.empty((n, model.V, 3), device="cuda")
    return dict(model=model, bt=bt, params=_params(seed, n)[1], verts=verts,
                d_verts=torch.randn(verts.shape, generator=_gen(seed), device="cuda") / model.V,
                d_params=torch.empty((n, 61), device="cuda"))


def _prepare_resample(c, seed):
    gen = _gen(seed)
    n, h, w, ho, wo = c["views"], c["height"], c["width"], c["out_h"], c["out_w"]
    mask = F.max_pool2d((torch.rand((n, 1, h, w), generator=gen, device="cuda") > 0.9995).float(), 17, 1, 8)
    return dict(src=torch.rand((n, h, w, 3), generator=gen, device="cuda"), mask=mask[:, 0].to(torch.uint8).contiguous(),
                dst=torch.empty((n, ho, wo, 3), device="cuda"),
                dmask=torch.empty((n, ho, wo), dtype=torch.uint8, device="cuda"))


_PREPARE = dict(step=_prepare_step, textured=_prepare_textured, batch=_prepare_batch, pairs=_prepare_batch,
                loss=_prepare_loss, objective=_prepare_objective, propose=_prepare_net, train=_prepare_net,
                gemm=_prepare_gemm, geometry=_prepare_geometry, resample=_prepare_resample)


def prepare(case, seed):
    return dict(_PREPARE[case["kind"]](case, seed), kind=case["kind"])


# --------------------------------------------------------------------------------------
# One pass
# --------------------------------------------------------------------------------------

def _run_step(s):
    s["graph"].replay()
    r = s["ref"]
    return dict(image=r.image, loss=r.loss, d_verts=r.d_verts, d_params=r.d_params)


def _run_textured(s):
    r, v = s["ref"], s["ref"].views
    B.hr_skin(r.ctx, r.model, s["params"], r.verts)
    B.hr_build_bvh(r.ctx, r.model, r.verts)
    B.hr_render_fwd(r.ctx, r.model, r.verts, v.cams, v.H, v.W, v.background, r.opts, r.image)
    s["d_tex"].zero_()
    B.hr_render_bwd(r.ctx, r.model, r.verts, v.cams, v.H, v.W, v.background, r.opts, r.adjoint, r.d_verts)
    B.hr_skin_bwd(r.ctx, r.model, s["params"], r.d_verts, r.d_params)
    return dict(image=r.image, d_verts=r.d_verts, d_tex=s["d_tex"], d_params=r.d_params)


def _run_batch(s):
    _batch_forward(s, s["params"], s["opts"])
    B.hr_render_bwd_batch(s["bt"], s["model"], s["verts"], s["cams"], s["plate"], s["opts"], s["adjoint"], s["d_verts"])
    B.hr_skin_bwd_batch(s["bt"], s["model"], s["params"], s["d_verts"], s["d_params"])
    return dict(image=s["image"], d_verts=s["d_verts"], d_params=s["d_params"])


def _run_pairs(s):
    _batch_forward(s, s["params"], s["opts"])
    return dict(image=s["image"], verts=s["verts"])


def _run_loss(s):
    B.hr_loss(s["ctx"], s["image"], s["observed"], s["mask"], s["loss"], s["adjoint"])
    return dict(loss=s["loss"], adjoint=s["adjoint"])


def _run_objective(s):
    B.hr_colour_map(s["low"], s["high"], s["tex"])
    B.hr_loss_ct(s["ctx"], s["image"], s["observed"], s["mask"], s["T"], s["loss"], s["adjoint"], s["dT"])
    B.hr_edge_loss(s["ctx"], s["image"], s["edges_obs"], s["mask"], s["edge_loss"], s["adjoint"], T=s["T"], dT=s["dT"])
    B.hr_colour_map_bwd(s["d_tex"], s["d_low"])
    return {k: s[k] for k in ("tex", "loss", "edge_loss", "adjoint", "dT", "d_low")}


def _run_propose(s):
    s["net"].inputs(s["image"], s["observed"])
    s["net"].forward(s["cams"], s["out"], base=s["base"])
    return s["out"]


def _run_train(s):
    _run_propose(s)
    s["net"].backward(s["d_out"])
    s["net"].get_params(grads=s["grads"])
    return dict(out=s["out"], grads=s["grads"])


def _run_gemm(s):
    B.hr_gemm_bf16(s["ctx"], s["a"], s["b"], s["out"], bias=s["bias"], relu=s["relu"], splits=s["splits"], split_buf=s["buf"])
    return s["out"]


def _run_geometry(s):
    B.hr_skin_batch(s["bt"], s["model"], s["params"], s["verts"])
    B.hr_build_bvh_batch(s["bt"], s["model"], s["verts"])
    B.hr_skin_bwd_batch(s["bt"], s["model"], s["params"], s["d_verts"], s["d_params"])
    return dict(verts=s["verts"], d_params=s["d_params"])


def _run_resample(s):
    B.hr_area_resample(s["src"], s["dst"])
    B.hr_mask_resample(s["mask"], s["dmask"])
    return dict(dst=s["dst"], dmask=s["dmask"])


_RUN = dict(step=_run_step, textured=_run_textured, batch=_run_batch, pairs=_run_pairs, loss=_run_loss,
            objective=_run_objective, propose=_run_propose, train=_run_train, gemm=_run_gemm,
            geometry=_run_geometry, resample=_run_resample)


def run(state):
    return _RUN[state["kind"]](state)


# --------------------------------------------------------------------------------------
# What a pass cannot do without
# --------------------------------------------------------------------------------------

def _render_work(cfgs, backward, loss=False):
    """Images: plate in, render out (forward), observation, mask (loss), adjoint in (backward) once each.  Per
    covered sample: 40 operations of sampling, 50 of one intersection and 60 of shading, 250 of differentiation;
    per edge sample 120 of set-up and two shaded rays."""
    px = sum(k.views * k.width * k.height for k in cfgs)
    hits = sum(k.views * HAND_AREA * k.width ** 2 * k.spp for k in cfgs)
    edge = sum(k.views * k.edge_samples for k in cfgs)
    if not backward:
        return dict(bytes=24 * px, flops=150 * hits)
    return dict(bytes=(24 + 12 + (13 if loss else 0)) * px, flops=(150 + 340) * hits + 340 * edge)


def _net_work(c, backward):
    nv = c["n"] * c["views"]
    macs = nv * (64 * 64 * 72 * 32 + 32 * 32 * 288 * 64 + 16 * 16 * 576 * 128 + 8 * 8 * 1152 * 128 + 4 * 4 * 1152 * 128 +
                 2060 * 256) + c["n"] * (256 * 256 + 256 * 61)
    weights = 1_020_000
    images = nv * 2 * 256 * 256 * 12
    if not backward:
        return dict(bytes=images + 2 * weights + c["n"] * 61 * 8, flops=2 * macs)
    return dict(bytes=images + 6 * weights + c["n"] * 61 * 12, flops=2 * macs + 4 * macs - 2 * nv * 64 * 64 * 72 * 32)


def work(case):
    c, k = case, case["kind"]
    if k in ("step", "textured"):
        return _render_work([_config(c["views"], c["width"], c["height"], c["spp"], c["edge_samples"])], True, k == "step")
    if k in ("batch", "pairs"):
        return _render_work(_batch_configs(c), k == "batch")
    if k in ("loss", "objective"):
        px = c["views"] * c["width"] * c["height"]
        if k == "loss":
            return dict(bytes=37 * px, flops=10 * px)
        return dict(bytes=41 * px + 36 * c["texture"] ** 2, flops=200 * px + 6 * c["texture"] ** 2)
    if k in ("propose", "train"):
        return _net_work(c, k == "train")
    if k == "gemm":
        m, n, kk = c["m"], c["n"], c["k"]
        return dict(bytes=2 * kk * (m + n) + m * n * (2 if c["bf16"] else 4), flops=2 * m * n * kk)
    if k == "geometry":
        # vertices out and their adjoints in, triangle records and tree nodes out, the model once
        return dict(bytes=c["n"] * (778 * 24 + 1538 * (48 + 64) + 488) + 150_000, flops=c["n"] * 778 * 1200)
    return dict(bytes=c["views"] * 13 * (c["width"] * c["height"] + c["out_w"] * c["out_h"]),
                flops=c["views"] * 6 * c["width"] * c["height"])


# --------------------------------------------------------------------------------------
# The method in 64 bits
# --------------------------------------------------------------------------------------

D = torch.float64
MASK32 = 0xFFFFFFFF


def _dev(a, dtype=None):
    t = torch.as_tensor(a, device="cuda")
    return t if dtype is None else t.to(dtype)


@dataclasses.dataclass
class _Mesh:
    faces: torch.Tensor
    edges: torch.Tensor
    edge_faces: torch.Tensor
    albedo: torch.Tensor
    uv: torch.Tensor
    arrays: dict


@functools.lru_cache(maxsize=None)
def _mesh(levels):
    h = _hand(levels)
    arrays = {k: _dev(getattr(h, k), D) for k in ("v_template", "shapedirs", "weights", "j_template", "j_shapedirs")}
    return _Mesh(_dev(h.faces, torch.int64), _dev(h.edges, torch.int64), _dev(h.edge_faces, torch.int64),
                 _dev(h.albedo, D), _dev(h.uv, D), dict(arrays, parents=list(h.parents)))


def _rotation(r):
    """Rodrigues' formula, [n][3] -> [n][3][3]."""
    t = (r * r).sum(-1).clamp_min(1e-30).sqrt()[:, None, None]
    z = torch.zeros_like(r[:, 0])
    k = torch.stack([z, -r[:, 2], r[:, 1], r[:, 2], z, -r[:, 0], -r[:, 1], r[:, 0], z], -1).view(-1, 3, 3)
    return torch.eye(3, dtype=D, device="cuda") + torch.sin(t) / t * k + 2 * (torch.sin(t / 2) / t) ** 2 * (k @ k)


def _skin(x, a):
    """Linear blend skinning of parameters [n][61] -> vertices [n][V][3]."""
    n = x.shape[0]
    beta, pose, root, tau = x[:, :10], x[:, 10:55].reshape(n, 15, 3), x[:, 55:58], x[:, 58:61]
    joints = a["j_template"] + torch.einsum("jck,nk->njc", a["j_shapedirs"], beta)
    rot = _rotation(torch.cat([root[:, None], pose], 1).reshape(-1, 3)).view(n, 16, 3, 3)
    g_rot, g_pos = [], []
    for j, p in enumerate(a["parents"]):
        if p < 0:
            g_rot.append(rot[:, j])
            g_pos.append(joints[:, j])
        else:
            g_rot.append(g_rot[p] @ rot[:, j])
            g_pos.append(g_pos[p] + (g_rot[p] @ (joints[:, j] - joints[:, p])[..., None])[..., 0])
    g_rot, g_pos = torch.stack(g_rot, 1), torch.stack(g_pos, 1)
    shift = g_pos - (g_rot @ joints[..., None])[..., 0]
    shaped = a["v_template"] + torch.einsum("vck,nk->nvc", a["shapedirs"], beta)
    blend = torch.einsum("vj,njab->nvab", a["weights"], g_rot)
    return (blend @ shaped[..., None])[..., 0] + torch.einsum("vj,nja->nva", a["weights"], shift) + tau[:, None]


def _normals(v, faces):
    a, b, c = v[faces[:, 0]], v[faces[:, 1]], v[faces[:, 2]]
    area = torch.cross(b - a, c - a, dim=-1)
    m = torch.zeros_like(v)
    for k in range(3):
        m = m.index_add(0, faces[:, k], area)
    return m / m.norm(dim=-1, keepdim=True)


def _philox(c0, c1, c2, c3, seed):
    """Philox4x32-10 of counters (int64 tensors or numbers), key = the 64-bit seed; the first two words."""
    c = list(torch.broadcast_tensors(*[torch.as_tensor(t, device="cuda") for t in (c0, c1, c2, c3)]))
    k0, k1 = seed & MASK32, (seed >> 32) & MASK32
    for _ in range(10):
        p0, p1 = c[0] * 0xD2511F53, c[2] * 0xCD9E8D57      # low 64 bits of the product, wrapped
        c = [((p1 >> 32) & MASK32) ^ c[1] ^ k0, p1 & MASK32, ((p0 >> 32) & MASK32) ^ c[3] ^ k1, p0 & MASK32]
        k0, k1 = (k0 + 0x9E3779B9) & MASK32, (k1 + 0xBB67AE85) & MASK32
    return c[0], c[1]


def _u24(r):
    return (r >> 8).to(D) * 2.0 ** -24


def _dot(a, b):
    return (a * b).sum(-1)


def _expand(count):
    """For counts per item: (item of each entry, its index within the item)."""
    item = torch.repeat_interleave(torch.arange(len(count), device="cuda"), count)
    return item, torch.arange(len(item), device="cuda") - (count.cumsum(0) - count)[item]


class _View:
    """One pinhole view of a mesh: which triangles can meet which pixel, and rays through screen points."""

    def __init__(self, cam, v, mesh, H, W):
        self.H, self.W, self.mesh, self.v = H, W, mesh, v
        self.fx, self.fy, self.cx, self.cy = (cam[i] for i in range(4))
        self.R, self.t, self.o = cam[4:13].view(3, 3), cam[13:16], cam[16:19]
        self.p = v[mesh.faces]                                     # [F][3][3]
        self.xy = self.project(v)
        q = self.xy[mesh.faces]
        lim = torch.tensor([W - 1, H - 1], device="cuda")
        lo = (q.amin(1) - 0.1).floor().long().clamp_min(0)
        hi = torch.minimum((q.amax(1) + 0.1).floor().long(), lim)
        ext = (hi - lo + 1).clamp_min(0)
        tri, i = _expand(ext[:, 0] * ext[:, 1])
        w = ext[tri, 0].clamp_min(1)
        pix = (lo[tri, 1] + i // w) * W + lo[tri, 0] + i % w
        order = torch.argsort(pix, stable=True)
        self.cand = tri[order]
        self.count = torch.bincount(pix, minlength=H * W)
        self.start = self.count.cumsum(0) - self.count

    def project(self, v):
        c = v @ self.R.T + self.t
        return torch.stack([self.fx * c[:, 0] / c[:, 2] + self.cx, self.fy * c[:, 1] / c[:, 2] + self.cy], -1)

    def direction(self, x, y):
        d = torch.stack([(x - self.cx) / self.fx, (y - self.cy) / self.fy, torch.ones_like(x)], -1)
        return d @ self.R

    def closest(self, pix, d):
        """Triangle of the nearest hit of rays d through pixels pix, -1 for a miss."""
        ray, i = _expand(self.count[pix])
        tri = self.cand[self.start[pix][ray] + i]
        a, dr = self.p[tri], d[ray]
        e1, e2, s = a[:, 1] - a[:, 0], a[:, 2] - a[:, 0], self.o - a[:, 0]
        q = torch.cross(dr, e2, dim=-1)
        inv = 1.0 / _dot(e1, q)
        u = _dot(s, q) * inv
        q = torch.cross(s, e1, dim=-1)
        w, t = _dot(dr, q) * inv, _dot(e2, q) * inv
        ok = (u >= 0) & (w >= 0) & (u + w <= 1) & (t > 0)
        t = torch.where(ok, t, math.inf)
        best = torch.full((len(pix),), math.inf, dtype=D, device="cuda").scatter_reduce_(0, ray, t, "amin")
        win = ok & (t == best[ray])
        none = len(self.p)
        hit = torch.full((len(pix),), none, device="cuda").scatter_reduce_(0, ray[win], tri[win], "amin")
        return torch.where(hit == none, -1, hit)

    def shade(self, a, n, tri, d, tex):
        """Radiance of hits on triangles with corners a and corner normals n ([h][3][3] each) along rays d.
        tex: the texture's four texels under each hit come from `tex` ([S][S][3]), else per-vertex albedo."""
        e1, e2, s = a[:, 1] - a[:, 0], a[:, 2] - a[:, 0], self.o - a[:, 0]
        q = torch.cross(d, e2, dim=-1)
        inv = 1.0 / _dot(e1, q)
        u = _dot(s, q) * inv
        w = _dot(d, torch.cross(s, e1, dim=-1)) * inv
        b = torch.stack([1 - u - w, u, w], -1)[..., None]
        nm = (b * n).sum(1)
        light = torch.tensor(I.LIGHT_DIR, dtype=D, device="cuda")
        k = I.K_AMBIENT + I.K_DIFFUSE * (nm @ light).clamp_min(0) / nm.norm(dim=-1)
        f = self.mesh.faces[tri]
        if tex is None:
            return (b * self.mesh.albedo[f]).sum(1) * k[:, None], None
        size = tex.shape[0]
        st = (b * self.mesh.uv[f]).sum(1) * size - 0.5
        cell = st.detach().floor()
        fr = st - cell
        i0, i1 = cell.long().clamp(0, size - 1), (cell.long() + 1).clamp(0, size - 1)
        idx = torch.stack([i0[:, 1] * size + i0[:, 0], i0[:, 1] * size + i1[:, 0], i1[:, 1] * size + i0[:, 0],
                           i1[:, 1] * size + i1[:, 0]], 1)
        wx, wy = fr[:, 0], fr[:, 1]
        wt = torch.stack([(1 - wx) * (1 - wy), wx * (1 - wy), (1 - wx) * wy, wx * wy], 1)
        return (wt[..., None] * tex.view(-1, 3)[idx]).sum(1) * k[:, None], (idx, wt, k)


def _samples(view, spp, ctr1, seed, most=12_000_000):
    """The primary samples of a view that can hit something, in groups: (pixel, ray) of whole pixels."""
    pix = torch.nonzero(view.count)[:, 0]
    cost = (view.count[pix] * spp).cumsum(0)
    part = (cost // most).tolist() if len(pix) else []
    cuts = [0] + [i for i in range(1, len(part)) if part[i] != part[i - 1]] + [len(pix)]
    for lo, hi in zip(cuts[:-1], cuts[1:]):
        p = pix[lo:hi].repeat_interleave(spp)
        s = torch.arange(spp, device="cuda").repeat(hi - lo)
        r0, r1 = _philox(p, ctr1, s, 0, seed)
        # sample points are single-precision numbers by definition
        x = ((p % view.W).to(D) + _u24(r0)).float().to(D)
        y = (torch.div(p, view.W, rounding_mode="floor").to(D) + _u24(r1)).float().to(D)
        yield p, view.direction(x, y)


def _render(view, n, plate, spp, ctr1, seed, tex, adjoint=None, grads=None):
    """The view's image [HW][3]; with `adjoint`, adds the interior gradient to grads (v, n, tex)."""
    total = torch.zeros_like(plate)
    hits = torch.zeros(len(plate), dtype=D, device="cuda")
    for p, d in _samples(view, spp, ctr1, seed):
        tri = view.closest(p, d)
        h = tri >= 0
        p, d, tri = p[h], d[h], tri[h]
        f = view.mesh.faces[tri]
        a, nn = view.p[tri], n[f]
        if adjoint is not None:
            a, nn = a.clone().requires_grad_(), nn.clone().requires_grad_()
        rgb, texel = view.shade(a, nn, tri, d, tex)
        total.index_add_(0, p, rgb.detach())
        hits.index_add_(0, p, torch.ones_like(p, dtype=D))
        if adjoint is None:
            continue
        g = adjoint[p] / spp
        ga, gn = torch.autograd.grad((rgb * g).sum(), (a, nn))
        grads["v"].index_add_(0, f.reshape(-1), ga.reshape(-1, 3))
        grads["n"].index_add_(0, f.reshape(-1), gn.reshape(-1, 3))
        if texel is not None:
            idx, wt, k = texel
            grads["tex"].view(-1, 3).index_add_(0, idx.reshape(-1), (wt[..., None] * (g * k[:, None])[:, None]).detach().reshape(-1, 3))
    return (total + plate * (spp - hits)[:, None]) / spp


def _edge_term(view, n, plate, adjoint, ne, ctr1, seed, tex, grads):
    """Adds the silhouette-edge samples' gradient to grads["v"]."""
    mesh, v = view.mesh, view.v
    fn = torch.cross(view.p[:, 1] - view.p[:, 0], view.p[:, 2] - view.p[:, 0], dim=-1)
    w = v[mesh.edges[:, 0]] - view.o
    two = mesh.edge_faces[:, 1] >= 0
    sign = [_dot(fn[mesh.edge_faces[:, k].clamp_min(0)], w) < 0 for k in (0, 1)]
    sil = torch.nonzero(~two | (sign[0] != sign[1]))[:, 0]
    if ne == 0 or len(sil) == 0:
        return
    r0, r1 = _philox(torch.arange(ne, device="cuda"), ctr1, 0, 1, seed)
    e = mesh.edges[sil[(r0 * len(sil)) >> 32]]
    a, b = view.xy[e[:, 0]], view.xy[e[:, 1]]
    x = a + _u24(r1)[:, None] * (b - a)
    normal = torch.stack([a[:, 1] - b[:, 1], b[:, 0] - a[:, 0]], -1)
    length = normal.norm(dim=-1, keepdim=True)
    cell = x.floor().long()
    ok = (length[:, 0] > 0) & (cell >= 0).all(-1) & (cell[:, 0] < view.W) & (cell[:, 1] < view.H)
    e, a, b, x, cell = e[ok], a[ok], b[ok], x[ok], cell[ok]
    off = I.EDGE_EPS_PX * normal[ok] / length[ok]
    lim = torch.tensor([view.W - 1, view.H - 1], device="cuda")
    rgb = []
    for side in (1, -1):
        q = x + side * off
        d = view.direction(q[:, 0], q[:, 1])
        tri = view.closest(cell[:, 1] * view.W + cell[:, 0], d)
        c = torch.minimum(q.floor().long().clamp_min(0), lim)
        out = plate[c[:, 1] * view.W + c[:, 0]].clone()
        h = tri >= 0
        out[h] = view.shade(view.p[tri[h]], n[mesh.faces[tri[h]]], tri[h], d[h], tex)[0]
        rgb.append(out)
    g = _dot(adjoint[cell[:, 1] * view.W + cell[:, 0]], rgb[0] - rgb[1]) * (len(sil) / ne)
    da = g[:, None] * torch.stack([b[:, 1] - x[:, 1], x[:, 0] - b[:, 0]], -1)
    db = g[:, None] * torch.stack([x[:, 1] - a[:, 1], a[:, 0] - x[:, 0]], -1)
    ends = v[e].clone().requires_grad_()
    gv, = torch.autograd.grad((view.project(ends[:, 0]) * da + view.project(ends[:, 1]) * db).sum(), ends)
    grads["v"].index_add_(0, e.reshape(-1), gv.reshape(-1, 3))


def _exact_instance(mesh, x, cams, cfg, plate, seed, instance, adjoint, tex):
    """Image, vertices and (with an adjoint image, or a function of the image that gives one) gradients."""
    x = x.to(D).view(1, 61).requires_grad_(adjoint is not None)
    verts = _skin(x, mesh.arrays)[0]
    v = verts.detach().requires_grad_(adjoint is not None)
    n = _normals(v, mesh.faces)
    shape = (cfg.views, cfg.height * cfg.width, 3)
    plate = plate.view(shape)
    views = [_View(cams[i].to(D), v.detach(), mesh, cfg.height, cfg.width) for i in range(cfg.views)]
    tex = None if tex is None else tex.to(D)
    grads = dict(v=torch.zeros_like(v), n=torch.zeros_like(v), tex=None if tex is None else torch.zeros_like(tex))

    def render(adj):
        return torch.stack([_render(w, n.detach(), plate[i].to(D), cfg.spp, i | instance << 16, seed, tex,
                                    None if adj is None else adj[i], grads) for i, w in enumerate(views)])

    if adjoint is None:
        return render(None), verts
    if callable(adjoint):
        adjoint = adjoint(render(None))
    adjoint = adjoint.to(D).view(shape)
    image = render(adjoint)
    for i, w in enumerate(views):
        _edge_term(w, n.detach(), plate[i].to(D), adjoint[i], cfg.edge_samples, i | instance << 16, seed, tex, grads)
    gv, = torch.autograd.grad((n * grads["n"]).sum(), v)
    d_verts = gv + grads["v"]
    d_params, = torch.autograd.grad((verts * d_verts).sum(), x)
    return image, d_verts, d_params[0], grads["tex"]


def _l1(image, observed, mask, T=None):
    """Masked L1 loss, its adjoint in the image and in the colour transforms."""
    image = image.detach().to(D).requires_grad_()
    t = None if T is None else T.to(D).requires_grad_()
    r = image if T is None else torch.einsum("nij,nhwj->nhwi", t.view(-1, 3, 3), image)
    m = (mask != 0).to(D)
    loss = ((r - observed.to(D)).abs() * m[..., None]).sum() / (3 * m.sum())
    g = torch.autograd.grad(loss, [image] if T is None else [image, t])
    return loss.detach().view(1), g[0], None if T is None else g[1]


def _exact_scene(s, c, seed, given):
    cfg = _config(c["views"], c["width"], c["height"], c["spp"], c["edge_samples"])
    r = s["ref"]
    loss = []

    def from_loss(image):
        out = _l1(image.view(r.image.shape), r.views.observed, r.views.mask)
        loss.append(out[0])
        return out[1]

    image, d_verts, d_params, d_tex = _exact_instance(
        _mesh(c.get("levels", 0)), s["params"], r.views.cams, cfg, r.views.background, 7919 * seed + 17, 0,
        r.adjoint if given else from_loss, s.get("tex"))
    out = dict(image=image.view(r.image.shape), d_verts=d_verts, d_params=d_params)
    if given:
        return dict(out, d_tex=d_tex)
    return dict(out, loss=loss[0])


def _exact_batch(s, c, seed):
    bt, image, rest = s["bt"], torch.empty(s["image"].shape, dtype=D, device="cuda"), []
    for i, cfg in enumerate(_batch_configs(c)):
        sl = slice(int(bt.pixel_offsets[i]), int(bt.pixel_offsets[i + 1]))
        cams = s["cams"][int(bt.view_offsets[i]):int(bt.view_offsets[i + 1])]
        got = _exact_instance(_mesh(0), s["params"][i], cams, cfg, s["plate"][sl], 7919 * seed + 17, i,
                              s["adjoint"][sl] if c["kind"] == "batch" else None, None)
        image[sl] = got[0].view(-1, 3)
        rest.append(got[1:])
    if c["kind"] == "pairs":
        return dict(image=image, verts=torch.stack([r[0] for r in rest]))
    return dict(image=image, d_verts=torch.stack([r[0] for r in rest]), d_params=torch.stack([r[1] for r in rest]))


def _taps(x, taps, dim, zero=False):
    """Correlation along dim of [N][H][W] with symmetric or antisymmetric taps, replicated or zero border."""
    k = len(taps) // 2
    pad = (k, k, 0, 0) if dim == 2 else (0, 0, k, k)
    x = F.pad(x[:, None], pad, mode="constant" if zero else "replicate")[:, 0]
    n = x.shape[dim] - 2 * k
    return sum(w * x.narrow(dim, i, n) for i, w in enumerate(taps))


def _gauss(radius, sigma):
    w = [math.exp(-0.5 * (i / sigma) ** 2) for i in range(-radius, radius + 1)]
    return [x / sum(w) for x in w]


def _edge_map(image, T):
    """Canny's detector on the luma of T R, blurred by the 11 x 11 Gaussian of sigma 5."""
    w = torch.tensor([0.299, 0.587, 0.114], dtype=D, device="cuda")
    luma = torch.einsum("nij,i,nhwj->nhw", T.view(-1, 3, 3), w, image)
    g = _taps(_taps(luma, _gauss(2, 1.0), 2), _gauss(2, 1.0), 1)
    gx = _taps(_taps(g, [0.25, 0.5, 0.25], 1), [-0.5, 0, 0.5], 2)
    gy = _taps(_taps(g, [0.25, 0.5, 0.25], 2), [-0.5, 0, 0.5], 1)
    m = (gx * gx + gy * gy + 1e-12).sqrt()
    with torch.no_grad():
        big = F.pad(m[:, None], (1, 1, 1, 1), mode="replicate")[:, 0]
        H, W = m.shape[1:]
        at = lambda dy, dx: big[:, 1 + dy:1 + dy + H, 1 + dx:1 + dx + W]
        ax, ay, t = gx.abs(), gy.abs(), math.tan(math.pi / 8)
        horizontal, vertical = ay <= t * ax, ax <= t * ay
        rising = gx * gy > 0
        keep = torch.where(horizontal, (m >= at(0, 1)) & (m >= at(0, -1)), torch.where(
            vertical, (m >= at(1, 0)) & (m >= at(-1, 0)), torch.where(
                rising, (m >= at(1, 1)) & (m >= at(-1, -1)), (m >= at(1, -1)) & (m >= at(-1, 1)))))
        cand = keep & (m > B.EDGE_LOW)
        kept, before = cand & (m > B.EDGE_HIGH), -1
        while int(kept.sum()) != before:
            before = int(kept.sum())
            for _ in range(16):
                kept = cand & (F.max_pool2d(kept[:, None].float(), 3, 1, 1)[:, 0] > 0)
    e = torch.where(kept, m, 0.0)
    return _taps(_taps(e, _gauss(5, 5.0), 2, True), _gauss(5, 5.0), 1, True)


def _exact_objective(s, c):
    loss, adjoint, d_t = _l1(s["image"], s["observed"], s["mask"], s["T"])
    image, T = s["image"].to(D).requires_grad_(), s["T"].to(D).requires_grad_()
    m = (s["mask"] != 0).to(D)
    eye = torch.eye(3, dtype=D, device="cuda").expand(len(T), 3, 3)
    target = _edge_map(s["observed"].to(D), eye).detach()
    edge = ((_edge_map(image, T) - target).abs() * m).sum() / m.sum()
    g_image, g_t = torch.autograd.grad(edge, (image, T))
    k = c["texture"] // 8
    low = s["low"].to(D).repeat_interleave(k, 0).repeat_interleave(k, 1)
    return dict(tex=low + s["high"].to(D), loss=loss, edge_loss=edge.detach().view(1), adjoint=adjoint + g_image,
                dT=(d_t + g_t).view(-1, 9), d_low=s["d_tex"].to(D).view(8, k, 8, k, 3).sum((1, 3)))


def _exact_net(s, c, backward):
    n, k = c["n"], c["views"]
    p = s["weights"].to(D).requires_grad_(backward)
    shapes = [(32, 128), (64, 320), (128, 576), (128, 1152), (128, 1152), (256, 2112), (256, 256), (64, 256)]
    layers, at = [], 0
    for rows, cols in shapes:
        layers.append((p[at:at + rows * cols].view(rows, cols), p[at + rows * cols:at + rows * cols + rows]))
        at += rows * cols + rows
    box = lambda x: F.avg_pool2d(x.to(D).permute(0, 3, 1, 2), 2)
    r, o = box(s["image"]), box(s["observed"])
    y = torch.cat([r - o, o, torch.zeros_like(o[:, :2])], 1)
    for (w, b), cin in zip(layers[:5], (8, 32, 64, 128, 128)):
        kernel = w[:, :9 * cin].reshape(-1, 3, 3, cin).permute(0, 3, 1, 2)
        y = F.conv2d(y, kernel, b, stride=2, padding=1).relu()
    cam = s["cams"].to(D)
    z = torch.cat([y.permute(0, 2, 3, 1).reshape(n * k, 2048), cam[:, 4:13], cam[:, 16:19] / 0.6], 1)
    z = F.pad(z, (0, 2112 - z.shape[1]))
    f = (z @ layers[5][0].T + layers[5][1]).relu().view(n, k, 256).amax(1)
    h = (f @ layers[6][0].T + layers[6][1]).relu()
    scale = torch.tensor([0.5] * 10 + [0.1] * 48 + [0.005] * 3, dtype=D, device="cuda")
    delta = (h @ layers[7][0].T + layers[7][1])[:, :61] * scale
    out = (s["base"].to(D) + delta).detach()
    if not backward:
        return out
    return dict(out=out, grads=torch.autograd.grad((delta * s["d_out"].to(D)).sum(), p)[0])


def _overlap(n_in, n_out):
    """[n_out][n_in] shares of each output pixel's footprint."""
    o, i = torch.arange(n_out, device="cuda", dtype=D)[:, None], torch.arange(n_in, device="cuda", dtype=D)[None]
    lo = torch.maximum(o * n_in, i * n_out)
    return (torch.minimum((o + 1) * n_in, (i + 1) * n_out) - lo).clamp_min(0) / n_in


def exact(case, seed):
    c, k = case, case["kind"]
    s = prepare(case, seed)
    if k in ("step", "textured"):
        return _exact_scene(s, c, seed, k == "textured")
    if k in ("batch", "pairs"):
        return _exact_batch(s, c, seed)
    if k == "loss":
        loss, adjoint, _ = _l1(s["image"], s["observed"], s["mask"])
        return dict(loss=loss, adjoint=adjoint)
    if k == "objective":
        return _exact_objective(s, c)
    if k in ("propose", "train"):
        return _exact_net(s, c, k == "train")
    if k == "gemm":
        y = s["a"].to(D) @ s["b"].to(D).T
        y = y if s["bias"] is None else y + s["bias"].to(D)
        return y.relu() if s["relu"] else y
    if k == "geometry":
        x = s["params"].to(D).requires_grad_()
        v = _skin(x, _mesh(0).arrays)
        return dict(verts=v.detach(), d_params=torch.autograd.grad((v * s["d_verts"].to(D)).sum(), x)[0])
    rows, cols = _overlap(c["height"], c["out_h"]), _overlap(c["width"], c["out_w"])
    dst = torch.stack([torch.einsum("yh,hwc,xw->yxc", rows, v.to(D), cols) for v in s["src"]])
    return dict(dst=dst, dmask=None)
