"""Timed cases of the library: what a user's program has it do, through its public entry points.

A case is a dict of plain values.  ``listed()`` gives the fixed ones, ``draw``
another of the same ranges, ``prepare`` a program's state before the call,
``run`` one pass, ``work`` the bytes and operations that a pass cannot do
without, ``exact`` its outputs in 64 bits.

Kinds:
  render   Context.raster_forward of one soup (stochastic, or the deployment threshold)
  train    Context.train_l2: forward, L2 loss and every gradient in one call
  fit      raster.render + l2_stochastic_loss + backward(): the autograd route
  serve    Context.raster_forward_multi: a batch of requests on resident soups
  paper    PaperStep.step: levels, shading, L1 + SSIM, both backwards, optimisers
  shade    Context.shade_forward;  shade_grad  Context.shade_backward
  ssim     native.loss_l1_ssim with its gradients
  adapt    one round of adaptive control: coverage, edge ratios, plan, rebuild
"""
from __future__ import annotations

import math

import numpy as np
import torch

from paper_2603_27151_gb300 import inputs as I
from paper_2603_27151_gb300 import native as N
from paper_2603_27151_gb300.paper_step import PaperStep
from paper_2603_27151_gb300.raster import Rasterizer, l2_stochastic_loss, render

HD, QHD = "1920x1080", "960x540"


def listed():
    return [
        # an interactive preview of a toy soup: the smallest call, all latency
        dict(name="render_tiny", kind="render", T=64, N=4, C=4, S=1, views="64x64", half=False, tile=16, bits=-1),
        # unit-scale fitting (RGB + opacity), the smallest training call
        dict(name="train_tiny", kind="train", T=64, N=4, C=4, S=1, views="64x64", tile=16, bits=-1),
        # a research script through autograd: few triangles, mixed and ragged view sizes, two mask samples
        dict(name="fit_views", kind="fit", T=2000, N=8, C=8, S=2,
             views="128x128,131x97,256x256,256x256,251x255,320x240,320x240,97x61", tile=16, bits=-1),
        # the training loop: 20,000 triangles, four views a step, one sample, default launch parameters
        dict(name="train_20k", kind="train", T=20_000, N=8, C=8, S=1, views="1024x768*4", tile=16, bits=-1),
        # the large training batch: 4 mask samples, mixed resolutions, the launch parameters autotuning picks there
        dict(name="train_1080p", kind="train", T=100_000, N=8, C=8, S=4, views="%s*4,%s*4" % (HD, QHD), tile=8, bits=0),
        # deployment: a large optimised soup at full HD with the fixed threshold
        dict(name="render_hd", kind="render", T=200_000, N=8, C=8, S=1, views=HD, half=True, tile=16, bits=-1),
        # the server's batch: requests of mixed sizes on several resident soups
        dict(name="serve_batch", kind="serve", T=50_000, soups=4, N=8, C=8, S=1,
             views="256x256*4,640x480*4,1280x720*4,%s*4" % HD, tile=16, bits=-1),
        # the paper's whole training step at its scale: level soup, shading, L1 + SSIM, optimisers
        dict(name="paper_step", kind="paper", T=20_000, r_min=2, r_max=5, S=1, views=HD + "*4"),
        # deferred shading of a training step's features, and its backward
        dict(name="shade_fwd", kind="shade", S=2, views="%s*4,1023x577" % HD),
        dict(name="shade_bwd", kind="shade_grad", S=2, views="%s*4,1023x577" % HD),
        # the paper's photometric loss on the shaded images, ragged tiles included
        dict(name="loss_ssim", kind="ssim", S=1, Co=3, views="%s*4,1297x839" % HD),
        # one round of splitting and pruning on a level soup after a threshold render of the views
        dict(name="adapt_round", kind="adapt", T=20_000, r_min=2, r_max=5, views=HD + "*4"),
    ]


# ------------------------------------------------------------------ drawing
def _log(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def _draw_views(rng, n, lo, hi):
    """n views of lo..hi pixels on the longer side, any aspect between square and 16:9, odd sizes among them."""
    out = []
    for _ in range(n):
        w = _log(rng, lo, hi)
        out.append("%dx%d" % (w, max(1, int(w * rng.uniform(0.5625, 1.0)))))
    return ",".join(out)


def draw(rng):
    kind = rng.choice(["render", "train", "train", "fit", "serve", "paper", "shade", "shade_grad", "ssim", "adapt"])
    tune = rng.choice([dict(tile=16, bits=-1), dict(tile=16, bits=-1), dict(tile=8, bits=0), dict(tile=32, bits=0)])
    shape = rng.choice([dict(N=8, C=8), dict(N=8, C=8), dict(N=4, C=4), dict(N=8, C=5), dict(N=16, C=8)])
    if kind == "render":
        T = _log(rng, 64, 200_000)
        return dict(kind=kind, T=T, S=rng.choice([1, 1, 4]), half=rng.random() < 0.5,
                    views=_draw_views(rng, rng.choice([1, 2, 4]), 64, 1920 if T >= 256 else 640), **shape, **tune)
    if kind == "train":   # the handful of triangles covers whole images: small ones
        T = _log(rng, 64, 100_000 if shape["N"] < 16 else 50_000)
        return dict(kind=kind, T=T, S=rng.choice([1, 1, 2, 3, 4]), views=_draw_views(rng, 4, 64, 1600 if T >= 256 else 320),
                    **shape, **tune)
    if kind == "fit":
        return dict(kind=kind, T=_log(rng, 256, 20_000), S=rng.choice([1, 2, 4]), views=_draw_views(rng, 8, 96, 640),
                    **shape, **tune)
    if kind == "serve":
        return dict(kind=kind, T=_log(rng, 10_000, 50_000), soups=rng.choice([1, 4, 8]), N=8, C=8, S=1,
                    views=_draw_views(rng, rng.choice([3, 8, 16]), 256, 1920), tile=16, bits=-1)
    if kind == "paper":
        return dict(kind=kind, T=_log(rng, 2_000, 20_000), r_min=rng.choice([1, 2, 3]), r_max=rng.choice([4, 5]), S=1,
                    views=_draw_views(rng, 4, 320, 1920))
    if kind in ("shade", "shade_grad"):
        return dict(kind=kind, S=rng.choice([1, 2, 3]), views=_draw_views(rng, 4, 128, 1920))
    if kind == "ssim":
        return dict(kind=kind, S=rng.choice([1, 2]), Co=rng.choice([3, 3, 7]), views=_draw_views(rng, 4, 128, 1920))
    return dict(kind=kind, T=_log(rng, 2_000, 20_000), r_min=2, r_max=5, views=_draw_views(rng, 4, 320, 1920))


# ------------------------------------------------------------------ inputs
def _sizes(case):
    out = []
    for part in case["views"].split(","):
        wh, _, n = part.partition("*")
        w, h = wh.split("x")
        out += [(int(w), int(h))] * int(n or 1)
    return out


def _rngs(seed):
    gen = torch.Generator(device="cuda")
    gen.manual_seed(seed)
    return np.random.default_rng(seed), gen


def _cameras(case, rng):
    """Pinholes on a sphere of radius 3 looking at the soup."""
    sizes = _sizes(case)
    return [I.look_at(e, w, h) for e, (w, h) in zip(I.sphere_eyes(len(sizes), 3.0, rng), sizes)]


def _verts(T, rng):
    """The random initialisation; a handful of triangles as large i.i.d. ones."""
    v = I.iid_soup(T, rng) if T < 256 else I.box_soup(T, I.edge_length_for(T), rng)
    return torch.from_numpy(v).cuda()


def _soup(case, rng, gen):
    verts = _verts(case["T"], rng)
    tex = torch.randn((case["T"], I.n_texels(case["N"]), case["C"]), generator=gen, device="cuda")
    return verts, tex


def _levels(case, gen):
    sizes = N.level_sizes(case["T"], case["r_min"], case["r_max"], 8)
    return torch.randn(sum(sizes), generator=gen, device="cuda").div_(math.sqrt(len(sizes)))


def _seeds(rng, n):
    return rng.integers(0, 2 ** 63, size=n, dtype=np.uint64)


def _images(case, channels, gen, S=None):
    """Smooth images with some noise, in [0, 1]: [S, channels, H, W] per view (no S: [channels, H, W])."""
    out = []
    for w, h in _sizes(case):
        shape = (channels, h, w) if S is None else (S, channels, h, w)
        coarse = torch.rand((1 if S is None else S, channels, (h + 31) // 32 + 1, (w + 31) // 32 + 1), generator=gen,
                            device="cuda")
        img = torch.nn.functional.interpolate(coarse, size=(h, w), mode="bilinear", align_corners=True).reshape(shape)
        out.append(img.mul_(0.9).add_(torch.rand(shape, generator=gen, device="cuda"), alpha=0.1).contiguous())
    return out


def _context(case):
    ctx = N.Context(torch.cuda.current_device())
    ctx.set_tuning(tile_w=case["tile"], depth_bits=case["bits"])
    return ctx


def _mlp(gen):
    """MLP parameters after some training: Xavier-scaled weights and small biases."""
    p = torch.randn(595, generator=gen, device="cuda")
    scale = torch.full((595,), 0.1, device="cuda")
    for o, n, width in ((0, 256, 32), (272, 256, 32), (544, 48, 19)):
        scale[o:o + n] = math.sqrt(2.0 / width)
    return p.mul_(scale).contiguous()


# ------------------------------------------------------------------ states
def prepare(case, seed):
    kind = case["kind"]
    rng, gen = _rngs(seed)
    st = dict(case=case, kind=kind)
    if kind in ("render", "train"):
        verts, tex = _soup(case, rng, gen)
        cams = _cameras(case, rng)
        ctx = _context(case)
        S, C = case["S"], case["C"]
        static = kind == "render"
        g, col, _ = N.alloc_outputs(cams, S, C)
        st.update(ctx=ctx, sid=ctx.soup_upload(verts, tex, case["N"], borrow=True, static=static), verts=verts, tex=tex,
                  cams=cams, seeds=_seeds(rng, len(cams)), bg=np.zeros(C - 1, np.float32), g=g, col=col)
        if kind == "train":
            st.update(targets=_images(case, C - 1, gen), gcol=[torch.empty_like(c) for c in col],
                      sw=[torch.empty((S, c.height, c.width), device="cuda") for c in cams],
                      loss=torch.zeros(1, device="cuda"), gv=torch.empty_like(verts), gt=torch.empty_like(tex))
    elif kind == "fit":
        verts, tex = _soup(case, rng, gen)
        cams = _cameras(case, rng)
        rast = Rasterizer(verts.requires_grad_(), tex.requires_grad_(), case["N"])
        rast.ctx.set_tuning(tile_w=case["tile"], depth_bits=case["bits"])
        targets = _images(case, case["C"] - 1, gen)
        st.update(rast=rast, cams=cams, seeds=_seeds(rng, len(cams)), targets=targets)
    elif kind == "serve":
        ctx = _context(case)
        soups, ids = [], []
        for k in range(case["soups"]):   # triangle counts spread over a factor of ten below T
            one = dict(case, T=max(64, int(case["T"] * 10.0 ** (-k / max(1, case["soups"] - 1)))))
            verts, tex = _soup(one, rng, gen)
            soups.append((verts, tex))
            ids.append(ctx.soup_upload(verts, tex, case["N"], borrow=True, static=True))
        cams = _cameras(case, rng)
        g, col, _ = N.alloc_outputs(cams, 1, case["C"])
        st.update(ctx=ctx, soups=soups, ids=[ids[v % len(ids)] for v in range(len(cams))], cams=cams,
                  seeds=_seeds(rng, len(cams)), bg=np.zeros(case["C"] - 1, np.float32), g=g, col=col)
    elif kind == "paper":
        verts = _verts(case["T"], rng)
        cams = _cameras(case, rng)
        ps = PaperStep(verts, _levels(case, gen), case["T"], case["r_min"], case["r_max"], 8, cams,
                       _images(case, 3, gen), S=case["S"], per_step=len(cams), params=_mlp(gen), seed=seed)
        # a run in progress: moments of the size that earlier steps leave
        for k, scale in (("verts", 1e-2), ("tex", 1e-3), ("mlp", 1.0)):
            ps.m[k].normal_(generator=gen).mul_(scale)
            ps.v[k].uniform_(0.5, 1.5, generator=gen).mul_(4.0 * scale * scale)
        ps.step_no = 1000
        st.update(ps=ps)
    elif kind in ("shade", "shade_grad"):
        cams = _cameras(case, rng)
        feats = _images(case, 7, gen, case["S"])
        st.update(ctx=N.Context(torch.cuda.current_device()), cams=cams, params=_mlp(gen), feats=feats)
        if kind == "shade":
            st["rgb"] = [torch.empty_like(f[:, :3]).contiguous() for f in feats]
        else:
            st.update(grgb=[torch.randn(f[:, :3].shape, generator=gen, device="cuda") for f in feats],
                      gfeat=[torch.empty_like(f) for f in feats], gparams=torch.empty(595, device="cuda"))
    elif kind == "ssim":
        col, tgt = _images(case, case["Co"], gen, case["S"]), _images(case, case["Co"], gen)
        st.update(col=col, tgt=tgt, gcol=[torch.empty_like(c) for c in col],
                  sw=[torch.empty_like(c[:, 0]).contiguous() for c in col], loss=torch.zeros(1, device="cuda"))
    else:
        verts, tex = _verts(case["T"], rng), _levels(case, gen)
        cams = _cameras(case, rng)
        ctx = N.Context(torch.cuda.current_device())
        sid = ctx.soup_upload_levels(verts, tex, case["T"], case["r_min"], case["r_max"], 8, borrow=True)
        g, col, _ = N.alloc_outputs(cams, 1, 8)
        ctx.raster_forward(sid, cams, None, 1, N.DS_MODE_THRESHOLD_HALF, np.zeros(7, np.float32), g, col)
        torch.cuda.synchronize()
        st.update(ctx=ctx, verts=verts, tex=tex, cams=cams, g=g)
    return st


# ------------------------------------------------------------------ passes
def _gbuf_parts(gbufs):
    return [dict(zip(("tri", "bary", "depth"), N.split_gbuf(g))) for g in gbufs]


def run(st):
    kind, case = st["kind"], st["case"]
    if kind == "render":
        mode = N.DS_MODE_THRESHOLD_HALF if case["half"] else N.DS_MODE_STOCHASTIC
        st["ctx"].raster_forward(st["sid"], st["cams"], st["seeds"], case["S"], mode, st["bg"], st["g"], st["col"])
        return dict(gbuf=_gbuf_parts(st["g"]), color=st["col"])
    if kind == "train":
        st["loss"].zero_()
        st["ctx"].train_l2(st["sid"], st["cams"], st["seeds"], case["S"], N.DS_MODE_STOCHASTIC, st["bg"], st["g"],
                           st["col"], st["targets"], st["gcol"], st["sw"], 1.0 / case["S"], st["loss"],
                           N.DS_G_ALL | N.DS_OVERWRITE, st["gv"], st["gt"])
        return dict(gbuf=_gbuf_parts(st["g"]), color=st["col"], grad_color=st["gcol"], score_w=st["sw"],
                    loss=st["loss"], grad_verts=st["gv"], grad_tex=st["gt"])
    if kind == "fit":
        rast = st["rast"]
        rast.verts.grad = rast.tex.grad = None
        colors, logps, gbufs = render(rast, st["cams"], st["seeds"], S=case["S"])
        loss = l2_stochastic_loss(colors, logps, st["targets"], case["S"])
        loss.backward()
        return dict(gbuf=_gbuf_parts(gbufs), color=[c.detach() for c in colors], loss=loss.detach(),
                    grad_verts=rast.verts.grad, grad_tex=rast.tex.grad)
    if kind == "serve":
        st["ctx"].raster_forward_multi(st["ids"], st["cams"], st["seeds"], 1, N.DS_MODE_THRESHOLD_HALF, st["bg"],
                                       st["g"], st["col"])
        return dict(gbuf=_gbuf_parts(st["g"]), color=st["col"])
    if kind == "paper":
        ps = st["ps"]
        loss = ps.step()
        return dict(loss=loss, grad_verts=ps.g_verts, grad_mlp=ps.g_params, verts=ps.verts, tex=ps.tex, mlp=ps.params,
                    m_tex=ps.m["tex"], v_tex=ps.v["tex"])
    if kind == "shade":
        st["ctx"].shade_forward(st["cams"], st["params"], st["feats"], st["rgb"])
        return dict(rgb=st["rgb"])
    if kind == "shade_grad":
        st["ctx"].shade_backward(st["cams"], st["params"], st["feats"], st["grgb"], st["gfeat"], st["gparams"],
                                 overwrite=True)
        return dict(grad_feat=st["gfeat"], grad_mlp=st["gparams"])
    if kind == "ssim":
        st["loss"].zero_()
        N.loss_l1_ssim(st["col"], st["tgt"], st["gcol"], st["sw"], st["loss"], lam=0.8, scale=1.0 / case["S"])
        return dict(grad_color=st["gcol"], score_w=st["sw"], loss=st["loss"])
    T, dev = case["T"], st["verts"].device
    counts = torch.zeros(T, dtype=torch.int32, device=dev)
    N.coverage_count(st["g"], T, counts)
    ratios = torch.empty((T, 3), device=dev)
    N.edge_ratios(st["verts"], st["cams"], ratios)
    plan = N.adapt_plan(counts.cpu().numpy(), ratios.cpu().numpy(), 0.02, T)
    n = len(plan)
    levels = range(case["r_min"], case["r_max"] + 1)
    verts = torch.empty((n, 3, 3), device=dev)
    tex = torch.empty(sum(N.level_sizes(n, levels[0], levels[-1], 8)), device=dev)
    st["ctx"].soup_rebuild(st["verts"], st["tex"], T, [1 << R for R in levels], 8, plan, verts, tex)
    return dict(counts=counts, ratios=ratios, plan=plan, verts=verts, tex=tex)


# ------------------------------------------------------------------ work
def work(case):
    """Inputs read once and outputs written once; operations of the dense parts."""
    kind = case["kind"]
    px = sum(w * h for w, h in _sizes(case))
    S = case.get("S", 1)
    if kind in ("render", "train", "fit", "serve"):
        Co, V = case["C"] - 1, I.n_texels(case["N"])
        n = px * S
        soup = case["T"] * (36 + 4 * V * case["C"])
        if kind == "serve":
            soup *= sum(10.0 ** (-k / max(1, case["soups"] - 1)) for k in range(case["soups"]))
        fwd = n * (16 + 4 * Co) + soup
        if kind in ("render", "serve"):
            return dict(bytes=int(fwd), flops=0)
        # target read, upstream gradients and score weights written, both soup gradients written
        return dict(bytes=int(fwd + 4 * px * Co + 4 * n * (Co + 1) + soup), flops=0)
    if kind == "shade":
        return dict(bytes=40 * px * S, flops=1120 * px * S)
    if kind == "shade_grad":
        return dict(bytes=68 * px * S, flops=3072 * px * S)
    if kind == "ssim":
        # colours read, gradients written, target read once, score weights; five moments and three derivative
        # maps blurred by two passes of eleven taps
        return dict(bytes=4 * px * (2 * S * case["Co"] + case["Co"] + S), flops=2 * 176 * px * S * case["Co"])
    level_floats = sum(N.level_sizes(case["T"], case["r_min"], case["r_max"], 8))
    if kind == "paper":
        # levels and both moments read and written, vertices alike, the targets read; the shading both ways
        return dict(bytes=24 * level_floats + case["T"] * 9 * 4 * 5 + 12 * px, flops=(1120 + 3072 + 1056) * px * S)
    # G-buffers read, soup read and rebuilt
    return dict(bytes=16 * px + 2 * (4 * level_floats + 36 * case["T"]), flops=0)


# ------------------------------------------------------------------ 64 bits
def exact(case, seed):
    """The outputs in 64 bits by plain torch.

    Of the rasterised cases only those of a few triangles: every pixel against
    every triangle takes too long beyond.  Vertex gradients (whose boundary
    terms are an estimator over the sampled image) and G-buffers (decided at
    the pixel grid's snapping) have no value of their own there."""
    kind = case["kind"]
    if kind == "shade":
        return _exact_shade(prepare(case, seed), False)
    if kind == "shade_grad":
        return _exact_shade(prepare(case, seed), True)
    if kind == "ssim":
        return _exact_ssim(prepare(case, seed))
    if kind == "adapt":
        st = prepare(case, seed)
        return dict(counts=None, ratios=_exact_ratios(st["verts"].double(), st["cams"]), plan=None, verts=None, tex=None)
    if kind in ("render", "train") and case["T"] <= 128 and sum(w * h for w, h in _sizes(case)) <= 1 << 16:
        return _exact_raster(prepare(case, seed))
    return None


def _f64(x):
    return torch.as_tensor(np.asarray(x, np.float32), device="cuda").double()


def _sh(cam):
    """The nine real spherical harmonics of degree <= 2 of every pixel's ray: [9, H, W]."""
    y, x = torch.meshgrid(torch.arange(cam.height, device="cuda").double() + 0.5,
                          torch.arange(cam.width, device="cuda").double() + 0.5, indexing="ij")
    fx, fy, cx, cy = (float(np.float32(v)) for v in (cam.fx, cam.fy, cam.cx, cam.cy))
    d = torch.stack([(x - cx) / fx, (y - cy) / fy, torch.ones_like(x)])
    x, y, z = torch.einsum("ki,khw->ihw", _f64(cam.R), d / d.norm(dim=0, keepdim=True))
    c1, c2, c0 = math.sqrt(3 / (4 * math.pi)), math.sqrt(15 / (4 * math.pi)), math.sqrt(1 / (4 * math.pi))
    return torch.stack([torch.full_like(x, c0), -c1 * y, c1 * z, -c1 * x, c2 * x * y, -c2 * y * z,
                        math.sqrt(5 / (16 * math.pi)) * (2 * z * z - x * x - y * y), -c2 * x * z,
                        c2 / 2 * (x * x - y * y)])


def _exact_shade(st, grads):
    p = st["params"].double()
    W1, b1, W2, b2, W3, b3 = (p[a:b].reshape(s) for a, b, s in (
        (0, 256, (16, 16)), (256, 272, (16, 1)), (272, 528, (16, 16)), (528, 544, (16, 1)), (544, 592, (3, 16)),
        (592, 595, (3, 1))))
    rgb, gfeat, gp = [], [], torch.zeros(595, dtype=torch.float64, device="cuda")
    for v, (cam, feat) in enumerate(zip(st["cams"], st["feats"])):
        sh = _sh(cam).reshape(9, -1)
        for s in range(feat.shape[0]):
            f = feat[s].double().reshape(7, -1)
            x = torch.cat([f, sh])
            h1 = (W1 @ x + b1).relu_()
            h2 = (W2 @ h1 + b2).relu_()
            o = torch.sigmoid(W3 @ h2 + b3)
            A = f[3]
            if not grads:
                rgb.append((A * f[:3] + (1 - A) * o).reshape(3, cam.height, cam.width))
                continue
            g = st["grgb"][v][s].double().reshape(3, -1)
            d3 = (1 - A) * g * o * (1 - o)
            d2 = (W3.T @ d3) * (h2 > 0)
            d1 = (W2.T @ d2) * (h1 > 0)
            gf = (W1.T @ d1)[:7]
            gf[:3] += A * g
            gf[3] += (g * (f[:3] - o)).sum(0)
            gfeat.append(gf.reshape(7, cam.height, cam.width))
            gp += torch.cat([t.reshape(-1) for t in (d1 @ x.T, d1.sum(1), d2 @ h1.T, d2.sum(1), d3 @ h2.T, d3.sum(1))])
    S = st["case"]["S"]
    stack = lambda ts: [torch.stack(ts[k:k + S]) for k in range(0, len(ts), S)]
    return dict(grad_feat=stack(gfeat), grad_mlp=gp) if grads else dict(rgb=stack(rgb))


def _exact_ssim(st):
    k = torch.arange(-5, 6, dtype=torch.float64, device="cuda")
    w = torch.exp(-k * k / (2 * 1.5 ** 2))
    w = w / w.sum()

    def blur(a):
        for dim in (-1, -2):
            pad = torch.nn.functional.pad(a, (5, 5, 0, 0) if dim == -1 else (0, 0, 5, 5))
            a = sum(w[j] * pad.narrow(dim, j, a.shape[dim]) for j in range(11))
        return a

    lam, S, Co = 0.8, st["case"]["S"], st["case"]["Co"]
    total, gcol, sws = 0.0, [], []
    for col, tgt in zip(st["col"], st["tgt"]):
        g, ell = [], []
        for s in range(S):
            e, gs = 0.0, []
            for c in range(Co):
                x, y = col[s, c].double(), tgt[c].double()
                mx, my = blur(x), blur(y)
                a, b = 2 * mx * my + 1e-4, 2 * (blur(x * y) - mx * my) + 9e-4
                cc, d = mx * mx + my * my + 1e-4, blur(x * x) - mx * mx + blur(y * y) - my * my + 9e-4
                ssim = a * b / (cc * d)
                var, cov = -ssim / d, 2 * a / (cc * d)
                mu = 2 * my * b / (cc * d) - 2 * mx * ssim / cc - 2 * mx * var - my * cov
                back = blur(mu) + 2 * x * blur(var) + y * blur(cov)
                gs.append((lam * torch.sign(x - y) - (1 - lam) * back) / (Co * S))
                e = e + (lam * (x - y).abs() + (1 - lam) * (1 - ssim)) / (Co * S)
            g.append(torch.stack(gs))
            ell.append(e)
        gcol.append(torch.stack(g))
        sws.append(torch.stack(ell))
        total = total + sws[-1].sum()
    return dict(grad_color=gcol, score_w=sws, loss=total.reshape(1))


def _exact_ratios(verts, cams):
    best = torch.zeros((verts.shape[0], 3), dtype=torch.float64, device="cuda")
    for c in cams:
        p = verts @ _f64(c.R).T + _f64(c.t)
        s = p[..., :2] / p[..., 2:] * _f64([c.fx, c.fy]) + _f64([c.cx, c.cy])
        seen = (p[..., 2] > c.near).all(1) & (s.amax(1) > 0).all(1) & (s.amin(1) < _f64([c.width, c.height])).all(1)
        r = (s.roll(-1, 1) - s).norm(dim=-1) / c.height
        best = torch.where(seen[:, None], torch.maximum(best, r), best)
    return best


def _philox(px, py, t, seed):
    """First word of Philox4x32-10 of counter (px, py, t, 0), key = the seed's halves, on the grid of [0, 1)."""
    m = 0xFFFFFFFF
    c = [px.long(), py.long(), t.long(), torch.zeros_like(px.long())]
    k0, k1 = int(seed) & m, int(seed) >> 32

    def mulhilo(a, x):   # a * x of 32 bits each in 63-bit integers, by halves of a
        lo, hi = (a & 0xFFFF) * x, (a >> 16) * x
        mid = hi + (lo >> 16)
        return (mid >> 16) & m, ((mid & 0xFFFF) << 16) | (lo & 0xFFFF)

    for _ in range(10):
        h0, l0 = mulhilo(0xD2511F53, c[0])
        h1, l1 = mulhilo(0xCD9E8D57, c[2])
        c = [h1 ^ c[1] ^ k0, l1, h0 ^ c[3] ^ k1, l0]
        k0, k1 = (k0 + 0x9E3779B9) & m, (k1 + 0xBB67AE85) & m
    return (c[0] >> 8).double() * 2.0 ** -24


def _exact_raster(st):
    """Every pixel against every triangle (one mask sample), at vertices snapped to 1/256 pixel."""
    case = st["case"]
    Ng, Co = case["N"], case["C"] - 1
    if case["S"] != 1:
        return None
    T, dev = case["T"], "cuda"
    act = torch.sigmoid(st["tex"].double())
    gtex = torch.zeros_like(act)
    verts, total = st["verts"].double(), 0.0
    colors, gcols, sws = [], [], []
    tri = torch.arange(T, device=dev)
    for v, cam in enumerate(st["cams"]):
        p = verts @ _f64(cam.R).T + _f64(cam.t)
        z = p[..., 2]
        s = p[..., :2] / z[..., None] * _f64([cam.fx, cam.fy]) + _f64([cam.cx, cam.cy])
        drawn = (z > float(np.float32(cam.near))).all(1) & (s.abs() <= 16384).all(2).all(1)
        X = torch.round(torch.where(drawn[:, None, None], s, torch.zeros_like(s)) * 256).long()
        area = (X[:, 1, 0] - X[:, 0, 0]) * (X[:, 2, 1] - X[:, 0, 1]) - (X[:, 2, 0] - X[:, 0, 0]) * (X[:, 1, 1] - X[:, 0, 1])
        drawn &= area != 0
        py, px = torch.meshgrid(torch.arange(cam.height, device=dev), torch.arange(cam.width, device=dev), indexing="ij")
        px, py = px.reshape(-1, 1), py.reshape(-1, 1)
        cover, q = drawn[None, :].expand(px.shape[0], T).clone(), []
        for i in range(3):
            j, k = (i + 1) % 3, (i + 2) % 3
            a, b = torch.sign(area) * (X[:, j, 1] - X[:, k, 1]), torch.sign(area) * (X[:, k, 0] - X[:, j, 0])
            e = a * (256 * px + 128 - X[:, j, 0]) + b * (256 * py + 128 - X[:, j, 1])
            owns = (a > 0) | ((a == 0) & (b > 0))
            cover &= (e > 0) | ((e == 0) & owns)
            q.append(e.double() / z[:, i] / area.abs().clamp(min=1))
        rho = q[0] + q[1] + q[2]
        b1, b2 = q[1] / rho, q[2] / rho
        ci = (Ng * b1).floor().clamp(0, Ng - 1).nan_to_num().long()
        cj = torch.minimum((Ng * b2).floor().clamp(min=0).nan_to_num().long(), Ng - 1 - ci).clamp(min=0)
        fu, fv = Ng * b1 - ci, Ng * b2 - cj
        low = (fu + fv <= 1) | (ci + cj == Ng - 1)
        at = lambda i, j: j * (Ng + 1) - j * (j - 1) // 2 + i
        up = (~low).long()
        ks = torch.stack([at(ci + up, cj + up), at(ci + 1 - up, cj + up), at(ci + up, cj + 1 - up)])
        wa, wb = torch.where(low, fu, 1 - fu), torch.where(low, fv, 1 - fv)
        ws = torch.stack([1 - wa - wb, wa, wb])
        alpha = sum(ws[m] * act[tri, ks[m].clamp(0, act.shape[1] - 1), -1] for m in range(3))
        tau = 0.5 if case.get("half") else _philox(px.expand_as(b1), py.expand_as(b1), tri.expand_as(b1), st["seeds"][v])
        key = torch.where(cover & (alpha > tau), rho, torch.full_like(rho, -math.inf))
        best, t = key.max(1)
        hit = best > -math.inf
        rows = torch.arange(len(t), device=dev)
        kw, ww = ks[:, rows, t], torch.where(hit, ws[:, rows, t], torch.zeros(3, len(t), dtype=torch.float64, device=dev))
        kw = torch.where(hit, kw, torch.zeros_like(kw))
        col = sum(ww[m][:, None] * act[t, kw[m], :Co] for m in range(3))
        colors.append(col.T.reshape(1, Co, cam.height, cam.width))
        if st["kind"] == "render":
            continue
        diff = col - st["targets"][v].double().reshape(Co, -1).T
        ell = (diff ** 2).sum(1)
        total = total + ell.sum()
        gcols.append((2 * diff).T.reshape(1, Co, cam.height, cam.width))
        sws.append(ell.reshape(1, cam.height, cam.width))
        # colour and +w/alpha at the winner, -w/(1 - alpha) at what lies in front of it
        up_win = torch.cat([2 * diff, torch.where(hit, ell / alpha[rows, t], torch.zeros_like(ell))[:, None]], 1)
        for m in range(3):
            a = act[t, kw[m]]
            gtex.index_put_((t, kw[m]), up_win * ww[m][:, None] * a * (1 - a), accumulate=True)
        r, f = torch.nonzero(cover & (rho > torch.where(hit, best, torch.full_like(best, -math.inf))[:, None]), as_tuple=True)
        g = -ell[r] / (1 - alpha[r, f])
        for m in range(3):
            k = ks[m][r, f]
            a = act[f, k, -1]
            gtex.index_put_((f, k, torch.full_like(f, Co)), g * ws[m][r, f] * a * (1 - a), accumulate=True)
    none = [dict(tri=None, bary=None, depth=None) for _ in colors]
    if st["kind"] == "render":
        return dict(gbuf=none, color=colors)
    return dict(gbuf=none, color=colors, grad_color=gcols, score_w=sws, loss=total.reshape(1), grad_verts=None,
                grad_tex=gtex)
