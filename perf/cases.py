"""Performance cases of the training step: what a program using this package
runs, over the range of sizes it is used at.

A case is a dict of plain values; `prepare` makes what the program holds
before the call (scene buffers, plan and workspace, targets), `run` makes one
pass through the public entry points, `work` counts the bytes and operations
one pass cannot do without, `exact` restates small passes in plain float64.

Kinds:
  step      one training step, Trainer.step (eager) or Trainer.replay (graph)
  render    Trainer.forward alone: evaluation images, no backward
  autograd  Renderer.render and its backward to the stored parameters
  ssim      gs_loss_l1_ssim or its masked form: loss gradient of given images
  l1        gs_loss_l1_noalloc: L1 loss and gradient without a plan
  densify   gs_densify_count, _counts and _apply into new buffers
"""
from __future__ import annotations

import math

import numpy as np
import torch
import torch.nn.functional as F

from paper_2605_00219_gb300 import autograd, gsstep, step, synth

DEV = "cuda"
# late-training rates (a hundredth of the initial ones): repeated passes leave
# the scene's statistics as they are
LR = tuple(0.01 * x for x in step.DEFAULT_LR)
ADAM_STEP = 1000                       # steps taken before the measured one
B1, B2, EPS = 0.9, 0.999, 1e-15        # make_adam's defaults

HD = "1920x1080"
UNEVEN = ",".join(f"{w}x{h}" for w, h in synth.BATCH_RESOLUTIONS)


def listed():
    return [
        # The smallest training step: a test-sized scene, one small view, each
        # stage called eagerly.  Launches and host calls are most of it.
        {"name": "tiny_step", "kind": "step", "scene": "uniform", "sizes": "2000", "views": "128x128",
         "bf16": False, "graph": False, "loss": "l1", "threads": 0},
        # The smallest differentiable render: the same scene inside a torch
        # program (a loss of its own, an optimiser of its own).
        {"name": "tiny_autograd", "kind": "autograd", "scene": "uniform", "sizes": "2000", "views": "128x128",
         "bf16": False},
        # An ordinary small training run: 200k Gaussians, one 720p view a step,
        # the step replayed as a graph.
        {"name": "mid_step_graph", "kind": "step", "scene": "room", "sizes": "200000", "views": "1280x720",
         "bf16": False, "graph": True, "loss": "l1", "threads": 0},
        # Evaluation of a held-out view during such a run; a ragged image size.
        {"name": "mid_render_ragged", "kind": "render", "scene": "room", "sizes": "200000", "views": "1237x822"},
        # The plain form: 3M Gaussians, FP32 storage, one 1080p view a step.
        {"name": "plain_step_1080p", "kind": "step", "scene": "site", "sizes": "3000000", "views": HD,
         "bf16": False, "graph": False, "loss": "l1", "threads": 0},
        # The headline: four 1080p views a step, BF16 storage, one graph, the
        # launch shape the autotuner picks.
        {"name": "batched_step_bf16", "kind": "step", "scene": "site", "sizes": "3000000",
         "views": ",".join([HD] * 4), "bf16": True, "graph": True, "loss": "l1", "threads": 128},
        # The paper's loss (L1 + SSIM against 8-bit references, alpha masked)
        # on a batch of views of different resolutions, one million Gaussians.
        {"name": "ssim_masked_step", "kind": "step", "scene": "site", "sizes": "1000000", "views": UNEVEN,
         "bf16": True, "graph": False, "loss": "l1_ssim_masked", "threads": 128},
        # Several scenes in one differentiable render and backward, BF16
        # coefficients: the largest working set.
        {"name": "multiscene_autograd", "kind": "autograd", "scene": "site",
         "sizes": ",".join(str(n) for n in synth.MULTI_SIZES), "views": f"{HD},960x540", "bf16": True},
        # The loss gradient alone on a 1080p batch, for a program that renders
        # by other means or computes several losses.
        {"name": "ssim_loss_1080p", "kind": "ssim", "views": ",".join([HD] * 4), "masked": False},
        # The same on one small, ragged image.
        {"name": "ssim_loss_ragged", "kind": "ssim", "views": "403x301", "masked": True},
        # The L1 gradient for a frame loop that may not allocate.
        {"name": "l1_noalloc_1080p", "kind": "l1", "pixels": 1920 * 1080},
        # One refinement of the default strategy, as a training run does every
        # hundred steps.
        {"name": "densify_3m", "kind": "densify", "sizes": "3000000", "bf16": True},
    ]


def _log(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def _views(rng, n, lo, hi):
    out = []
    for _ in range(n):
        w = _log(rng, lo, hi)
        out.append(f"{w}x{max(16, int(w * rng.uniform(0.5, 0.8)))}")
    return ",".join(out)


def draw(rng):
    kind = rng.choice(["step", "step", "step", "render", "autograd", "ssim", "l1", "densify"])
    if kind == "ssim":
        return {"kind": kind, "views": _views(rng, rng.randint(1, 4), 65, 1920), "masked": rng.random() < 0.5}
    if kind == "l1":
        return {"kind": kind, "pixels": _log(rng, 4096, 4 * 1920 * 1080)}
    if kind == "densify":
        return {"kind": kind, "sizes": str(_log(rng, 2000, 3_000_000)), "bf16": rng.random() < 0.5}
    if rng.random() < 0.25:      # small scenes, small views
        scene, sizes, views = "uniform", str(_log(rng, 500, 8000)), _views(rng, 1, 64, 256)
    elif rng.random() < 0.5:     # one room, 10 m
        scene, sizes = "room", str(_log(rng, 20_000, 400_000))
        views = _views(rng, rng.randint(1, 3), 320, 1600)
    else:                        # a 30 m site
        scene, sizes = "site", str(_log(rng, 100_000, 2_500_000))
        views = _views(rng, rng.randint(1, 4), 480, 1920)
    if kind == "render":
        return {"kind": kind, "scene": scene, "sizes": sizes, "views": views}
    bf16 = rng.random() < 0.5
    if kind == "autograd":
        if scene == "site":
            sizes += "," + str(_log(rng, 100_000, 1_000_000))
        return {"kind": kind, "scene": scene, "sizes": sizes, "views": views, "bf16": bf16}
    return {"kind": kind, "scene": scene, "sizes": sizes, "views": views, "bf16": bf16, "graph": rng.random() < 0.5,
            "loss": rng.choice(["l1", "l1", "l1_ssim", "l1_ssim_masked"]), "threads": rng.choice([0, 128])}


# --------------------------------------------------------------------------
# Inputs, drawn on the device from the seed (synth.py's recipes)
# --------------------------------------------------------------------------

def _sizes(case):
    return [int(x) for x in case["sizes"].split(",")]


def _shapes(case):
    return [tuple(int(a) for a in v.split("x")) for v in case["views"].split(",")]


def _gen(seed):
    return torch.Generator(device=DEV).manual_seed(int(seed))


def _means(scene, n, g):
    if scene == "uniform":
        return 2.0 * torch.rand((n, 3), device=DEV, generator=g) - 1.0
    box = 10.0 if scene == "room" else 30.0
    c = 64 if scene == "room" else 256
    centres = (torch.rand((c, 3), device=DEV, generator=g) - 0.5) * box
    sd = (0.1 + 1.4 * torch.rand((c, 3), device=DEV, generator=g)).sqrt()
    q = torch.randn((c, 4), device=DEV, generator=g)
    rot = _rotation(q)
    which = torch.randint(0, c, (n,), device=DEV, generator=g)
    z = torch.randn((n, 3), device=DEV, generator=g) * sd[which]
    return (rot[which] * z[:, None, :]).sum(-1) + centres[which]


def _rotation(q):
    w, x, y, z = (q / q.norm(dim=-1, keepdim=True)).unbind(-1)
    return torch.stack([1 - 2 * (y * y + z * z), 2 * (x * y - w * z), 2 * (x * z + w * y),
                        2 * (x * y + w * z), 1 - 2 * (x * x + z * z), 2 * (y * z - w * x),
                        2 * (x * z - w * y), 2 * (y * z + w * x), 1 - 2 * (x * x + y * y)], -1).view(-1, 3, 3)


def _scene(scene, n, g, bf16, moment_scale=None):
    """SceneBuffers of n Gaussians; with moment_scale, Adam moments as they
    are in mid-training (v near the squared gradient scale, m below it)."""
    ls, lo = ((-3.5, 0.5), (0.0, 1.0)) if scene == "uniform" else ((-4.0, 0.7), (-1.0, 1.5))
    geom = torch.zeros((3, n, 4), device=DEV)
    geom[0, :, :3] = _means(scene, n, g)
    q = torch.randn((n, 4), device=DEV, generator=g)
    geom[1] = q / q.norm(dim=1, keepdim=True)
    geom[2, :, :3] = torch.exp(ls[0] + ls[1] * torch.randn((n, 3), device=DEV, generator=g))
    geom[2, :, 3] = torch.sigmoid(lo[0] + lo[1] * torch.randn((n,), device=DEV, generator=g))
    # flat coefficient 3 k + c; the first three are degree 0
    sh = 0.05 * torch.randn((12, n, 4), device=DEV, generator=g)
    sh[0, :, :3] *= 10.0
    if bf16:
        sh = sh.view(6, 2, n, 4).permute(0, 2, 1, 3).reshape(6, n, 8).to(torch.bfloat16)
    m = v = None
    if moment_scale is not None:
        mdt = torch.bfloat16 if bf16 else torch.float32
        m = (0.2 * moment_scale * torch.randn((15, n, 4), device=DEV, generator=g))
        v = moment_scale * moment_scale * torch.exp(torch.randn((15, n, 4), device=DEV, generator=g))
        m[0, :, 3] = 0.0
        v[0, :, 3] = 0.0
        m, v = m.to(mdt), v.to(mdt)
    return step.SceneBuffers(n, geom, sh.contiguous(), m, v)


def _cameras(scene, shapes, index=0, phase=0.0):
    if scene == "uniform":
        return [synth.Camera(np.eye(3, dtype=np.float32), np.array([0, 0, 4], np.float32), 150.0 * w / 128.0,
                             150.0 * w / 128.0, w / 2.0, h / 2.0, w, h, index) for w, h in shapes]
    out = []
    for i, (w, h) in enumerate(shapes):
        out += synth.orbit_cameras(1, 12.0 if scene == "room" else 36.0, w, h, scene=index,
                                   phase_deg=phase + 360.0 * i / len(shapes))
    return out


def _images(shapes, g, rgba=False):
    """A (pixels, 3) float image in [0, 1] per view, concatenated: smooth
    colour with noise, as a photograph against a partly fitted render; with
    rgba the 8-bit reference with an alpha that is 0, 255 or a ramp between."""
    parts = []
    for w, h in shapes:
        x = torch.linspace(0, 1, w, device=DEV)[None, :, None]
        y = torch.linspace(0, 1, h, device=DEV)[:, None, None]
        f = 2.0 + 10.0 * torch.rand((3, 2), device=DEV, generator=g)
        ph = 6.28 * torch.rand((3,), device=DEV, generator=g)
        im = 0.5 + 0.35 * torch.sin(f[:, 0] * x + f[:, 1] * y + ph)
        im = (im + 0.08 * torch.randn((h, w, 3), device=DEV, generator=g)).clamp(0, 1)
        if rgba:
            ramp = (3.0 * (x + y) - 1.0).clamp(0, 1).expand(h, w, 1)
            im = torch.cat([im, ramp], -1).mul(255.0).round().to(torch.uint8)
        parts.append(im.reshape(h * w, -1))
    return torch.cat(parts).contiguous()


class _State:
    pass


def prepare(case, seed):
    s = _State()
    s.case, g = case, _gen(seed)
    kind = case["kind"]
    if kind in ("step", "render"):
        shapes = _shapes(case)
        pixels = sum(w * h for w, h in shapes)
        sizes, bf16 = _sizes(case), bool(case.get("bf16", False))
        scenes = [_scene(case["scene"], n, g, bf16, 5.0 / (3 * pixels)) for n in sizes]
        cams = _cameras(case["scene"], shapes)
        s.tr = step.Trainer(scenes, cams, sh_bf16=bf16, mom_bf16=bf16, lr=LR, loss=case.get("loss", "l1"),
                            threads_per_tile=case.get("threads", 0), seed=int(seed) & 0x7FFFFFFF)
        if kind == "step":
            s.tr.target.copy_(_images(shapes, g, rgba=s.tr.loss != "l1"))
            gsstep.gs_workspace_set_step(s.tr.plan, s.tr.ws, ADAM_STEP)
            if case["graph"]:
                s.tr.capture()
    elif kind == "autograd":
        shapes, sizes, bf16 = _shapes(case), _sizes(case), bool(case["bf16"])
        cams = []
        for k in range(len(sizes)):
            cams += _cameras(case["scene"], shapes, k, 45.0 * k)
        s.r = autograd.Renderer(sizes, cams, sh_bf16=bf16)
        s.params = []
        for n in sizes:
            b = _scene(case["scene"], n, g, bf16)
            s.params += [b.geom.requires_grad_(), b.sh.requires_grad_()]
        pixels = sum(w * h for w, h in shapes) * len(sizes)
        s.dl = torch.randn((pixels, 3), device=DEV, generator=g) / (3 * pixels)
    elif kind == "ssim":
        shapes = _shapes(case)
        s.plan = gsstep.Plan([1], [(w, h, 0) for w, h in shapes])
        s.ws = torch.empty(s.plan.workspace_bytes(), dtype=torch.uint8, device=DEV)
        gsstep.gs_workspace_init(s.plan, s.ws)
        s.image, s.target = _images(shapes, g), _images(shapes, g, rgba=True)
        s.dl = torch.empty_like(s.image)
    elif kind == "l1":
        s.image = torch.rand((case["pixels"], 3), device=DEV, generator=g)
        s.target = torch.rand((case["pixels"], 3), device=DEV, generator=g)
        s.dl, s.loss = torch.empty_like(s.image), torch.empty(1, device=DEV)
    else:
        n, bf16 = _sizes(case)[0], bool(case["bf16"])
        s.sb = _scene("site", n, g, bf16, 1e-6)
        # the same numbers of each fate for every seed: 3% faint enough to be
        # pruned, 6% above the gradient threshold and small (cloned), 4% above
        # it and large (split)
        cnt = torch.randint(1, 40, (n,), device=DEV, generator=g).float()
        mean = 1.9e-4 * torch.rand((n,), device=DEV, generator=g)
        who = torch.randperm(n, device=DEV, generator=g)
        faint, small, large = who[:3 * n // 100], who[3 * n // 100:9 * n // 100], who[9 * n // 100:13 * n // 100]
        mean[small] += 2.5e-4
        mean[large] += 2.5e-4
        sc, op = s.sb.geom[2, :, :3], s.sb.geom[2, :, 3]
        op.clamp_(min=0.006)
        op[faint] = 0.004
        sc[small] = sc[small].clamp(max=0.019)
        sc[large, 0] = sc[large, 0].clamp(min=0.021)
        s.sb.stats = torch.stack([mean * cnt, cnt], 1).contiguous()
        s.eps = torch.randn((n, 6), device=DEV, generator=g)
        s.cfg = gsstep.make_densify_cfg(2.0)
    return s


def run(s):
    case = s.case
    kind = case["kind"]
    if kind == "step":
        tr = s.tr
        if case["graph"]:
            tr.replay()
        else:
            tr.step(0)
        sb = tr.scenes
        return {"image": tr.image, "geom": [b.geom for b in sb], "sh": [b.sh for b in sb], "m": [b.m for b in sb],
                "v": [b.v for b in sb]}
    if kind == "render":
        return {"image": s.tr.forward()}
    if kind == "autograd":
        img = s.r.render([(s.params[2 * k], s.params[2 * k + 1]) for k in range(len(s.params) // 2)])
        grads = torch.autograd.grad(img, s.params, grad_outputs=s.dl)
        return {"image": img.detach(), "grads": list(grads)}
    if kind == "ssim":
        call = gsstep.gs_loss_l1_ssim_masked if case["masked"] else gsstep.gs_loss_l1_ssim
        call(s.plan, s.ws, s.image, s.target, 0.2, s.dl)
        return {"dl": s.dl}
    if kind == "l1":
        gsstep.gs_loss_l1_noalloc(s.image, s.target, s.dl, s.loss)
        return {"dl": s.dl, "loss": s.loss}
    sb, flags = s.sb, s.sb.storage_flags
    scratch = torch.empty(gsstep.gs_densify_scratch_bytes(sb.n), dtype=torch.uint8, device=DEV)
    gsstep.gs_densify_count(sb, flags, s.cfg, scratch)
    counts = gsstep.gs_densify_counts(scratch)
    out = step.SceneBuffers.empty_like_layout(sb, counts[3])
    gsstep.gs_densify_apply(sb, flags, s.cfg, s.eps, scratch, out)
    return {"geom": out.geom, "sh": out.sh, "m": out.m, "v": out.v, "stats": out.stats,
            "counts": torch.tensor(counts)}


# --------------------------------------------------------------------------
# Work that a pass cannot do without
# --------------------------------------------------------------------------

# Tile intersections and blended pixels of one (view, Gaussian) pair, as
# counted for each scene recipe: intersections a pair, and blends a pair at
# 1920 pixels of image width (fewer where a pixel is covered early).
TILES_PER_PAIR = {"uniform": 2.0, "room": 2.0, "site": 1.4}
BLENDS_PER_PAIR = {"uniform": 13500.0, "room": 250.0, "site": 38.0}
MAX_BLENDS_PER_PIXEL = 40.0


def work(case):
    kind = case["kind"]
    if kind == "ssim":
        px = sum(w * h for w, h in _shapes(case))
        # render, reference, gradient; 8 separable 11-tap windows a channel
        return {"bytes": 28.0 * px, "flops": 3.0 * px * (2 * 8 * 22 + 66)}
    if kind == "l1":
        return {"bytes": 36.0 * case["pixels"], "flops": 9.0 * case["pixels"]}
    row = 48 + (96 if case.get("bf16") else 192)
    if kind == "densify":
        n, mom = _sizes(case)[0], 120 if case["bf16"] else 240
        return {"bytes": 2.0 * n * (row + 2 * mom) + 48.0 * n, "flops": 30.0 * n}
    shapes, sizes = _shapes(case), _sizes(case)
    n, px = float(sum(sizes)), float(sum(w * h for w, h in shapes))
    per_scene = px * (len(sizes) if kind == "autograd" else 1)
    pairs = n * len(shapes)
    scale = sum((w / 1920.0) ** 2 for w, h in shapes) / len(shapes)
    isect = pairs * TILES_PER_PAIR[case["scene"]]
    blend = min(pairs * BLENDS_PER_PAIR[case["scene"]] * scale, MAX_BLENDS_PER_PIXEL * per_scene)
    # projection: parameters in, a record out a pair; a key and value written
    # and read an intersection; 12 bytes out a pixel; 14 + 13 operations a
    # blended pair
    nbytes = n * row + 48.0 * pairs + 16.0 * isect + 12.0 * per_scene
    flops = pairs * 250.0 + blend * 2 * 27.0
    if kind == "render":
        return {"bytes": nbytes, "flops": flops}
    # loss (target in, gradient out), backward of every blended pair, its
    # record written and read, the parameters' gradients
    nbytes += 36.0 * per_scene + 72.0 * isect
    flops += blend * 2 * 45.0 + pairs * 450.0
    if kind == "autograd":
        return {"bytes": nbytes + 2.0 * n * row, "flops": flops}
    mom = 120 if case["bf16"] else 240
    nbytes += n * (2 * row + 4.0 * mom)
    if case["loss"] != "l1":
        flops += 3.0 * px * (2 * 8 * 22 + 66)
    return {"bytes": nbytes, "flops": flops}


# --------------------------------------------------------------------------
# Plain float64 restatements
# --------------------------------------------------------------------------

def _sh_basis(d):
    x, y, z = d.unbind(-1)
    xx, yy, zz = x * x, y * y, z * z
    return torch.stack([
        torch.full_like(x, 0.5 * math.sqrt(1 / math.pi)),
        -math.sqrt(3 / (4 * math.pi)) * y, math.sqrt(3 / (4 * math.pi)) * z, -math.sqrt(3 / (4 * math.pi)) * x,
        0.5 * math.sqrt(15 / math.pi) * x * y, -0.5 * math.sqrt(15 / math.pi) * y * z,
        0.25 * math.sqrt(5 / math.pi) * (2 * zz - xx - yy), -0.5 * math.sqrt(15 / math.pi) * x * z,
        0.25 * math.sqrt(15 / math.pi) * (xx - yy),
        -0.25 * math.sqrt(35 / (2 * math.pi)) * y * (3 * xx - yy), 0.5 * math.sqrt(105 / math.pi) * x * y * z,
        -0.25 * math.sqrt(21 / (2 * math.pi)) * y * (4 * zz - xx - yy),
        0.25 * math.sqrt(7 / math.pi) * z * (2 * zz - 3 * xx - 3 * yy),
        -0.25 * math.sqrt(21 / (2 * math.pi)) * x * (4 * zz - xx - yy),
        0.25 * math.sqrt(105 / math.pi) * z * (xx - yy),
        -0.25 * math.sqrt(35 / (2 * math.pi)) * x * (xx - 3 * yy)], -1)


def _dense_pixels(geom, sh, w, h, chunk):
    """Yields (first pixel, rendered pixels) of the camera at z = -4 looking
    along z: every pixel over all Gaussians, nearest first."""
    f, dev = 150.0 * w / 128.0, geom.device
    mu, q, sc, op = geom[0, :, :3], geom[1], geom[2, :, :3], geom[2, :, 3]
    t = mu + torch.tensor([0.0, 0.0, 4.0], dtype=mu.dtype, device=dev)
    tz = t[:, 2]
    M = _rotation(q) * sc[:, None, :]
    limx, limy = 1.3 * 0.5 * w / f, 1.3 * 0.5 * h / f
    ux, uy = (t[:, 0] / tz).clamp(-limx, limx), (t[:, 1] / tz).clamp(-limy, limy)
    z0 = torch.zeros_like(tz)
    T = torch.stack([torch.stack([f / tz, z0, -f * ux / tz], -1), torch.stack([z0, f / tz, -f * uy / tz], -1)], 1)
    J = T @ M
    cov = J @ J.transpose(1, 2)
    a, b, c = cov[:, 0, 0] + 0.3, cov[:, 0, 1], cov[:, 1, 1] + 0.3
    det = a * c - b * b
    mx, my = f * t[:, 0] / tz + w / 2.0, f * t[:, 1] / tz + h / 2.0
    d = t / t.norm(dim=1, keepdim=True)          # the camera is at t = 0
    col = (0.5 + (_sh_basis(d)[:, :, None] * sh.permute(1, 0, 2).reshape(-1, 16, 3)).sum(1)).clamp_min(0.0)
    order = torch.argsort(tz.detach(), stable=True)
    order = order[(tz.detach()[order] >= 0.01) & (255.0 * op.detach()[order] > 1.0)]
    mx, my, A, B, C, op, col = (v[order] for v in (mx, my, c / det, -b / det, a / det, op, col))
    for p0 in range(0, w * h, chunk):
        p = torch.arange(p0, min(p0 + chunk, w * h), device=dev)
        dx, dy = (p % w + 0.5)[:, None] - mx[None], (torch.div(p, w, rounding_mode="floor") + 0.5)[:, None] - my[None]
        d2 = A * dx * dx + 2.0 * B * dx * dy + C * dy * dy
        raw = op * torch.exp(-0.5 * d2)
        with torch.no_grad():
            al = torch.where((d2 <= 9.0) & (raw >= 1.0 / 255.0), raw.clamp_max(0.99), 0.0)
            keep = (al > 0.0) & (torch.cumprod(1.0 - al, 1) >= 1e-4)
        al = torch.where(keep, raw.clamp_max(0.99), 0.0)
        tr = torch.cumprod(1.0 - al, 1)
        before = torch.cat([torch.ones_like(tr[:, :1]), tr[:, :-1]], 1)
        yield p0, (al * before) @ col


def _exact_render(geom, sh, w, h, dl_of):
    """Image, and gradients with respect to geom and sh of the loss whose
    image gradient is dl_of(first pixel, pixels); leaves of their own."""
    geom, sh = geom.detach().double().requires_grad_(), sh.detach().double().requires_grad_()
    out = []
    for p0, px in _dense_pixels(geom, sh, w, h, max(64, 4_000_000 // geom.shape[1])):
        out.append(px.detach())
        if dl_of is not None:
            px.backward(dl_of(p0, px.detach()), retain_graph=True)
    return torch.cat(out), geom.grad, sh.grad


def _ssim_dl(image, target, w, h, masked, lam=0.2, total=None):
    """Gradient of (1 - lam) mean|x - y| + lam (1 - mean SSIM) for one view."""
    y = target.view(h, w, 4).double() / 255.0
    m = y[..., 3:] if masked else torch.ones_like(y[..., 3:])
    leaf = image.view(h, w, 3).double().requires_grad_()
    x, y = leaf * m, y[..., :3] * m
    k = torch.exp(-(torch.arange(11, device=image.device, dtype=torch.float64) - 5) ** 2 / (2 * 1.5 ** 2))
    k = k / k.sum()

    def window(u):
        u = u.permute(2, 0, 1)[:, None]
        u = F.pad(u, (5, 5, 5, 5))
        u = sum(k[i] * u[..., i:i + w] for i in range(11))
        return sum(k[i] * u[:, :, i:i + h] for i in range(11))[:, 0].permute(1, 2, 0)

    mx, my = window(x), window(y)
    vx, vy, cxy = window(x * x) - mx * mx, window(y * y) - my * my, window(x * y) - mx * my
    c1, c2 = 0.01 ** 2, 0.03 ** 2
    ssim = (2 * mx * my + c1) * (2 * cxy + c2) / ((mx * mx + my * my + c1) * (vx + vy + c2))
    n = 3.0 * total
    loss = (1 - lam) * (x - y).abs().sum() / n + lam * (3.0 * w * h - ssim.sum()) / n
    return torch.autograd.grad(loss, leaf)[0].reshape(-1, 3)


def _adam64(sb, geom, ggrad, shgrad, t):
    """One Adam step in float64 from the stored buffers: (geom, sh, m, v)."""
    th = torch.cat([geom, sb["sh"]])
    g = torch.cat([ggrad, shgrad])
    so, o = geom[2, :, :3], geom[2, :, 3]
    th[2, :, :3], th[2, :, 3] = so.log(), torch.log(o / (1.0 - o))
    g[2, :, :3], g[2, :, 3] = g[2, :, :3] * so, g[2, :, 3] * o * (1.0 - o)
    g[0, :, 3] = 0.0
    m, v = B1 * sb["m"] + (1 - B1) * g, B2 * sb["v"] + (1 - B2) * g * g
    lr = torch.full_like(th, LR[5])
    lr[0], lr[1], lr[2, :, :3], lr[2, :, 3] = LR[0], LR[1], LR[2], LR[3]
    lr[3, :, :3] = LR[4]
    th = th - lr * (m / (1 - B1 ** t)) / ((v / (1 - B2 ** t)).sqrt() + EPS)
    m[0, :, 3], v[0, :, 3] = sb["m"][0, :, 3], sb["v"][0, :, 3]
    out = th[:3].clone()
    out[0, :, 3] = geom[0, :, 3]
    out[2, :, :3], out[2, :, 3] = th[2, :, :3].exp(), torch.sigmoid(th[2, :, 3])
    return out, th[3:], m, v


def _exact_densify(s):
    """Clone, split and prune in the order of gs_densify_apply."""
    sb, n, dev = s.sb, s.sb.n, DEV
    g = sb.geom.double()
    thr = 2e-4, np.float32(0.01) * np.float32(2.0), 0.005
    avg = sb.stats[:, 0] / sb.stats[:, 1].clamp_min(1.0)
    top = sb.geom[2, :, :3].amax(1)
    high, small = avg > thr[0], top <= torch.tensor(float(thr[1]), device=dev)
    low = sb.geom[2, :, 3] < thr[2]
    clone, split = high & small & ~low, high & ~small & ~low
    keep = ~(high & ~small) & ~low
    ik, ic, isp = (torch.nonzero(x)[:, 0] for x in (keep, clone, split))
    src = torch.cat([ik, ic, isp, isp])
    geom = g[:, src].clone()
    first = len(ik) + len(ic)
    R = _rotation(g[1, isp])
    for k in range(2):
        at = slice(first + k * len(isp), first + (k + 1) * len(isp))
        e = s.eps[isp, 3 * k:3 * k + 3].double()
        geom[0, at, :3] += (R @ (g[2, isp, :3] * e)[:, :, None])[:, :, 0]
        geom[2, at, :3] = g[2, isp, :3] / 1.6
    m, v = sb.m[:, src].double(), sb.v[:, src].double()
    m[:, len(ik):] = 0.0
    v[:, len(ik):] = 0.0
    return {"geom": geom, "sh": sb.sh[:, src].double(), "m": m, "v": v, "stats": None, "counts": None}


def exact(case, seed):
    kind = case["kind"]
    if kind in ("step", "render", "autograd"):
        if case["scene"] != "uniform" or case.get("bf16") or case.get("loss", "l1") != "l1":
            return None
        (w, h), n = _shapes(case)[0], _sizes(case)[0]
        s = prepare(dict(case, graph=False), seed)
        if kind == "render":
            sb = s.tr.scenes[0]
            return {"image": _exact_render(sb.geom, sb.sh, w, h, None)[0]}
        if kind == "autograd":
            image, gg, gs = _exact_render(s.params[0], s.params[1], w, h, lambda p, px: s.dl[p:p + len(px)].double())
            return {"image": image, "grads": [gg, gs]}
        sb, tgt = s.tr.scenes[0], s.tr.target.double()
        image, gg, gs = _exact_render(sb.geom, sb.sh, w, h,
                                      lambda p, px: torch.sign(px - tgt[p:p + len(px)]) / (3.0 * w * h))
        b64 = {"sh": sb.sh.double(), "m": sb.m.double(), "v": sb.v.double()}
        geom, sh, m, v = _adam64(b64, sb.geom.double(), gg, gs, ADAM_STEP + 1)
        return {"image": image, "geom": [geom], "sh": [sh], "m": [m], "v": [v]}
    s = prepare(case, seed)
    if kind == "ssim":
        total, o, out = sum(w * h for w, h in _shapes(case)), 0, []
        for w, h in _shapes(case):
            out.append(_ssim_dl(s.image[o:o + w * h], s.target[o:o + w * h], w, h, case["masked"], total=total))
            o += w * h
        return {"dl": torch.cat(out)}
    if kind == "l1":
        d = s.image.double() - s.target.double()
        return {"dl": torch.sign(d) / d.numel(), "loss": d.abs().mean().reshape(1)}
    return _exact_densify(s)
