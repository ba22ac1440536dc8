"""The workloads whose speed this repository is measured by.

Each case is one call (or the short fixed sequence of calls) that a program
using the framework makes over and over: a render, the geometry stage, the
compositing passes on their own, a training step, an opacity-guided training
iteration, a set of ground-truth images.  `prepare` makes what such a program
holds before the call, `run` makes the call, `work` counts what the call
cannot do without, and `exact` gives the same results in 64-bit arithmetic
from the method's equations in plain torch.
"""
from __future__ import annotations

import math

import numpy as np
import torch
import torch.nn.functional as F

from paper_2504_13339_gb300 import _lib, scenes
from paper_2504_13339_gb300.render import SplatPipeline, headlight_dirs, lut_tensor
from paper_2504_13339_gb300.train import (OpacityGuidedTrainer, TrainParams, default_lr,
                                          opacity_guided_luts)

DEV = "cuda"
MAPS = 10             # opacity maps of the guided training and of the ground truth
CELL = 8              # vertex cells per macrocell of the empty-space mask
MATERIAL = (0.3, 0.6, 0.25, 12.0)
LAMBDA = 0.2          # SSIM weight of the training loss


def listed():
    return [
        # the smallest call: a thumbnail of a small model (latency and launches count)
        dict(name="render_thumbnail", kind="render", n=4096, blobs=0, width=128, height=128,
             views=1, tfs=1),
        # an interactive viewer's frame: one mid-sized model, one view, one table
        dict(name="render_frame", kind="render", n=500_000, blobs=16, width=512, height=512,
             views=1, tfs=1),
        # a server's batch: several small ragged views of one model in one call
        dict(name="render_batch_ragged", kind="render", n=200_000, blobs=16, width=257,
             height=193, views=5, tfs=1),
        # exploring transfer functions: one sort of a large model, sixteen tables, a large image
        dict(name="render_sweep", kind="render", n=3_000_000, blobs=32, width=2048, height=2048,
             views=1, tfs=16),
        # projection, binning and sort alone: the training scene's view
        dict(name="geometry_1m", kind="geometry", n=1_000_000, blobs=8, width=1024, height=1024,
             views=1, tfs=4),
        # the same for a batched launch: a large model, several views of an odd size
        dict(name="geometry_views", kind="geometry", n=3_000_000, blobs=16, width=1601,
             height=1199, views=2, tfs=4),
        # compositing of the training scene, forward and backward each on their own
        dict(name="composite_fwd", kind="composite_fwd", n=1_000_000, blobs=8, width=1024,
             height=1024, views=1, tfs=4),
        dict(name="composite_bwd", kind="composite_bwd", n=1_000_000, blobs=8, width=1024,
             height=1024, views=1, tfs=4),
        # the training step under several tables (the benchmark's default workload)
        dict(name="train_step", kind="train", n=1_000_000, blobs=8, width=1024, height=1024,
             views=1, tfs=4, lit=False),
        # a shaded training step over several small views of an odd size
        dict(name="train_views_lit", kind="train", n=300_000, blobs=8, width=641, height=479,
             views=3, tfs=2, lit=True),
        # one iteration of the paper's training: shaded, one map, L1 + SSIM, Adam
        dict(name="guided_iteration", kind="guided", n=500_000, blobs=8, width=800, height=800,
             views=1, tfs=MAPS),
        # ground-truth images for training: the raymarched volume under ten maps
        dict(name="ground_truth", kind="march", res=256, blobs=8, width=800, height=800, views=3,
             tfs=MAPS),
    ]


def draw(rng):
    def spread(lo, hi):
        return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))

    kind = rng.choice(["render", "render", "geometry", "composite_fwd", "composite_bwd", "train",
                       "train", "guided", "march"])
    w = spread(64, 1600)
    h = max(48, min(1600, int(w * rng.uniform(0.6, 1.5))))
    if kind == "march":
        return dict(kind=kind, res=spread(48, 256), blobs=8, width=min(w, 800),
                    height=min(h, 800), views=rng.randint(1, 3), tfs=rng.randint(1, MAPS))
    if kind == "guided":
        return dict(kind=kind, n=spread(20_000, 600_000), blobs=8, width=min(w, 900),
                    height=min(h, 900), views=1, tfs=MAPS)
    if rng.random() < 0.15:  # a small model: uniform points, a small image
        n, blobs, w, h = spread(500, 8192), 0, min(w, 256), min(h, 256)
    else:
        n, blobs = spread(20_000, 2_000_000), rng.choice([8, 16, 32])
    views, tfs = rng.randint(1, 5), rng.choice([1, 1, 2, 3, 4, 5, 8])
    # no dearer than the listed calls: pixels x tables x depth of the lists
    most = 2.0e9 if kind == "render" else 0.5e9
    while views > 1 and (views * n > 4_000_000 or views * tfs * w * h * n ** (1 / 3) > most):
        views -= 1
    while tfs > 1 and views * tfs * w * h * n ** (1 / 3) > most:
        tfs -= 1
    case = dict(kind=kind, n=n, blobs=blobs, width=w, height=h, views=views, tfs=tfs)
    if kind == "train":
        case["lit"] = rng.random() < 0.4
    return case


# ---------------------------------------------------------------------------
# inputs
# ---------------------------------------------------------------------------

def _rng(seed, what):
    g = torch.Generator(device=DEV)
    g.manual_seed(seed * 16 + what)
    return g


def _field_value(bf, pts):
    """The blob field at pts (N, 3), float64."""
    out = torch.zeros(pts.shape[0], dtype=torch.float64, device=DEV)
    for k in range(len(bf.amp)):
        d = (pts - torch.as_tensor(bf.center[k], device=DEV)) @ torch.as_tensor(bf.rot[k],
                                                                              device=DEV)
        q = (d / torch.as_tensor(bf.sigma[k], device=DEV)).square().sum(1)
        out += float(bf.amp[k]) * torch.exp(-0.5 * q)
    return out


def _points(n, bf, gen):
    """n points of [-1,1]^3 with the field's density (mixture sampling)."""
    mass = torch.as_tensor(bf.amp * np.prod(bf.sigma, axis=1), device=DEV)
    center, rot, sigma = (torch.as_tensor(a, device=DEV) for a in (bf.center, bf.rot, bf.sigma))
    got = torch.empty(0, 3, dtype=torch.float64, device=DEV)
    while got.shape[0] < n:
        m = int((n - got.shape[0]) * 1.3) + 1024
        k = torch.multinomial(mass, m, replacement=True, generator=gen)
        z = torch.randn(m, 3, generator=gen, device=DEV, dtype=torch.float64) * sigma[k]
        x = torch.einsum("mij,mj->mi", rot[k], z) + center[k]
        got = torch.cat([got, x[(x.abs() <= 1).all(1)]])
    return got[:n]


def _model(case, seed):
    """(mean_v, logscale_w, quat): a fitted model's Gaussians (means where the
    field is dense, about half the mean spacing wide), a small uniform one
    (blobs = 0), or the start of a training (weights 0.1)."""
    n, gen = case["n"], _rng(seed, 1)
    rand = lambda *s: torch.rand(*s, generator=gen, device=DEV, dtype=torch.float64)
    randn = lambda *s: torch.randn(*s, generator=gen, device=DEV, dtype=torch.float64)
    weight = 1.0
    if case["blobs"] == 0:
        pts, v, mu = rand(n, 3) * 2 - 1, rand(n), -3.5
    else:
        bf = scenes.blob_field(case["blobs"], seed)
        if case["kind"] == "guided":
            pts, weight = rand(n, 3) * 2 - 1, 0.1
        else:
            pts = _points(n, bf, gen)
        f = _field_value(bf, pts)
        v, mu = (f / f.max()).clamp(0, 1), math.log(0.5 * 2.0 / n ** (1 / 3))
    ls = mu + 0.3 * randn(n, 3)
    q = F.normalize(randn(n, 4), dim=1)
    w = torch.full((n, 1), weight, dtype=torch.float64, device=DEV)
    return [torch.cat(p, 1).float().contiguous() for p in ((pts, v[:, None]), (ls, w), (q,))]


def _lighting(n, seed):
    """(normal_beta, k_ads): random normals, the material of a training's start."""
    gen = _rng(seed, 2)
    nrm = F.normalize(torch.randn(n, 3, generator=gen, device=DEV, dtype=torch.float64), dim=1)
    nb = torch.cat([nrm, torch.full((n, 1), 10.0, dtype=torch.float64, device=DEV)], 1).float()
    k = torch.tensor([0.3, 0.6, 0.2, 0.0], device=DEV).repeat(n, 1)
    return nb.contiguous(), k.contiguous()


def _cameras(case, seed):
    return scenes.orbit_cameras(case["views"], seed, case["width"], case["height"])


def _tables(case, seed):
    if case["kind"] in ("guided", "march"):
        return lut_tensor(opacity_guided_luts(MAPS, scenes.colour_ramp(seed))[:case["tfs"]], DEV)
    return lut_tensor(scenes.bump_tfs(case["tfs"], seed), DEV)


def _image(case, seed, images):
    """A smooth target [V][images][H][W][4] (the loss's cost and the density
    of its gradient do not depend on what it shows)."""
    gen = _rng(seed, 3)
    low = torch.rand(case["views"] * images, 4, 9, 9, generator=gen, device=DEV)
    up = F.interpolate(low, size=(case["height"], case["width"]), mode="bilinear",
                       align_corners=True)
    up = up.permute(0, 2, 3, 1).contiguous() * 0.6
    return up.view(case["views"], images, case["height"], case["width"], 4)


def _upstream(case, seed):
    """The gradient of a mean L1 loss: +-1/(3 pixels) on RGB, 0 on T."""
    d = torch.sign(_image(case, seed, case["tfs"]) - 0.3)
    d[..., 3] = 0
    return d / (3 * d.numel() // 4)


def _volume(case, seed):
    """The blob field on the R^3 vertices of [-1,1]^3 ([z][y][x]), normalised."""
    R = case["res"]
    bf = scenes.blob_field(case["blobs"], seed)
    x = torch.linspace(-1, 1, R, dtype=torch.float64, device=DEV)
    z, y, x = torch.meshgrid(x, x, x, indexing="ij")
    f = _field_value(bf, torch.stack([x.reshape(-1), y.reshape(-1), z.reshape(-1)], 1))
    return (f / f.max()).float().view(R, R, R).contiguous()


# ---------------------------------------------------------------------------
# the calls
# ---------------------------------------------------------------------------

class _State:
    pass


def _capacity(case):
    """Tile instances to hold, from the sizes alone: each Gaussian's 3-sigma
    square at the orbit's distance, with room for nearer and wider ones."""
    sigma = case["n"] ** (-1 / 3) * case["width"] * 1.207 / 3
    if case["blobs"] == 0:
        sigma = 0.03 * case["width"] * 1.207 / 3
    per = (6 * 1.4 * sigma / 16 + 1) ** 2
    return int(1.6 * per * case["n"] * case["views"]) + (1 << 16)


def _guided_lr():
    """Learning rates late in a schedule: the model hardly moves, so that
    every iteration costs the same however many are run."""
    return default_lr() * 1e-4


def prepare(case, seed):
    s = _State()
    s.kind = case["kind"]
    cams = _cameras(case, seed)
    s.luts = _tables(case, seed)
    if s.kind == "march":
        R = case["res"]
        s.vol4 = torch.empty(R, R, R, 4, device=DEV)
        _lib.veg_volume_prepare(_volume(case, seed), s.vol4)
        s.R, s.step = R, (2.0 / (R - 1)) / 2
        s.mask = torch.empty(_lib.veg_raymarch_cells_count(R, CELL), dtype=torch.int32, device=DEV)
        s.cams = [_lib.cameras([c]) for c in cams]
        s.out = torch.empty(case["views"], case["tfs"], case["height"], case["width"], 4,
                            device=DEV)
        return s
    s.tens = _model(case, seed)
    if s.kind == "guided":
        g = scenes.Gaussians(*(t.cpu().numpy() for t in s.tens))
        lit = scenes.Lighting(*(t.cpu().numpy() for t in _lighting(case["n"], seed)))
        targets = _image(case, seed, MAPS)
        s.map = MAPS // 3
        s.trainer = OpacityGuidedTrainer(TrainParams(g, lit), cams, s.luts, targets,
                                         lr=_guided_lr(), seed=seed, capacity=16 * case["n"])
        s.trainer.render(0, s.map)
        _, m = s.trainer.pipe.status()
        s.trainer.pipe.set_capacity(int(m * 1.25) + 4096)
        return s
    s.pipe = SplatPipeline(case["n"], cams, n_tf=case["tfs"], device=DEV)
    if s.kind == "geometry":  # the whole list buffer is an output: one size for every seed
        s.pipe.set_capacity(_capacity(case))
        s.pipe.vals.zero_()
        return s
    s.pipe.render(*s.tens, s.luts)  # a first frame: sizes the instance capacity
    s.pipe.set_capacity(int(s.pipe.status()[1] * 1.25) + 4096)
    s.lighting = None
    if s.kind in ("composite_fwd", "composite_bwd"):
        s.pipe.render(*s.tens, s.luts)
        if s.kind == "composite_bwd":
            s.dout = _upstream(case, seed)
    elif s.kind == "train":
        s.target = _image(case, seed, case["tfs"])
        s.grads = [torch.zeros_like(t) for t in s.tens]
        if case["lit"]:
            s.lighting = _lighting(case["n"], seed) + (headlight_dirs(cams).astype(np.float32),)
            s.grads += [torch.zeros_like(t) for t in s.lighting[:2]]
    return s


def run(s):
    if s.kind == "march":  # one mask per table set, one launch per view
        tf = _lib.tf_desc(s.luts)
        _lib.veg_raymarch_cells(s.vol4, tf, CELL, s.mask)
        for v, cam in enumerate(s.cams):
            _lib.veg_raymarch_masked(cam, s.vol4, tf, s.step, s.out[v:v + 1], s.mask, CELL,
                                     MATERIAL)
        return {"out": s.out}
    if s.kind == "guided":
        t = s.trainer
        t.step(0, s.map)
        return {"loss": t.loss, "out": t.pipe.out, "grads": t.P.grads, "raw": t.P.raw,
                "m": t.P.m, "v": t.P.v, "mean_v": t.P.mean_v, "logscale_w": t.P.logscale_w}
    p = s.pipe
    if s.kind == "render":
        return {"out": p.render(*s.tens, s.luts)}
    if s.kind == "geometry":
        p.project(*s.tens, s.luts)
        p.bin_sort()
        return {"geo": p.geo, "aux": p.aux, "tiles": p.tiles, "rect": p.rect,
                "vals": p.vals, "ranges": p.ranges}
    if s.kind == "composite_fwd":
        return {"out": p.composite(s.luts), "n_contrib": p.n_contrib}
    if s.kind == "composite_bwd":
        p.backward_2d(s.dout)
        return {"grad2d": p.grad2d}
    loss = p.train_step(*s.tens, s.luts, s.target, s.grads, lighting=s.lighting)
    return {"loss": loss, "out": p.out, "grads": s.grads}


# ---------------------------------------------------------------------------
# what a call cannot do without
# ---------------------------------------------------------------------------

# Splats blended per pixel and table before a pixel is done, in units of the
# cube root of the Gaussians (the lists deepen with it): measured on the
# training scene with the compositor's own pair counts.
BLENDED = 0.53


def work(case):
    px, V, T = case["width"] * case["height"], case["views"], case["tfs"]
    if case["kind"] == "march":
        R = case["res"]
        # each volume vertex once, each image once; a ray crosses about 0.35
        # of the volume's steps where some table has opacity
        return {"bytes": 16.0 * R ** 3 + 16.0 * V * T * px,
                "flops": V * px * 0.1 * 2 * R * (98.0 + 2 * 28.0)}
    n = case["n"]
    images = V * (1 if case["kind"] == "guided" else T)
    pairs = images * px * BLENDED * n ** (1 / 3)
    model, records, pixels = 48.0 * n, 56.0 * n * V, 16.0 * images * px
    if case["kind"] == "render":
        return {"bytes": model + pixels, "flops": 27 * pairs + 200.0 * n * V}
    if case["kind"] == "geometry":
        return {"bytes": model + records + 4.0 * 9 * n * V, "flops": 200.0 * n * V}
    if case["kind"] == "composite_fwd":
        return {"bytes": 32.0 * n * V + 4.0 * 9 * n * V + pixels * 1.25, "flops": 27 * pairs}
    if case["kind"] == "composite_bwd":
        return {"bytes": 64.0 * n * V + 4.0 * 9 * n * V + pixels * 2.25, "flops": 59 * pairs}
    step = {"bytes": 2 * model + 2 * pixels, "flops": 86 * pairs + 800.0 * n * V}
    if case["kind"] == "guided":  # five packed arrays: parameter, two moments, gradient
        return {"bytes": n * 5 * 16 * 7.0 + 2 * pixels, "flops": step["flops"] + 520 * 3 * px}
    if case["lit"]:
        step["bytes"] += 64.0 * n
    return step


# ---------------------------------------------------------------------------
# the same results in 64 bits
# ---------------------------------------------------------------------------

A_MIN, A_MAX, T_MIN = 1 / 255, 0.99, 1e-4


def _tf64(luts, v):
    """Tables at v: (value, slope) [T][N][4] of the linear interpolation."""
    L = luts.shape[1]
    p = v.clamp(0, 1) * (L - 1)
    k = p.floor().clamp(max=L - 2).long()
    lo, hi = luts[:, k], luts[:, k + 1]
    inside = ((v >= 0) & (v <= 1)).to(luts.dtype)[:, None]
    return lo + (hi - lo) * (p - k)[:, None], (hi - lo) * (L - 1) * inside


def _project64(cam, mean, ls, q, v, w, luts):
    """One view: screen means, depths, conics (a, b, c), tile rectangles and
    which Gaussians touch a tile."""
    R = torch.as_tensor(cam.world_to_cam, dtype=torch.float64, device=DEV)
    t = mean @ R[:, :3].T + R[:, 3]
    ok = (t[:, 2] > float(np.float32(cam.near))) & (q.square().sum(1) > 0)
    z = torch.where(ok, t[:, 2], torch.ones_like(t[:, 2]))
    xr, yr = t[:, 0] / z, t[:, 1] / z
    u = torch.stack([cam.fx * xr + cam.cx, cam.fy * yr + cam.cy], 1)
    lx, ly = 1.3 * 0.5 * cam.width / cam.fx, 1.3 * 0.5 * cam.height / cam.fy
    xc, yc, zero = xr.clamp(-lx, lx), yr.clamp(-ly, ly), torch.zeros_like(z)
    J = torch.stack([torch.stack([cam.fx / z, zero, -cam.fx * xc / z], 1),
                     torch.stack([zero, cam.fy / z, -cam.fy * yc / z], 1)], 1)
    a, b, c, d = F.normalize(q, dim=1).unbind(1)
    rot = torch.stack([1 - 2 * (c * c + d * d), 2 * (b * c - a * d), 2 * (b * d + a * c),
                       2 * (b * c + a * d), 1 - 2 * (b * b + d * d), 2 * (c * d - a * b),
                       2 * (b * d - a * c), 2 * (c * d + a * b), 1 - 2 * (b * b + c * c)],
                      1).view(-1, 3, 3)
    M = J @ R[:, :3] @ (rot * torch.exp(ls)[:, None, :])
    S = M @ M.transpose(1, 2)
    sa, sb, sc = S[:, 0, 0] + 0.3, S[:, 0, 1], S[:, 1, 1] + 0.3
    det = sa * sc - sb * sb
    conic = torch.stack([sc, -sb, sa], 1) / det[:, None]
    with torch.no_grad():
        m = 0.5 * (sa + sc)
        rad = (3 * (m + (m * m - det).clamp(min=0.1).sqrt()).sqrt()).ceil()[:, None]
        lo, hi = (u - rad).ceil(), (u + rad).floor()
        last = torch.tensor([cam.width - 1, cam.height - 1], dtype=torch.float64, device=DEV)
        ok = ok & (lo <= hi).all(1) & (lo <= last).all(1) & (hi >= 0).all(1)
        ok = ok & ((_tf64(luts, v)[0][..., 3] * w) >= A_MIN).any(0)
        r0 = (lo.clamp(min=0) / 16).floor().long()
        r1 = (torch.minimum(hi, last) / 16).floor().long() + 1
    return u, t[:, 2], conic, r0, r1, ok


def _lists64(cam, depth, r0, r1, ok):
    """(record per instance, first instance per tile): each tile's records by depth."""
    idx = torch.nonzero(ok).squeeze(1)
    idx = idx[torch.argsort(depth[idx], stable=True)]
    wx = (r1 - r0)[idx, 0]
    cnt = wx * (r1 - r0)[idx, 1]
    rec = torch.repeat_interleave(idx, cnt)
    at = torch.arange(rec.numel(), device=DEV) - torch.repeat_interleave(cnt.cumsum(0) - cnt, cnt)
    wr = torch.repeat_interleave(wx, cnt)
    tile = (r0[rec, 1] + at // wr) * cam.tiles_x + r0[rec, 0] + at % wr
    order = torch.argsort(tile, stable=True)
    first = torch.zeros(cam.tiles_x * cam.tiles_y + 1, dtype=torch.int64, device=DEV)
    first[1:] = torch.bincount(tile, minlength=first.numel() - 1).cumsum(0)
    return rec[order], first


def _tiles64(cam, rec, first, budget=1 << 17):
    """Batches of tiles of similar list lengths: (tile ids, records [B][L],
    valid [B][L], pixel coordinates [B][256][2])."""
    length = first[1:] - first[:-1]
    order = torch.argsort(length, descending=True)
    host, i = length[order].tolist(), 0
    px = torch.arange(256, device=DEV)
    while i < len(host) and host[i] > 0:
        k = max(1, budget // host[i])
        ids = order[i:i + k][length[order[i:i + k]] > 0]
        pos = torch.arange(host[i], device=DEV)[None]
        valid = pos < length[ids][:, None]
        r = rec[(first[ids][:, None] + pos).clamp(max=rec.numel() - 1)]
        x = (ids % cam.tiles_x)[:, None] * 16 + px % 16
        y = (ids // cam.tiles_x)[:, None] * 16 + px // 16
        yield ids, r, valid, torch.stack([x, y], 2)
        i += k


def _pairs64(u, conic, w, r, valid, xy):
    """Offsets and the Gaussian of every (splat, pixel) pair [B][L][256]."""
    d = u[r][:, :, None, :] - xy[:, None].double()
    c = conic[r][:, :, None, :]
    power = -0.5 * (c[..., 0] * d[..., 0] ** 2 + c[..., 2] * d[..., 1] ** 2) \
        - c[..., 1] * d[..., 0] * d[..., 1]
    G = torch.exp(power) * (valid[:, :, None] & (power <= 0))
    return d, G


def _alpha64(aw, G):
    """alpha (0 where the pair is skipped or behind the stop) and the
    transmittance behind it."""
    alpha = (aw[:, :, None] * G).clamp(max=A_MAX)
    alpha = alpha * (alpha >= A_MIN)
    behind = torch.cumprod(1 - alpha, 1)
    on = behind >= T_MIN
    return alpha * on, torch.where(on, behind, torch.ones_like(behind)), on


def _splat64(case, seed, tens, luts, shade=None, loss=None, upstream=None):
    """The render of every view in 64 bits and, given `loss` (out -> scalar)
    or `upstream` (dL/dout), the screen-space gradients [V][n][8] (and those
    of the shading factors [V][n][2]).  `tens` are the leaves (mean, v,
    log-scale, w, quaternion); returns also each view's (u, conic) graph."""
    mean, v, ls, w, q = tens
    cams, luts = _cameras(case, seed), luts.double()
    V, T, W, H = len(cams), luts.shape[0], case["width"], case["height"]
    out = torch.zeros(V, T, H, W, 4, dtype=torch.float64, device=DEV)
    out[..., 3] = 1
    graphs, lists = [], []
    val, slope = _tf64(luts, v.detach())
    wd = w.detach()

    def colours(view, t, r):
        col = val[t][r]
        if shade is None:
            return col[..., :3], col[..., 3] * wd[r]
        sd = shade[view].detach()[r]
        return col[..., :3] * sd[..., :1] + sd[..., 1:], col[..., 3] * wd[r]

    for view, cam in enumerate(cams):
        u, depth, conic, r0, r1, ok = _project64(cam, mean, ls, q, v.detach(), wd, luts)
        graphs.append((u, conic, depth, ok))
        lists.append(_lists64(cam, depth.detach(), r0, r1, ok))
        ud, cd = u.detach(), conic.detach()
        for ids, r, valid, xy in _tiles64(cam, *lists[view]):
            _, G = _pairs64(ud, cd, wd, r, valid, xy)
            inside = (xy[..., 0] < W) & (xy[..., 1] < H)
            x, y = xy[..., 0][inside], xy[..., 1][inside]
            for t in range(T):
                col, aw = colours(view, t, r)
                alpha, behind, _ = _alpha64(aw, G)
                front = behind / (1 - alpha)
                end = behind.amin(1)
                rgb = torch.einsum("blp,blc->bpc", alpha * front, col)
                out[view, t, y, x] = torch.cat([rgb, end[..., None]], 2)[inside]
    if loss is None and upstream is None:
        return out, graphs, None, None, None
    value = None
    if loss is not None:
        leaf = out.clone().requires_grad_()
        value = loss(leaf)
        upstream, = torch.autograd.grad(value[0], leaf)
    upstream = upstream.double()
    g2 = torch.zeros(V, mean.shape[0], 8, dtype=torch.float64, device=DEV)
    gs = torch.zeros(V, mean.shape[0], 2, dtype=torch.float64, device=DEV)
    for view, cam in enumerate(cams):
        ud, cd = (x.detach() for x in graphs[view][:2])
        for ids, r, valid, xy in _tiles64(cam, *lists[view]):
            d, G = _pairs64(ud, cd, wd, r, valid, xy)
            inside = ((xy[..., 0] < W) & (xy[..., 1] < H))[..., None]
            x, y = xy[..., 0].clamp(max=W - 1), xy[..., 1].clamp(max=H - 1)
            dG = torch.zeros_like(G)
            dv = torch.zeros(r.shape, dtype=torch.float64, device=DEV)
            dw, ds = torch.zeros_like(dv), torch.zeros(*r.shape, 2, dtype=torch.float64, device=DEV)
            for t in range(T):
                up = upstream[view, t, y, x] * inside
                col, aw = colours(view, t, r)
                alpha, behind, on = _alpha64(aw, G)
                front = behind / (1 - alpha)
                wgt = alpha * front
                cg = torch.einsum("blc,bpc->blp", col, up[..., :3])
                tail = cg * wgt
                suffix = tail.flip(1).cumsum(1).flip(1) - tail
                end = behind.amin(1)
                suffix = suffix + (end * up[..., 3])[:, None]  # black background
                da = (front * cg - suffix / (1 - alpha)) * (alpha > 0)
                da = da * ((aw[:, :, None] * G) <= A_MAX)
                dG += da * aw[:, :, None]
                dA = (da * G).sum(2)
                dw += dA * val[t][r][..., 3]
                dcol = torch.einsum("blp,bpc->blc", wgt, up[..., :3])
                sl = slope[t][r]
                scale = 1 if shade is None else shade[view].detach()[r][..., :1]
                dv += (dcol * scale * sl[..., :3]).sum(2) + dA * wd[r] * sl[..., 3]
                if shade is not None:
                    ds[..., 0] += (dcol * val[t][r][..., :3]).sum(2)
                    ds[..., 1] += dcol.sum(2)
            dp = dG * G
            c = cd[r][:, :, None, :]
            dx, dy = d[..., 0], d[..., 1]
            parts = torch.stack([
                (dp * -(c[..., 0] * dx + c[..., 1] * dy)).sum(2),
                (dp * -(c[..., 1] * dx + c[..., 2] * dy)).sum(2),
                (-0.5 * dp * dx * dx).sum(2), (-dp * dx * dy).sum(2), (-0.5 * dp * dy * dy).sum(2),
                dv, dw, torch.zeros_like(dv)], 2)
            g2[view].index_add_(0, r[valid], parts[valid])
            gs[view].index_add_(0, r[valid], ds[valid])
    return out, graphs, value, g2, gs


def _shade64(cam, light, mean, nb, k):
    """Blinn-Phong factors (s_d, s_s) of one view, differentiable."""
    R = torch.as_tensor(cam.world_to_cam, dtype=torch.float64, device=DEV)
    eye = -R[:, :3].T @ R[:, 3]
    light = F.normalize(torch.as_tensor(light, dtype=torch.float64, device=DEV), dim=0)
    nrm = F.normalize(nb[:, :3], dim=1)
    h = F.normalize(F.normalize(eye - mean, dim=1) + light, dim=1)
    nl, nh = (nrm @ light).abs(), (nrm * h).sum(1).abs()
    spec = torch.where((nl > 0) & (nh > 0), nh.clamp(min=1e-300) ** nb[:, 3], torch.zeros_like(nh))
    return torch.stack([k[:, 0] + k[:, 1] * nl, k[:, 2] * spec], 1)


def _loss64(case, target, ssim):
    """out -> (loss, [L1, SSIM]): mean L1 over RGB, or with the SSIM term."""
    t = target.double()
    x = torch.arange(-5, 6, dtype=torch.float64, device=DEV)
    win = torch.exp(-x * x / (2 * 1.5 ** 2))
    win = win / win.sum()

    def blur(a):  # [N][H][W][3], zero padding
        a = a.permute(0, 3, 1, 2).reshape(-1, 1, a.shape[1], a.shape[2])
        a = F.conv2d(a, win.view(1, 1, 1, 11), padding=(0, 5))
        return F.conv2d(a, win.view(1, 1, 11, 1), padding=(5, 0))

    def value(out):
        a, b = (z[..., :3].reshape(-1, case["height"], case["width"], 3) for z in (out, t))
        l1 = (a - b).abs().mean()
        if not ssim:
            return (l1,)
        m1, m2 = blur(a), blur(b)
        s11, s22, s12 = blur(a * a) - m1 * m1, blur(b * b) - m2 * m2, blur(a * b) - m1 * m2
        S = ((2 * m1 * m2 + 1e-4) * (2 * s12 + 9e-4)
             / ((m1 * m1 + m2 * m2 + 1e-4) * (s11 + s22 + 9e-4))).mean()
        return ((1 - LAMBDA) * l1 + LAMBDA * (1 - S), l1, S)

    return value


def _march64(case, seed):
    """Emission-absorption along every ray, all samples in step."""
    R, T = case["res"], case["tfs"]
    vol = _volume(case, seed).double()
    h = 2.0 / (R - 1)
    pad = torch.cat([2 * vol[:1] - vol[1:2], vol, 2 * vol[-1:] - vol[-2:-1]])
    gz = (pad[2:] - pad[:-2]) / (2 * h)
    pad = torch.cat([2 * vol[:, :1] - vol[:, 1:2], vol, 2 * vol[:, -1:] - vol[:, -2:-1]], 1)
    gy = (pad[:, 2:] - pad[:, :-2]) / (2 * h)
    pad = torch.cat([2 * vol[..., :1] - vol[..., 1:2], vol, 2 * vol[..., -1:] - vol[..., -2:-1]], 2)
    gx = (pad[..., 2:] - pad[..., :-2]) / (2 * h)
    v4 = torch.stack([vol, gx, gy, gz], 3).view(-1, 4)
    luts = _tables(case, seed).double()
    step = float(np.float32(h / 2))
    ka, kd, ks, beta = (float(np.float32(x)) for x in MATERIAL)
    out = torch.zeros(case["views"], T, case["height"] * case["width"], 4, dtype=torch.float64,
                      device=DEV)
    for view, cam in enumerate(_cameras(case, seed)):
        w2c = torch.as_tensor(cam.world_to_cam, dtype=torch.float64, device=DEV)
        eye, light = -w2c[:, :3].T @ w2c[:, 3], -w2c[2, :3]
        px = torch.arange(cam.width * cam.height, device=DEV)
        x, y = (px % cam.width).double(), (px // cam.width).double()
        d = torch.stack([(x - cam.cx) / cam.fx, (y - cam.cy) / cam.fy, torch.ones_like(x)], 1)
        d = F.normalize(d @ w2c[:, :3], dim=1)
        t1, t2 = (-1 - eye) / d, (1 - eye) / d
        ta = torch.minimum(t1, t2).amax(1).clamp(min=float(np.float32(cam.near)))
        tb = torch.maximum(t1, t2).amin(1)
        count = ((tb - ta) / step).floor().clamp(min=0)
        half = F.normalize(light - d, dim=1)
        trans = torch.ones(T, px.numel(), dtype=torch.float64, device=DEV)
        rgb = torch.zeros(T, px.numel(), 3, dtype=torch.float64, device=DEV)
        for k in range(int(count.max().item())):
            on = torch.nonzero((count > k) & (trans >= T_MIN).any(0)).squeeze(1)
            if on.numel() == 0:
                continue
            g = (eye + (ta[on] + (k + 0.5) * step)[:, None] * d[on] + 1) / h
            c = g.floor().clamp(0, R - 2)
            f = g - c
            base = ((c[:, 2] * R + c[:, 1]) * R + c[:, 0]).long()
            s = 0
            for dz in (0, 1):
                for dy in (0, 1):
                    for dx in (0, 1):
                        wt = ((f[:, 0] if dx else 1 - f[:, 0]) * (f[:, 1] if dy else 1 - f[:, 1])
                              * (f[:, 2] if dz else 1 - f[:, 2]))
                        s = s + wt[:, None] * v4[base + (dz * R + dy) * R + dx]
            grad = s[:, 1:]
            nrm = F.normalize(grad, dim=1, eps=1e-300)
            flat = (grad == 0).all(1)
            nl, nh = (nrm @ light).abs(), (nrm * half[on]).sum(1).abs()
            sd = torch.where(flat, torch.full_like(nl, ka), ka + kd * nl)
            ss = torch.where(flat | (nl == 0), torch.zeros_like(nl), ks * nh ** beta)
            val = _tf64(luts, s[:, 0])[0]
            alpha = 1 - (1 - val[..., 3].clamp(0, 1)) ** (step / h)
            alpha = alpha * (trans[:, on] >= T_MIN)
            wgt = alpha * trans[:, on]
            rgb[:, on] += wgt[..., None] * (val[..., :3] * sd[:, None] + ss[:, None])
            trans[:, on] *= 1 - alpha
        out[view] = torch.cat([rgb, trans[..., None]], 2)
    return out.view(case["views"], T, case["height"], case["width"], 4)


def exact(case, seed):
    kind = case["kind"]
    if kind == "march":
        return {"out": _march64(case, seed)}
    images = case["views"] * (1 if kind == "guided" else case["tfs"])
    if kind != "geometry" and case["width"] * case["height"] * images * case["n"] ** (1 / 3) > 1e9:
        return None  # the pairs of the large sweep take minutes in 64 bits
    mv, lw, q = (t.double() for t in _model(case, seed))
    luts = _tables(case, seed)
    mean, ls, quat = (t.clone().requires_grad_() for t in (mv[:, :3], lw[:, :3], q))
    tens = (mean, mv[:, 3], ls, lw[:, 3], quat)
    if kind == "geometry":
        geo, aux = [], []
        for cam in _cameras(case, seed):
            u, depth, conic, _, _, ok = _project64(cam, mean, ls, quat, mv[:, 3], lw[:, 3],
                                                   luts.double())
            on = ok.double()[:, None]
            geo.append(torch.cat([u, depth[:, None], lw[:, 3:]], 1) * on)
            aux.append(torch.cat([conic, mv[:, 3:]], 1) * on)
        return {"geo": torch.cat(geo), "aux": torch.cat(aux), "tiles": None, "rect": None,
                "vals": None, "ranges": None}
    if kind in ("render", "composite_fwd"):
        out = _splat64(case, seed, tens, luts)[0]
        return {"out": out} if kind == "render" else {"out": out, "n_contrib": None}
    if kind == "composite_bwd":
        g2 = _splat64(case, seed, tens, luts, upstream=_upstream(case, seed))[3]
        return {"grad2d": g2.view(-1, 4)}
    cams, shade, leaves = _cameras(case, seed), None, [mean, ls, quat]
    if kind == "guided" or case["lit"]:
        nb, k = (t.double().requires_grad_() for t in _lighting(case["n"], seed))
        lights = headlight_dirs(cams).astype(np.float32)
        shade = [_shade64(c, l, mean, nb, k) for c, l in zip(cams, lights)]
        leaves += [nb, k]
    if kind == "guided":
        m = MAPS // 3
        loss = _loss64(case, _image(case, seed, MAPS)[:, m:m + 1], True)
        luts = luts[m:m + 1]
    else:
        loss = _loss64(case, _image(case, seed, case["tfs"]), False)
    out, graphs, value, g2, gs = _splat64(case, seed, tens, luts, shade, loss)
    roots, ups = [], []
    for view, (u, conic, _, ok) in enumerate(graphs):
        on = ok.double()[:, None]
        roots += [u, conic]
        ups += [g2[view, :, :2] * on, g2[view, :, 2:5] * on]
        if shade is not None:
            roots.append(shade[view])
            ups.append(gs[view])
    grads = torch.autograd.grad(roots, leaves, ups)
    tail = g2.sum(0)
    grads = [torch.cat([grads[0], tail[:, 5:6]], 1), torch.cat([grads[1], tail[:, 6:7]], 1),
             *grads[2:]]
    if kind == "guided":
        return {"loss": torch.stack([z.detach() for z in value]), "out": out, "grads": grads,
                "raw": [None] * 5, "m": [None] * 5, "v": [None] * 5, "mean_v": None,
                "logscale_w": None}
    return {"loss": value[0].detach().view(1), "out": out, "grads": grads}
