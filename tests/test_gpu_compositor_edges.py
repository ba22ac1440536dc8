"""The compositor where its tiling can go wrong: list lengths around the
steps, chunks and batches of its walks (1-4, 32, 128, 256 splats), image
edges that leave a lane one of its two pixels or none, and splats whose
reach test has little room (needles, sub-pixel and very wide ones).  Images
and gradients against the oracle at the suite's bars, the forward's tile
batches bit for bit."""
import math

import numpy as np
import pytest
import torch

from oracle import veg_oracle as O
from paper_2504_13339_gb300 import _lib, scenes as S
from paper_2504_13339_gb300.render import SplatPipeline, lut_tensor
from parity import checked_forward, grad_check

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module", autouse=True)
def built():
    import __graft_entry__
    __graft_entry__.build()


def dev(a):
    return torch.as_tensor(np.ascontiguousarray(a), device="cuda")


def check(name, g, cams, tfs, bg=(0.1, 0.0, 0.2), tensors=("mean_v", "logscale_w", "quat")):
    p = SplatPipeline(g.n, cams, n_tf=len(tfs))
    tens = (dev(g.mean_v), dev(g.logscale_w), dev(g.quat))
    luts = lut_tensor(tfs)
    p.project(*tens, luts)
    p.bin_sort()
    assert p.status()[0] == _lib.VEG_OK
    imgs = []
    for batch in (128, 256, 512):
        p.tile_batch = batch
        p.out.fill_(-1.0)
        p.n_contrib.fill_(-1)
        p.composite(luts, bg)
        imgs.append((p.out.cpu().numpy().view(np.uint32).copy(), p.n_contrib.cpu().numpy().copy()))
    for o, n in imgs[1:]:
        assert np.array_equal(o, imgs[0][0]) and np.array_equal(n, imgs[0][1])
    proj, bins, fwd = O.render(cams, g, tfs, bg=bg, record=True)
    excl = checked_forward(name, fwd, proj, cams, bins, tfs, bg, p.out.cpu().numpy(),
                           p.n_contrib.cpu().numpy(), None)
    dout = np.random.default_rng(7).standard_normal(fwd["out"].shape)
    dout[excl] = 0.0
    grads = [torch.zeros_like(t) for t in tens]
    p.backward(dev(dout.astype(np.float32)), *grads)
    g2 = O.composite_bwd(proj, cams, bins, tfs, bg, fwd, dout)
    for a, b, what in zip(grads, O.params_grad(cams, g, proj, g2), ("mean_v", "logscale_w", "quat")):
        if what in tensors:
            grad_check(a.cpu().numpy(), b, f"{name} {what}", elementwise=False)


@pytest.mark.parametrize("n", [1, 2, 3, 4, 5, 31, 32, 33, 64, 65, 127, 128, 129, 256, 257, 513])
def test_list_lengths_around_the_steps_of_the_walk(n):
    """n faint splats over a 16 x 12 image: one tile whose list holds all."""
    rng = np.random.default_rng(200 + n)
    g = S.uniform_gaussians(n, 300 + n, logscale_mean=-1.5, logscale_std=0.3)
    g.mean_v[:, :2] = rng.uniform(-0.3, 0.3, (n, 2))
    g.logscale_w[:, 3] = rng.uniform(0.02, 0.2, n)
    check(f"length_{n}", g, [S.look_at_camera((0.0, 0.0, 3.0), 16, 12)], S.bump_tfs(2, 41))


@pytest.mark.parametrize("size", [(1, 1), (7, 5), (8, 4), (9, 9), (17, 13), (33, 21)])
def test_image_edges(size):
    g = S.uniform_gaussians(120, 77, logscale_mean=-1.8, logscale_std=0.5)
    check(f"edge_{size[0]}x{size[1]}", g, [S.orbit_camera(20.0, 10.0, 3.0, *size)],
          S.bump_tfs(3, 42))


@pytest.mark.parametrize("aspect", [1.0, 8.0, 60.0, 400.0])
def test_reach_of_needles_and_extreme_widths(aspect):
    """Random orientations; widths from a fraction of a pixel to the image,
    length over width `aspect` (400 is beyond the reach test's conditioning).
    A sphere's rotation has no gradient: its reference is zero up to rounding
    and gives no relative bar."""
    rng = np.random.default_rng(int(aspect))
    n = 250
    g = S.uniform_gaussians(n, 78)
    ls = rng.uniform(math.log(0.002), math.log(0.4), n)
    g.logscale_w[:, 0] = ls
    g.logscale_w[:, 1:3] = (ls - math.log(aspect))[:, None]
    g.logscale_w[:, 3] = rng.uniform(0.05, 1.0, n)
    check(f"aspect_{aspect:g}", g, [S.orbit_camera(200.0, -15.0, 2.5, 75, 50)], S.bump_tfs(2, 43),
          tensors=("mean_v", "logscale_w") if aspect == 1.0 else ("mean_v", "logscale_w", "quat"))
