"""The forward of few work items against the forward of many, bit for bit.

One table over a small image takes the kernel with producer and consumer
warps; the same table many times over takes the one with a warp per block.
Images, transmittances and contribution counts must be equal.
"""
import numpy as np
import pytest
import torch

from paper_2504_13339_gb300 import scenes as S
from paper_2504_13339_gb300.render import SplatPipeline, headlight_dirs, lut_tensor

pytestmark = pytest.mark.gpu

MANY = 40


@pytest.fixture(scope="module", autouse=True)
def built():
    import __graft_entry__
    __graft_entry__.build()


def images(g, cams, luts, lit, bg):
    dev = lambda a: torch.as_tensor(np.ascontiguousarray(a), device="cuda")
    p = SplatPipeline(g.n, cams, n_tf=luts.shape[0])
    tens = [dev(a) for a in (g.mean_v, g.logscale_w, g.quat)]
    if lit:
        rng = np.random.default_rng(4)
        nb = np.concatenate([rng.normal(size=(g.n, 3)), np.full((g.n, 1), 9.0)], 1)
        nb[:, :3] /= np.linalg.norm(nb[:, :3], axis=1, keepdims=True)
        k = np.tile(np.float32([0.3, 0.5, 0.2, 0]), (g.n, 1))
        p.shade(tens[0], dev(nb.astype(np.float32)), dev(k), headlight_dirs(cams))
    out = p.render(*tens, luts, bg=bg)
    return out.cpu().numpy(), p.n_contrib.cpu().numpy(), p.ranges.cpu().numpy()


# no splats, lists of less than a chunk, of a few chunks (ended early and
# not), and of hundreds; blocks beyond the image's edges; several views
@pytest.mark.parametrize("n,views,W,H,logscale,opacity", [
    (0, 1, 200, 170, -3.0, 1.0), (300, 1, 199, 171, -3.5, 1.0), (4000, 1, 200, 177, -2.5, 1.0),
    (4000, 2, 145, 161, -2.5, 0.02), (60_000, 1, 200, 170, -3.0, 1.0),
    (60_000, 1, 193, 170, -2.8, 0.02)])
@pytest.mark.parametrize("lit", [False, True])
def test_one_table_alone_equals_the_table_among_many(n, views, W, H, logscale, opacity, lit):
    g = S.uniform_gaussians(n, 11, logscale_mean=logscale)
    cams = S.orbit_cameras(views, 6, W, H)
    lut = lut_tensor(S.bump_tfs(1, 9)).clone()
    lut[..., 3] = torch.where(lut[..., 3] > 0, opacity * lut[..., 3], 0)
    bg = (0.1, 0.2, 0.3)
    one, nc1, ranges = images(g, cams, lut, lit, bg)
    many, ncm, _ = images(g, cams, lut.expand(MANY, -1, -1).contiguous(), lit, bg)
    tiles = views * ((W + 15) // 16) * ((H + 15) // 16)
    assert tiles < 2048 <= tiles * MANY  # the two kernels
    assert np.array_equal(one, many[:, :1]) and np.array_equal(nc1, ncm[:, :1])
    if n >= 60_000:
        assert (ranges[:, 1] - ranges[:, 0]).max() > 1000
