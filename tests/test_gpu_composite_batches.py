"""The forward's staged batches where they can go wrong, against the kernel of
few work items (which test_gpu_compositor_edges.py checks against the oracle),
bit for bit: list lengths around the walk's steps and the batches' ends, image
edges, needles and very wide splats.  Tables are repeated until the launch
stages batches; the route is asked of the library."""
import math

import numpy as np
import pytest
import torch

from paper_2504_13339_gb300 import _lib, scenes as S
from paper_2504_13339_gb300.render import SplatPipeline, headlight_dirs, lut_tensor

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module", autouse=True)
def built():
    import __graft_entry__
    __graft_entry__.build()


def dev(a):
    return torch.as_tensor(np.ascontiguousarray(a), device="cuda")


def check(g, cams, tfs, lit, bg=(0.1, 0.0, 0.2)):
    one = lut_tensor(tfs)
    c = _lib.cameras(cams)
    route = lambda luts, b: _lib.veg_composite_fwd_batch(c, g.n, _lib.tf_desc(luts), b)
    assert route(one, 0) == 0
    many = one.repeat(2, 1, 1)
    while route(many, 0) == 0:
        many = many.repeat(2, 1, 1)
    tens = (dev(g.mean_v), dev(g.logscale_w), dev(g.quat))
    rng = np.random.default_rng(4)
    nb = rng.normal(size=(g.n, 4)).astype(np.float32)
    nb[:, 3] = 9.0
    k = np.tile(np.float32([0.3, 0.5, 0.2, 0]), (g.n, 1))
    want = None
    for luts, batches in ((one, (0,)), (many, (128, 256, 512))):
        p = SplatPipeline(g.n, cams, n_tf=luts.shape[0])
        if lit:
            p.shade(tens[0], dev(nb), dev(k), headlight_dirs(cams))
        p.render(*tens, luts, bg=bg)
        for b in batches:
            assert luts is one or route(luts, b) == b
            p.tile_batch = b
            p.out.fill_(-1.0)
            p.n_contrib.fill_(-1)
            p.composite(luts, bg)
            if want is None:
                want = p.out.clone(), p.n_contrib.clone()
                continue
            times = luts.shape[0] // one.shape[0]
            for got, ref in ((p.out, want[0]), (p.n_contrib, want[1])):
                rep = (1, times) + (1,) * (got.ndim - 2)
                assert torch.equal(got, ref.repeat(rep))


@pytest.mark.parametrize("lit", [False, True])
@pytest.mark.parametrize("n", [0, 1, 3, 4, 5, 31, 33, 127, 128, 129, 256, 257, 511, 513, 1025])
def test_list_lengths(n, lit):
    rng = np.random.default_rng(200 + n)
    g = S.uniform_gaussians(n, 300 + n, logscale_mean=-1.5, logscale_std=0.3)
    g.mean_v[:, :2] = rng.uniform(-0.3, 0.3, (n, 2))
    g.logscale_w[:, 3] = rng.uniform(0.02, 0.2, n)
    check(g, [S.look_at_camera((0.0, 0.0, 3.0), 16, 12)], S.bump_tfs(2, 41), lit)


@pytest.mark.parametrize("size", [(1, 1), (7, 5), (8, 4), (9, 9), (17, 13), (33, 21)])
def test_image_edges(size):
    g = S.uniform_gaussians(120, 77, logscale_mean=-1.8, logscale_std=0.5)
    check(g, [S.orbit_camera(20.0, 10.0, 3.0, *size)], S.bump_tfs(3, 42), size[0] % 2 == 0)


@pytest.mark.parametrize("aspect", [1.0, 60.0, 400.0])
def test_needles_and_extreme_widths(aspect):
    rng = np.random.default_rng(int(aspect))
    g = S.uniform_gaussians(250, 78)
    ls = rng.uniform(math.log(0.002), math.log(0.4), 250)
    g.logscale_w[:, 0] = ls
    g.logscale_w[:, 1:3] = (ls - math.log(aspect))[:, None]
    g.logscale_w[:, 3] = rng.uniform(0.05, 1.0, 250)
    check(g, [S.orbit_camera(200.0, -15.0, 2.5, 75, 50)], S.bump_tfs(2, 43), False)


@pytest.mark.parametrize("L", [2, 1024, 2048, 4096])
def test_table_sizes(L):
    """Both kernels over the tables' range."""
    g = S.uniform_gaussians(3000, 79, logscale_mean=-2.5)
    check(g, S.orbit_cameras(2, 6, 60, 40), S.bump_tfs(1, 44, size=L), L == 2048)


def test_a_table_index_out_of_range_has_no_gradient():
    """Such a view reads as transparent in the backward too, also after a forward
    that saw a valid index."""
    g = S.uniform_gaussians(500, 80, logscale_mean=-2.5)
    cams = S.orbit_cameras(2, 6, 60, 40)
    tens = (dev(g.mean_v), dev(g.logscale_w), dev(g.quat))
    luts = lut_tensor(S.bump_tfs(2, 45))
    p = SplatPipeline(g.n, cams, n_tf=1)
    p.project(*tens)
    p.bin_sort()
    dout = torch.randn_like(p.out)
    got = []
    for view_tf in ([1, 0], [1, 5]):
        vt = torch.tensor(view_tf, dtype=torch.int32, device="cuda")
        if not got:
            _lib.veg_composite_fwd(p.c_cams, p.n, p.geo, p.aux, p.vals, p.ranges,
                                   _lib.tf_desc(luts, vt), (0.0, 0.0, 0.0), 0, p.out, p.n_contrib)
        _lib.veg_composite_bwd(p.c_cams, p._g, p.geo, p.aux, p.tiles, p.vals, p.ranges,
                               _lib.tf_desc(luts, vt), (0.0, 0.0, 0.0), 0, p.out, p.n_contrib,
                               dout, None, None, None, None, p.grad2d)
        got.append(p.grad2d.view(2, -1).clone())
    assert (got[0] != 0).any(1).all() and torch.allclose(got[0][0], got[1][0], rtol=1e-4, atol=1e-6)
    assert (got[1][1] == 0).all()
