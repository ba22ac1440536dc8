"""Opacities without bound: alpha is clamped to 0.99 everywhere, so a table with
infinite entries gives the image and the gradients of one with entries so large
that every pair is clamped too."""
import numpy as np
import pytest
import torch

from paper_2504_13339_gb300 import scenes as S
from paper_2504_13339_gb300.render import SplatPipeline, headlight_dirs, lut_tensor

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module", autouse=True)
def built():
    import __graft_entry__
    __graft_entry__.build()


@pytest.mark.parametrize("lit", [False, True])
def test_infinite_opacity(lit):
    dev = lambda a: torch.as_tensor(np.ascontiguousarray(a), device="cuda")
    n = 300
    g = S.uniform_gaussians(n, 3, logscale_mean=-0.7, logscale_std=0.1)  # wide: no exponent below -60
    cams = S.orbit_cameras(1, 4, 24, 20)
    tens = [dev(a) for a in (g.mean_v, g.logscale_w, g.quat)]
    rng = np.random.default_rng(5)
    nb = rng.normal(size=(n, 4)).astype(np.float32)
    nb[:, 3] = 9.0
    k = np.tile(np.float32([0.3, 0.5, 0.2, 0]), (n, 1))
    base = S.bump_tfs(2, 6)
    base[:, :128, 3] *= 0.1
    got = []
    for big in (1e30, np.inf):
        x = base.copy()
        x[0, 128:, 3] = big  # a step from faint to clamped
        x[1, 100:110, 3] = big
        luts = lut_tensor(x)
        p = SplatPipeline(n, cams, n_tf=2)
        if lit:
            p.shade(tens[0], dev(nb), dev(k), headlight_dirs(cams))
        out = p.render(*tens, luts, bg=(0.1, 0.2, 0.3))
        dout = dev(np.random.default_rng(7).normal(size=out.shape).astype(np.float32))
        p.backward_2d(dout)
        got.append([t.clone() for t in (out, p.n_contrib, p.grad2d) + ((p.grad_shade,) if lit else ())])
    assert torch.equal(got[0][0], got[1][0]) and torch.equal(got[0][1], got[1][1])
    assert (got[0][2] != 0).any() and torch.isfinite(got[0][2]).all()
    for a, b in zip(got[0][2:], got[1][2:]):  # sums in another order
        assert torch.isfinite(b).all()
        assert (a - b).abs().max() <= 1e-5 * a.abs().max()
