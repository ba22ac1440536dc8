"""The backward of four tables per pass against the one of a table per pass:
the same terms summed in another order.  Ragged groups, list lengths around the
chunks, image edges, shaded and not, tables that overlap, do not, and have
infinite entries; and a call that lets each group's overlap choose."""
import numpy as np
import pytest
import torch

from paper_2504_13339_gb300 import scenes as S
from paper_2504_13339_gb300.render import SplatPipeline, headlight_dirs, lut_tensor

pytestmark = pytest.mark.gpu

TOL = 2e-5  # of a tensor's largest entry: sums of some thousand float32 terms


@pytest.fixture(scope="module", autouse=True)
def built():
    import __graft_entry__
    __graft_entry__.build()


def dev(a):
    return torch.as_tensor(np.ascontiguousarray(a), device="cuda")


def compare(g, cams, tables, lit, groups, seed=1):
    luts = lut_tensor(tables)
    p = SplatPipeline(g.n, cams, n_tf=luts.shape[0])
    tens = [dev(a) for a in (g.mean_v, g.logscale_w, g.quat)]
    rng = np.random.default_rng(seed)
    if lit:
        nb = rng.normal(size=(g.n, 4)).astype(np.float32)
        nb[:, 3] = 9.0
        p.shade(tens[0], dev(nb), dev(np.tile(np.float32([0.3, 0.5, 0.2, 0]), (g.n, 1))),
                headlight_dirs(cams))
    out = p.render(*tens, luts, bg=(0.1, 0.2, 0.3))
    dout = torch.as_tensor(rng.normal(size=out.shape).astype(np.float32), device="cuda")
    got = []
    for group in (1,) + groups:
        p.tf_group_bwd = group
        p.backward_2d(dout)
        got.append([p.grad2d.clone()] + ([p.grad_shade.clone()] if lit else []))
    assert g.n < 31 or (got[0][0] != 0).any()  # (one splat may be transparent)
    for other in got[1:]:
        for a, b in zip(got[0], other):
            assert torch.isfinite(b).all()
            assert (a - b).abs().max() <= TOL * a.abs().max()


def same_opacity(n_tf, seed):
    x = S.bump_tfs(n_tf, seed)
    x[:, :, 3] = x[0, :, 3]
    return x


@pytest.mark.parametrize("lit", [False, True])
@pytest.mark.parametrize("n", [1, 2, 31, 32, 33, 64, 65, 513])
def test_list_lengths(n, lit):
    rng = np.random.default_rng(200 + n)
    g = S.uniform_gaussians(n, 300 + n, logscale_mean=-1.5, logscale_std=0.3)
    g.mean_v[:, :2] = rng.uniform(-0.3, 0.3, (n, 2))
    g.logscale_w[:, 3] = rng.uniform(0.02, 0.2, n)
    compare(g, [S.look_at_camera((0.0, 0.0, 3.0), 16, 12)], same_opacity(4, 41), lit, (2, 4))


@pytest.mark.parametrize("n_tf", [3, 4, 5, 7, 9])
@pytest.mark.parametrize("kind", ["same", "bump", "infinite"])
def test_groups_and_tables(n_tf, kind):
    g = S.uniform_gaussians(900, 77, logscale_mean=-2.0, logscale_std=0.5)
    tables = same_opacity(n_tf, 9) if kind == "same" else S.bump_tfs(n_tf, 9)
    if kind == "infinite":
        tables[::2, 100:120, 3] = np.inf
    compare(g, [S.orbit_camera(20.0, 10.0, 3.0, 45, 37), S.orbit_camera(80.0, -10.0, 3.0, 45, 37)],
            tables, n_tf == 5, (4,))


@pytest.mark.parametrize("lit", [False, True])
def test_each_group_by_its_overlap(lit):
    """1089 tiles: the first four tables overlap, the next four do not, the last
    is alone."""
    g = S.uniform_gaussians(20_000, 78, logscale_mean=-3.0)
    tables = np.concatenate([same_opacity(4, 5), S.bump_tfs(5, 6)])
    tables[4:8, :, 3] = 0.0
    for t in range(4):
        tables[4 + t, 64 * t:64 * t + 60, 3] = 0.5
    compare(g, [S.orbit_camera(20.0, 10.0, 3.0, 528, 517)], tables, lit, (0, 4))
