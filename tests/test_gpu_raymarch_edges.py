"""The march at the edges of its inputs: distant eyes, shades without bound, and
the macrocells' masks from single cells to macrocells wider than the volume."""
import math
from dataclasses import replace

import numpy as np
import pytest
import torch

from paper_2504_13339_gb300 import _lib, scenes as S
from paper_2504_13339_gb300.render import lut_tensor
from test_gpu_raymarch import MAT, march, prepared
from test_gpu_raymarch_groups import masked

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module", autouse=True)
def built():
    import __graft_entry__
    __graft_entry__.build()


@pytest.mark.parametrize("R,cell,distance", [(65, 4, 5e4), (130, 8, 2e4), (65, 2, 1e5)])
def test_steps_over_empty_space_from_far_away(R, cell, distance):
    """Beyond 2^13 or so a distance's rounding is a fair part of a vertex cell:
    the masked image must still be the plain one, bit for bit."""
    vol = np.zeros((R, R, R), np.float32)
    rng = np.random.default_rng(R)
    at = rng.integers(0, R, (R * R // 2, 3))
    vol[tuple(at.T)] = rng.uniform(0.3, 1, len(at))  # a dust of single vertices
    luts = np.zeros((2, 1024, 4), np.float32)  # opaque from a few thousandths on
    luts[..., :3] = rng.uniform(0, 1, (2, 1024, 3))
    luts[0, 4:, 3] = 0.2
    luts[1, 40:, 3] = 0.3
    fov = math.degrees(2 * math.atan(1.5 / distance))
    cams = [S.orbit_camera(a, b, distance, 150, 140, fov_deg=fov) for a, b in ((20, 10), (77, -40))]
    step, v4 = 2.0 / (R - 1) * 0.5, prepared(vol)
    plain = march(cams, v4, luts, step, MAT)
    assert (plain[..., 3] < 1).mean() > 0.05  # the dust is seen
    assert np.array_equal(masked(cams, v4, luts, step, cell, MAT), plain)


@pytest.mark.parametrize("beta,scale,colour", [(1e10, 1.0, 0.5), (12.0, 1e15, 1e28)])
def test_a_sample_shaded_to_infinity_reaches_the_image(beta, scale, colour):
    """A shininess that lifts a cosine of 1 + 1e-7 to infinity, or a camera whose
    rows (and headlight) are not unit: zero opacity times such a shade is NaN,
    as it is under an opacity too small to count."""
    R, eye = 24, np.array([1.0, 2.0, 3.0])
    cam = S.look_at_camera(eye, 64, 64, fov_deg=0.05)  # normals within 1e-3 of the half vectors
    x = np.linspace(-1, 1, R)
    vol = 0.5 + 0.1 * np.einsum("c,cijk->ijk", eye, np.stack(np.meshgrid(x, x, x, indexing="ij"))[::-1])
    vol = vol.astype(np.float32)
    w = np.array(cam.world_to_cam, np.float32)
    w[:, :3] *= scale
    w[:, 3] /= scale
    cam = replace(cam, world_to_cam=w)
    luts = np.full((2, 16, 4), colour, np.float32)
    luts[0, :, 3], luts[1, :, 3] = 0.0, 1e-30
    out = march([cam], prepared(vol), luts, 1.0 / (R - 1), (0.3, 0.6, 0.25, beta))
    assert np.isnan(out[0, 1]).any()
    assert np.array_equal(out[0, 0], out[0, 1], equal_nan=True)


# 65536 macrocells and more take a lane each up to cells of four, fewer eight
# lanes; cells of eight and more a warp
@pytest.mark.parametrize("R,cell", [(42, 1), (20, 1), (84, 2), (31, 2), (163, 4), (30, 4), (60, 8),
                                    (33, 16), (21, 64)])
@pytest.mark.parametrize("n_tf", [1, 9, 32, 33])
def test_masks(R, cell, n_tf):
    rng = np.random.default_rng(R + n_tf)
    vol = rng.uniform(-0.2, 1.2, (R, R, R)).astype(np.float32) ** 3
    vol[rng.integers(0, R, 3), 0, 1] = np.nan
    vol[1, rng.integers(0, R, 3), 2] = np.inf
    vol[2, 1, rng.integers(0, R, 3)] = -np.inf
    L = 64
    op = np.where(rng.random((n_tf, L)) < 0.06, 0.5, -0.1).astype(np.float32)
    luts = np.zeros((n_tf, L, 4), np.float32)
    luts[..., 3] = op
    v4 = prepared(vol)
    got = torch.empty(_lib.veg_raymarch_cells_count(R, cell), dtype=torch.int32, device="cuda")
    _lib.veg_raymarch_cells(v4, _lib.tf_desc(lut_tensor(luts)), cell, got)
    at = [slice(c, min(c + cell, R - 1) + 1) for c in range(0, R - 1, cell)]
    lo, hi = (np.stack([np.stack([np.stack([f(vol[z, y, x]) for x in at]) for y in at]) for z in at])
              for f in (np.min, np.max))  # a NaN vertex makes both NaN
    nan = np.isnan(lo)
    one = np.float32(1e-6)
    with np.errstate(invalid="ignore"):
        k0 = np.floor(np.clip(np.nan_to_num(lo) - one, 0, 1) * np.float32(L - 1)).astype(int) - 1
        k1 = np.floor(np.clip(np.nan_to_num(hi) + one, 0, 1) * np.float32(L - 1)).astype(int) + 2
    k0, k1 = np.maximum(k0, 0), np.minimum(k1, L - 1)
    seen = np.concatenate([np.zeros((n_tf, 1), int), np.cumsum(op > 0, 1)], 1)
    want = np.zeros(lo.shape, np.uint32)
    for t in range(min(n_tf, 32)):
        want |= (seen[t][k1 + 1] > seen[t][k0]).astype(np.uint32) << np.uint32(t)
    want[nan | (n_tf > 32)] = 0xffffffff
    assert np.array_equal(got.cpu().numpy().view(np.uint32).reshape(want.shape), want)
