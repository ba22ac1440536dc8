"""The march over groups of tables, empty macrocells passed in one step and
tables left out where they add nothing: every image equals the one of its
table marched alone without a cell mask, bit for bit."""
import numpy as np
import pytest
import torch

from paper_2504_13339_gb300 import _lib, scenes as S
from paper_2504_13339_gb300.render import lut_tensor
from paper_2504_13339_gb300.train import opacity_guided_luts
from test_gpu_raymarch import MAT, dev, march, prepared

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module", autouse=True)
def built():
    import __graft_entry__
    __graft_entry__.build()


def masked(cams, v4, luts, step, cell, material):
    lt = lut_tensor(luts)
    mask = torch.empty(_lib.veg_raymarch_cells_count(v4.shape[0], cell), dtype=torch.int32,
                       device="cuda")
    _lib.veg_raymarch_cells(v4, _lib.tf_desc(lt), cell, mask)
    out = torch.empty(len(cams), lt.shape[0], cams[0].height, cams[0].width, 4, device="cuda")
    _lib.veg_raymarch_masked(_lib.cameras(cams), v4, _lib.tf_desc(lt), step, out, mask, cell,
                             material)
    return out.cpu().numpy()


# one table, a full group, one more than a group, beyond the 32 mask bits;
# macrocells of one cell, ragged at the far faces, and wider than the volume;
# steps of a fraction of a cell and of several cells
@pytest.mark.parametrize("n_tf,R,cell,per", [(1, 34, 4, 0.5), (5, 19, 1, 0.3), (16, 33, 8, 0.5),
                                             (17, 30, 4, 0.7), (33, 24, 8, 0.5), (10, 20, 64, 0.2),
                                             (10, 40, 2, 3.3)])
@pytest.mark.parametrize("material", [None, MAT])
def test_every_table_of_a_call_equals_the_table_alone(n_tf, R, cell, per, material):
    v4 = prepared(S.field_volume(S.blob_field(4, 7), R))
    luts = opacity_guided_luts(n_tf, S.colour_ramp(3))
    cams = S.orbit_cameras(2, 5, 43, 37)
    step = 2.0 / (R - 1) * per
    alone = np.concatenate([march(cams, v4, luts[t:t + 1], step, material)
                            for t in range(n_tf)], 1)
    assert np.array_equal(march(cams, v4, luts, step, material), alone)
    assert np.array_equal(masked(cams, v4, luts, step, cell, material), alone)


def test_what_is_not_finite_still_reaches_the_image():
    """0 times an infinite colour, and any shading by a gradient with a NaN
    beside a nonzero component, is NaN: such samples are not left out."""
    R, cams = 16, S.orbit_cameras(1, 2, 32, 32)
    vol = np.full((R, R, R), 0.25, np.float32)
    luts = np.zeros((2, 16, 4), np.float32)
    luts[0, :, 0] = np.inf  # transparent, infinitely bright
    step = 2.0 / (R - 1) * 0.5
    out = march(cams, prepared(vol), luts, step)
    hit = np.isnan(out[0, 0, :, :, 0])
    assert hit.any() and (out[0, :, :, :, 3] == 1).all()
    assert (out[0, 1] == np.float32([0, 0, 0, 1])).all()
    v4 = prepared(vol)
    v4[..., 1] = float("nan")
    v4[..., 2] = 1.0
    luts[0, :, 0] = 0.5
    assert np.array_equal(np.isnan(march(cams, v4, luts, step, MAT)[0, 1, :, :, 0]), hit)
