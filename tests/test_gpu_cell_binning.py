"""The cell binning against the general tile sort, bit for bit.

A call that asks for the 64-bit keys takes the sort of all instances by tile
(itself checked against the oracle in test_gpu_parity.py); the same call
without keys takes the cell binning when the views have more than 256 tiles
and the capacity is at least 5 * 2^18 instances.  Records are random: depths
with many ties, rectangles from one tile to the whole image, empty ones, and
both sides of the cells' edges.
"""
import numpy as np
import pytest
import torch

from paper_2504_13339_gb300 import _lib, scenes as S

pytestmark = pytest.mark.gpu


def records(n, views, W, H, wide, seed):
    gen = torch.Generator(device="cuda")
    gen.manual_seed(seed)
    nr, tx, ty = n * views, (W + 15) // 16, (H + 15) // 16
    rand = lambda hi: torch.randint(0, hi, (nr,), generator=gen, device="cuda")
    depth = 0.5 + rand(max(2, n // 3)).float() / n
    x0, y0 = rand(tx), rand(ty)
    x1 = torch.minimum(x0 + 1 + rand(wide), torch.tensor(tx, device="cuda"))
    y1 = torch.minimum(y0 + 1 + rand(wide), torch.tensor(ty, device="cuda"))
    full = rand(max(nr // 5, 1)) == 0  # a few cover the whole image
    x0, y0 = torch.where(full, 0, x0), torch.where(full, 0, y0)
    x1, y1 = torch.where(full, tx, x1), torch.where(full, ty, y1)
    rect = torch.stack([x0, y0, x1, y1], 1)
    rect[rand(8) == 0] = 0  # culled
    tiles = ((rect[:, 2] - rect[:, 0]) * (rect[:, 3] - rect[:, 1])).int()
    geo = torch.zeros(nr, 4, device="cuda")
    geo[:, 2] = depth
    return geo, tiles.contiguous(), rect.short().contiguous()


# tiles per side at, one below and one above whole cells; one and several
# radix passes over the cells; records below and above the compaction's
# limit; packed and (2^23 records, 520 cells) unpacked pairs
@pytest.mark.parametrize("n,views,W,H,wide", [
    (40_000, 1, 400, 272, 30), (65_536, 1, 512, 512, 25), (100_000, 1, 513, 257, 40),
    (200_000, 3, 257, 193, 9), (150_000, 2, 1601, 1199, 12), (40_000, 5, 1100, 900, 20),
    (2_100_000, 4, 1601, 1199, 2)])
@pytest.mark.parametrize("cut", [None, 0.35, 1.0])
def test_lists_equal_those_of_the_tile_sort(n, views, W, H, wide, cut):
    cams = S.orbit_cameras(views, 3, W, H)
    cc = _lib.cameras(cams)
    geo, tiles, rect = records(n, views, W, H, wide, n + views)
    m = int(tiles.sum())
    cap = m + 1000 if cut is None else int(m * cut)  # cut 1: exactly full
    got = []
    for want in (True, False):
        ws = torch.zeros(_lib.veg_bin_sort_workspace_size(n, views, cap, W, H),
                         dtype=torch.uint8, device="cuda")
        vals = torch.full((cap,), -1, dtype=torch.int32, device="cuda")
        keys = torch.empty(cap, dtype=torch.int64, device="cuda") if want else None
        ranges = torch.full((views * ((W + 15) // 16) * ((H + 15) // 16), 2), 7,
                            dtype=torch.int32, device="cuda")
        before = _lib.veg_kernel_launches()
        _lib.veg_bin_sort(cc, n, geo, tiles, rect, ws, cap, keys, vals, ranges)
        st, count = _lib.veg_sync_status(ws)
        assert count == m and (st == _lib.VEG_OK) == (cap >= m)
        used = min(m, cap)
        got.append((vals[:used].cpu().numpy(), ranges.cpu().numpy(),
                    _lib.veg_kernel_launches() - before))
    assert np.array_equal(got[0][1], got[1][1])
    assert np.array_equal(got[0][0], got[1][0])
    assert got[0][2] != got[1][2]  # the two calls took different routes
