"""The binning in one CTA (up to 4096 records and 256 lists) against a stable
sort on the host: lists at, below and above a word of 32, rows that cross
words and rows of every list, several views, and a capacity that cuts a
record."""
import numpy as np
import pytest
import torch

from paper_2504_13339_gb300 import _lib, scenes as S
from test_gpu_cell_binning import records

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module", autouse=True)
def built():
    import __graft_entry__
    __graft_entry__.build()


def lists(geo, tiles, rect, n, views, tx, per_view, cap):
    order = np.argsort(geo[:, 2].view(np.uint32), kind="stable")
    order = order[tiles[order] > 0]
    tile, rec = [], []
    for g in order:
        x0, y0, x1, y1 = rect[g]
        ids = (np.arange(y0, y1)[:, None] * tx + np.arange(x0, x1)).ravel() + g // n * per_view
        tile.append(ids)
        rec.append(np.full(len(ids), g))
    tile, rec = (np.concatenate(a)[:cap] for a in (tile, rec))
    by = np.argsort(tile, kind="stable")
    count = np.bincount(tile, minlength=views * per_view)
    end = np.cumsum(count)
    ranges = np.where(count[:, None] > 0, np.stack([end - count, end], 1), 0)
    return rec[by], ranges


@pytest.mark.parametrize("n,views,W,H,wide", [
    (7, 1, 16, 16, 1), (300, 1, 16 * 31, 16, 31), (900, 1, 16 * 32, 16, 9), (1025, 1, 16 * 11, 48, 4),
    (4096, 1, 128, 128, 3), (4096, 1, 256, 256, 16), (4096, 1, 4096, 16, 200), (1365, 3, 80, 272, 6),
    (1024, 4, 128, 128, 2), (33, 1, 16 * 51, 80, 40)])
@pytest.mark.parametrize("cut", [None, 0.6])
def test_lists_equal_a_stable_sort_on_the_host(n, views, W, H, wide, cut):
    cams = S.orbit_cameras(views, 3, W, H)
    geo, tiles, rect = records(n, views, W, H, wide, n + W)
    tx, per_view = (W + 15) // 16, ((W + 15) // 16) * ((H + 15) // 16)
    assert n * views <= 4096 and views * per_view <= 256  # the one-CTA path
    m = int(tiles.sum())
    cap = m if cut is None else int(m * cut)
    ws = torch.zeros(_lib.veg_bin_sort_workspace_size(n, views, cap, W, H), dtype=torch.uint8,
                     device="cuda")
    vals = torch.full((cap,), -1, dtype=torch.int32, device="cuda")
    ranges = torch.full((views * per_view, 2), 7, dtype=torch.int32, device="cuda")
    before = _lib.veg_kernel_launches()
    _lib.veg_bin_sort(_lib.cameras(cams), n, geo, tiles, rect, ws, cap, None, vals, ranges)
    assert _lib.veg_kernel_launches() - before == 1
    st, count = _lib.veg_sync_status(ws)
    assert count == m and (st == _lib.VEG_OK) == (cap >= m)
    rec, ref = lists(*(t.cpu().numpy() for t in (geo, tiles, rect)), n, views, tx, per_view, cap)
    assert np.array_equal(ranges.cpu().numpy(), ref)
    assert np.array_equal(vals.cpu().numpy(), rec)
