"""Where the cell binning begins, its route counted by launches: a call with
keys takes the tile sort and one launch more than the same sort without; any
other difference is the other path.  Lists at both sides of the line, whole
and cut, equal those of the sort."""
import numpy as np
import pytest
import torch

from paper_2504_13339_gb300 import _lib, scenes as S
from test_gpu_cell_binning import records

pytestmark = pytest.mark.gpu

LINE = 5 << 18  # instances of capacity


@pytest.fixture(scope="module", autouse=True)
def built():
    import __graft_entry__
    __graft_entry__.build()


def binned(n, views, W, H, wide, cap):
    """(the lists with and without keys, whether the latter took the cells)"""
    cams = S.orbit_cameras(views, 3, W, H)
    cc = _lib.cameras(cams)
    geo, tiles, rect = records(n, views, W, H, wide, n + views)
    m, got, took = int(tiles.sum()), [], []
    for want in (True, False):
        ws = torch.zeros(_lib.veg_bin_sort_workspace_size(n, views, cap, W, H),
                         dtype=torch.uint8, device="cuda")
        vals = torch.full((cap,), -1, dtype=torch.int32, device="cuda")
        keys = torch.empty(cap, dtype=torch.int64, device="cuda") if want else None
        ranges = torch.full((views * ((W + 15) // 16) * ((H + 15) // 16), 2), 7,
                            dtype=torch.int32, device="cuda")
        before = _lib.veg_kernel_launches()
        _lib.veg_bin_sort(cc, n, geo, tiles, rect, ws, cap, keys, vals, ranges)
        took.append(_lib.veg_kernel_launches() - before)
        st, count = _lib.veg_sync_status(ws)
        assert count == m and (st == _lib.VEG_OK) == (cap >= m)
        got.append((vals[:min(m, cap)].cpu().numpy(), ranges.cpu().numpy()))
    return m, got, took[0] - took[1] != 1


@pytest.mark.parametrize("n,views,W,H,wide", [(40_000, 1, 400, 272, 30), (65_537, 1, 512, 512, 9),
                                              (3000, 2, 400, 400, 25)])
@pytest.mark.parametrize("cap,cells", [(LINE - 1, False), (LINE, True), (LINE + 300_000, True)])
def test_the_line_by_capacity(n, views, W, H, wide, cap, cells):
    m, got, took = binned(n, views, W, H, wide, cap)
    assert took == cells
    assert np.array_equal(got[0][1], got[1][1]) and np.array_equal(got[0][0], got[1][0])


def test_few_lists_and_few_records_keep_the_sort():
    assert not binned(40_000, 1, 256, 256, 9, 2 * LINE)[2]  # 256 lists
    assert not binned(1023, 1, 800, 800, 30, 2 * LINE)[2]


@pytest.mark.parametrize("n,views,W,H,wide", [(60_000, 1, 400, 272, 30), (100_000, 1, 513, 257, 40)])
def test_a_cut_list_of_the_cells(n, views, W, H, wide):
    m = binned(n, views, W, H, wide, LINE)[0]
    assert m > LINE + 1000  # the line itself cuts
    m, got, took = binned(n, views, W, H, wide, LINE + 1)
    assert took and np.array_equal(got[0][1], got[1][1]) and np.array_equal(got[0][0], got[1][0])
