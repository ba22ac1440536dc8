"""A radix sort whose wait ran out writes nothing outside its buffers: the
passes after it read places that nothing was written to, here keys of all
ones, whose digits no total has counted."""
import pytest
import torch

from paper_2504_13339_gb300 import _lib

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module", autouse=True)
def built():
    import __graft_entry__
    __graft_entry__.build()


@pytest.mark.parametrize("n", [2 * 2048, 9 * 2048 + 77, 64 * 2048])
def test_a_timed_out_sort_stays_in_its_buffers(n):
    size = _lib.veg_bin_sort_workspace_size(n, 1, 0, 16, 16)
    ws = torch.full((size,), 0xff, dtype=torch.uint8, device="cuda")
    out = torch.empty(2, n, dtype=torch.int32, device="cuda")
    _lib.veg_radix_lookback_check(ws, n, True, 1 << 12, out[0], out[1])
    assert _lib.veg_sync_status(ws)[0] == _lib.VEG_ERR_TIMEOUT
    # header, keys and values twice, then the block sums, which this call leaves alone
    piece = (4 * n + 255) // 256 * 256
    sums = ws[256 + 4 * piece:256 + 4 * piece + 8 * (n // 256)]
    assert (sums == 0xff).all()
    pad = ws[256:256 + 4 * piece].view(4, piece)[:, 4 * n:]
    assert (pad == 0xff).all()
