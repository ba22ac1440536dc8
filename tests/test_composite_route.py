"""Which forward kernel a launch takes, asked of the library on the host: both
sides of the lines by records."""
import os
import shutil

import pytest

from paper_2504_13339_gb300 import _lib


@pytest.fixture(scope="module", autouse=True)
def lib():
    if shutil.which("nvcc") is None and not os.path.exists("/usr/local/cuda/bin/nvcc"):
        pytest.skip("nvcc not available")
    from paper_2504_13339_gb300 import build
    build.build()


def cams(tiles):
    c = (_lib.veg_camera * 1)()
    c[0].width, c[0].height, c[0].fx, c[0].fy = 16 * tiles, 16, 10.0, 10.0
    return c


@pytest.mark.parametrize("n,line", [(0, 640), (4095, 640), (4096, 1280), (65535, 1280),
                                    (65536, 1536), (10_000_000, 1536)])
def test_few_items_stage_no_batches(n, line):
    for tables in (2, 4):
        tf = _lib.veg_tf(0, 256, tables)
        ask = lambda tiles, b: _lib.veg_composite_fwd_batch(cams(tiles), n, tf, b)
        assert ask(line // tables - 1, 128) == 0
        assert [ask(line // tables, b) for b in (0, 128, 512)] == [256, 128, 512]


def test_a_table_per_view_is_one_item_per_tile():
    tf = _lib.veg_tf(0, 256, 64, 1 << 20)
    assert _lib.veg_composite_fwd_batch(cams(600), 100, tf, 0) == 0
    tf = _lib.veg_tf(0, 256, 64)
    assert _lib.veg_composite_fwd_batch(cams(700), 100, tf, 0) == 256
    with pytest.raises(_lib.VegError):
        _lib.veg_composite_fwd_batch(cams(700), 100, tf, 64)
