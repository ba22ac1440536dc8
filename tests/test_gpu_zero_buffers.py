"""Zeroing many buffers: more than a launch takes, empty ones, unaligned ends,
and a tensor with gaps, whose neighbours stay."""
import pytest
import torch

from paper_2504_13339_gb300 import _lib

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module", autouse=True)
def built():
    import __graft_entry__
    __graft_entry__.build()


@pytest.mark.parametrize("count", [0, 1, 5, 8, 9, 17])
def test_every_byte_of_every_buffer_and_no_other(count):
    big = torch.full((count + 1, 1 << 16), 7, dtype=torch.uint8, device="cuda")
    sizes = [(0, 1, 3, 16, 17, 1000, 65000, 4096, 31)[i % 9] for i in range(count)]
    offs = [(5 * i) % 23 for i in range(count)]
    _lib.veg_zero_buffers([big[i, o:o + s] for i, (o, s) in enumerate(zip(offs, sizes))])
    want = torch.full_like(big, 7)
    for i, (o, s) in enumerate(zip(offs, sizes)):
        want[i, o:o + s] = 0
    assert torch.equal(big, want)


def test_a_tensor_with_gaps_leaves_its_neighbours():
    big = torch.ones(100, 8, device="cuda")
    flat = torch.ones(40, device="cuda")
    _lib.veg_zero_buffers([flat, big[:, 2:6]])
    assert (flat == 0).all() and (big[:, 2:6] == 0).all()
    assert (big[:, :2] == 1).all() and (big[:, 6:] == 1).all()


def test_buffers_beyond_a_grid_of_one_pass():
    bufs = [torch.ones(n, device="cuda") for n in (50_000_003, 12_345_677, 1)]
    _lib.veg_zero_buffers(bufs)
    assert all((b == 0).all() for b in bufs)
