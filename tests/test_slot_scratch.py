"""When a solver takes the memory of the slotted copy (host rule, no GPU)."""
import os

import pytest


@pytest.fixture(scope="module")
def fits():
    from paper_2308_16712_gb300 import build
    if not os.path.exists(build.LIB):
        build.build()
    from paper_2308_16712_gb300 import ed
    return ed._lib.edx_slot_scratch_fits


def copy_bytes(dim, row):
    return dim * 8533 // 7168 * row


@pytest.mark.parametrize("dim,row,vectors", [
    # 8 fp32 vectors on ring N=40 in 298 GB: basis, fp64 start block, two blocks of
    # float pairs, the product, three vectors
    (861725794, 32, 32 + 64 + 128 + 32 + 16),
    # one fp64 vector on ring N=40: basis, start, work and two ring vectors
    (861725794, 8, 32 + 8 * 5),
])
def test_large_blocks_take_it_when_it_fits(fits, dim, row, vectors):
    free = 298 * 10 ** 9 - 2 * 10 ** 9 - dim * vectors
    assert fits(copy_bytes(dim, row), free, 0)


def test_room_is_left_for_later_allocations(fits):
    gb = 1 << 30
    assert fits(10 * gb, 11 * gb, 0)
    assert not fits(10 * gb, 11 * gb, gb)
    assert not fits(11 * gb, 11 * gb, 0)
    assert not fits(10 * gb, 10 * gb + (256 << 20), 0)
