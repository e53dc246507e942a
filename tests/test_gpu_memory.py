"""Calls that are refused the work memory they can do without give the results
they give with it."""
import numpy as np
import pytest

import ed_inputs as ei
from gpu_util import gpu, gpu_basis_numpy

pytestmark = pytest.mark.gpu


@pytest.fixture(autouse=True)
def no_limit_afterwards():
    torch, ed = gpu()
    yield
    ed.optional_memory(None)


@pytest.mark.parametrize("n,n_up,z,grp", [
    (24, 12, +1, lambda: ei.ring_group(24, 0, +1)),
    (23, 10, 0, lambda: ei.ring_group(23, 3)),
    (24, 12, -1, lambda: ei.torus_group(4, 6, 2, 3)),
], ids=["ring24", "ring23_k3", "torus4x6"])
# none of it; only arrays of a few kilobytes
@pytest.mark.parametrize("limit", [0, 1 << 14])
def test_enumeration_without_the_prefix_filter(n, n_up, z, grp, limit):
    torch, ed = gpu()
    p, c = grp()
    want = gpu_basis_numpy(ed.basis_build(n, n_up, z, p, c))
    ed.optional_memory(limit)
    B = ed.basis_build(n, n_up, z, p, c)
    got = gpu_basis_numpy(B)
    assert np.array_equal(got[0], want[0]) and np.array_equal(got[1], want[1])
    assert not ed.basis_slots(B)[0]
    assert ed.basis_count(n, n_up, z, p, c) == len(want[0])
