"""Enumeration by viable top bits (sectors of at least 2^20 states before
symmetry) against the oracle's brute force: basis, norms, order and dimension,
for rings (odd words only), tori and groups with a coset of their own, with and
without spin inversion and Sz conservation, 32- and 64-bit words."""
import numpy as np
import pytest

import ed_inputs as ei
import oracle
from gpu_util import gpu, gpu_basis_numpy
from test_gpu_parity import affine_group

pytestmark = pytest.mark.gpu

CASES = {
    "ring24_k0_p+_z+": (24, 12, +1, lambda: ei.ring_group(24, 0, +1)),
    "ring24_k12_p-_z-": (24, 12, -1, lambda: ei.ring_group(24, 12, -1)),
    "ring23_k3": (23, 10, 0, lambda: ei.ring_group(23, 3)),
    "ring34_nup6_k1": (34, 6, 0, lambda: ei.ring_group(34, 1)),
    "ring44_nup5_k0_p+": (44, 5, 0, lambda: ei.ring_group(44, 0, +1)),
    "ring20_noU1_z+": (20, -1, +1, lambda: ei.ring_group(20, 0)),
    "torus4x6_z-": (24, 12, -1, lambda: ei.torus_group(4, 6, 2, 3)),
    "torus6x4_k10": (24, 11, 0, lambda: ei.torus_group(6, 4, 1, 0)),
    "affine24_a7": (24, 12, +1, lambda: affine_group(24, 7, -1.0)),
}


@pytest.mark.parametrize("name", CASES)
def test_basis_bit_exact(name):
    torch, ed = gpu()
    n, n_up, z, grp = CASES[name]
    p, c = grp()
    B = ed.basis_build(n, n_up, z, p, c)
    G = oracle.Group(n, p, c, z)
    st, nm = oracle.enumerate_basis(G, n_up)
    got_st, got_nm = gpu_basis_numpy(B)
    assert np.array_equal(got_st, st) and np.array_equal(got_nm, nm)
    assert ed.basis_count(n, n_up, z, p, c) == len(st)
