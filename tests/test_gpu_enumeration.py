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


SMALL = (
    [(f"ring{n}_k{k}_p{p}_z{z}", n, n // 2, z, lambda n=n, k=k, p=p: ei.ring_group(n, k, p))
     for n in (2, 4, 6, 8, 12, 16) for k, p in ((0, +1), (0, -1), (n // 2, None), (1, None)) for z in (0, +1, -1)
     if n > 2 or p is None]
    + [(f"ring{n}_noU1_z{z}", n, -1, z, lambda n=n: ei.ring_group(n, 0, +1)) for n in (3, 9, 12) for z in (0, +1)]
    + [(f"ring{n}_nup{u}_k{k}_p{p}", n, u, 0, lambda n=n, k=k, p=p: ei.ring_group(n, k, p))
       for n, u in ((33, 3), (48, 3), (49, 3), (60, 3), (64, 2), (64, 3)) for k, p in ((0, +1), (3, None))]
    + [(f"torus{a}x{b}_k{kx}{ky}_z{z}", a * b, -1, z, lambda a=a, b=b, kx=kx, ky=ky: ei.torus_group(a, b, kx, ky))
       for a, b in ((2, 4), (4, 2), (3, 3), (4, 4)) for kx, ky in ((0, 0), (1, 1)) for z in (0, +1)]
)


@pytest.mark.parametrize("case", SMALL, ids=[c[0] for c in SMALL])
def test_orbit_norms(case):
    """Norms of the states with every kind of symmetry (fixed by rotations,
    reflections, the complement of a half turn), against the oracle and against
    the search over every group element."""
    torch, ed = gpu()
    _, n, n_up, z, grp = case
    p, c = grp()
    got = gpu_basis_numpy(ed.basis_build(n, n_up, z, p, c))
    ed.force_all_rotations(True)
    try:
        every = gpu_basis_numpy(ed.basis_build(n, n_up, z, p, c))
    finally:
        ed.force_all_rotations(False)
    st, nm = oracle.enumerate_basis(oracle.Group(n, p, c, z), n_up)
    assert np.array_equal(got[0], st) and np.array_equal(got[1], nm)
    assert np.array_equal(every[0], st) and np.array_equal(every[1], nm)
