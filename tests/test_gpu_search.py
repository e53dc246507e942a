"""The pruned representative searches (ring runs, torus row keys) on the GPU
against the oracle's brute force, at the sizes where their word handling
changes: full words, words just above 32 bits, words too long to be held twice
in 64 bits, rows of 2 to 8 sites, keys of one row and of several."""
import numpy as np
import pytest

import ed_inputs as ei
import oracle
from gpu_util import build_pair, gpu, gpu_basis_numpy, rel_err, to_torch

pytestmark = pytest.mark.gpu

TORI = [(2, 8, 8, 1), (2, 16, 3, 0), (3, 4, 6, 1), (4, 4, 8, -1), (8, 4, 3, 0), (5, 5, 6, 0), (6, 6, 3, 0),
        (7, 5, 4, 0), (4, 10, 3, 0), (8, 8, 2, 0)]
RINGS = [(6, 3, 1), (17, 8, 0), (31, 4, 0), (32, 4, 0), (33, 4, 0), (48, 3, 0), (49, 3, 0), (63, 2, 0)]


def check(n, n_up, z, perms, chars, op):
    torch, ed = gpu()
    S = build_pair(n, n_up, z, perms, chars, op)
    st, nm = gpu_basis_numpy(S["B"])
    assert np.array_equal(st, S["st"]) and np.array_equal(nm, S["nm"])
    if not S["dim"]:
        return
    x = ei.x_by_index(3, S["dim"], 1, True)[:, 0]
    want = oracle.matvec(S["G"], S["H"], S["st"], S["nm"], x)
    for kernel in ("rowwise", "term_parallel"):
        ed.kernel_policy(kernel)
        try:
            xt = to_torch(x, np.complex128)
            got = ed.matvec(S["O"], S["B"], xt, torch.empty_like(xt)).cpu().numpy()
        finally:
            ed.kernel_policy("auto")
        assert rel_err(got, want) < 1e-12  # a few dozen terms of O(1), fp64


@pytest.mark.parametrize("lx,ly,n_up,z", TORI)
def test_torus_translations(lx, ly, n_up, z):
    for kx, ky in ((0, 0), (1, ly // 2)):
        p, c = ei.torus_group(lx, ly, kx, ky)
        check(lx * ly, n_up, z, p, c, ei.j1j2_torus(lx, ly, 1.0, 0.5))


@pytest.mark.parametrize("n,n_up,z", RINGS)
def test_ring_translations(n, n_up, z):
    for k, parity in ((0, 1), (1, None)):
        p, c = ei.ring_group(n, k, parity)
        check(n, n_up, z, p, c, ei.xxz_ring(n, 1.0, 1.5))


def test_torus_sectors_with_and_without_inversion_in_one_launch():
    torch, ed = gpu()
    op = ei.j1j2_torus(4, 4, 1.0, 0.5)
    O = ed.operator_create(16, op["sites"], op["coeff"], op["local"])
    items, alone = [], []
    for z, kx in ((0, 1), (1, 0), (-1, 2)):
        p, c = ei.torus_group(4, 4, kx, 1)
        B = ed.basis_build(16, 8, z, p, c)
        x = to_torch(ei.x_by_index(5, ed.basis_size(B), 1, True)[:, 0], np.complex128)
        items.append((B, x, torch.zeros_like(x)))
        alone.append(ed.matvec(O, B, x, torch.zeros_like(x)))
    ed.matvec_multi(O, items)
    for (_, _, y), want in zip(items, alone):
        assert torch.equal(y, want)
