"""Eigenvalues follow the units of the Hamiltonian: times a power of two, every
step of the solvers is the same up to that power, so the energies are equal bit
for bit after it."""
import numpy as np
import pytest

import ed_inputs as ei
from gpu_util import gpu, to_torch

pytestmark = pytest.mark.gpu


def energies(ed, n, exponent, steps):
    h = ei.xxz_ring(n, 1.0, 1.5)
    O = ed.operator_create(n, h["sites"], h["coeff"] * 2.0 ** exponent, h["local"])
    B = ed.basis_build(n, n // 2, +1, *ei.ring_group(n, 0, +1))
    x = to_torch(ei.x_by_index(2, ed.basis_size(B), 1)[:, 0], np.float64)
    out = [ed.lanczos(O, B, x, steps).e0]
    out += list(ed.lanczos_eigs(O, B, x, steps, 3)[0])
    items = []
    for k in (0, 1, n // 2):
        b = ed.basis_build(n, n // 2, 0, *ei.ring_group(n, k))
        items.append((b, to_torch(ei.x_by_index(k, ed.basis_size(b), 1, True)[:, 0], np.complex128), None))
    out += [r.e0 for r in ed.lanczos_multi(O, items, steps)] + [r.ritz for r in ed.lanczos_multi(O, items, steps)]
    X = to_torch(ei.x_by_index(3, ed.basis_size(B), 2), np.float64)
    eigs, r = ed.lanczos_block(O, B, X, 2, 12, ed.ED_LANCZOS_F64, n_eig=2)
    return np.array(out), np.array(list(eigs) + [r.e0])


@pytest.mark.parametrize("exponent", [-300, -250, 40, 250, 300])
def test_energies_scale_with_the_hamiltonian(exponent):
    torch, ed = gpu()
    one, block = energies(ed, 16, 0, 30)
    got, got_block = energies(ed, 16, exponent, 30)
    assert np.array_equal(got, one * 2.0 ** exponent)
    # the block recurrence carries single-precision pairs, whose range is less
    if abs(exponent) <= 40:
        assert np.array_equal(got_block, block * 2.0 ** exponent)
