"""The dot products of the Lanczos recurrence are compensated fp64 sums: small
contributions beside large ones are not lost."""
import math

import numpy as np
import pytest

import ed_inputs as ei
from gpu_util import gpu, to_torch

pytestmark = pytest.mark.gpu


def start_vector(dim):
    """2000 large entries, then entries whose squares are just under half a unit
    in the last place of theirs; the fp64 norm is exactly 1."""
    x = np.full(dim, 1.0)
    x[2000:] = math.sqrt(0.47 * 2.0 ** -52)  # the large squares lie just above 2 ** -11
    x /= math.sqrt(math.fsum(x * x))
    for _ in range(100):
        off = math.fsum(x * x) - 1.0
        if off == 0.0:
            return x
        x[0] -= 0.5 * off / x[0]
    raise AssertionError("no start vector of norm 1")


def test_first_alpha_is_compensated():
    torch, ed = gpu()
    n, m = 16, 8
    # 1 on every bond: H is 16 times the identity, products exact but for x's own rounding
    h = ei.heisenberg_ring(n)
    local = np.zeros((n, 16, 2))
    local[:, [0, 5, 10, 15], 0] = 1.0
    coeff = np.zeros((n, 2))
    coeff[:, 0] = 1.0
    O = ed.operator_create(n, h["sites"], coeff, local)
    p = np.arange(n, dtype=np.int32).reshape(1, n)
    B = ed.basis_build(n, m, 0, p, np.array([[1.0, 0.0]]))
    dim = ed.basis_size(B)
    assert dim == math.comb(n, m)
    x = start_vector(dim)
    want = math.fsum(16.0 * (x * x))
    for vectors in (ed.ED_LANCZOS_F64, ed.ED_LANCZOS_F64 | ed.ED_LANCZOS_RECOMPUTE):
        r = ed.lanczos(O, B, to_torch(x, np.float64), 1, vectors | ed.ED_LANCZOS_VALUES_ONLY)
        # the sum rounded once, give or take the last place
        assert abs(r.e0 - want) <= 2.0 ** -52 * want
