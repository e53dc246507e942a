"""Groups and operators whose tables nearly fill a block's shared memory: products
that fit without the round sums of the small-sector kernel still run."""
import itertools

import numpy as np
import pytest

import ed_inputs as ei
from gpu_util import gpu, rel_err, to_torch

pytestmark = pytest.mark.gpu

N, PAIRS = 64, 10


def swaps():
    """The 1024 products of swaps of sites (2p, 2p + 1), p < 10."""
    out = []
    for which in itertools.product((0, 1), repeat=PAIRS):
        p = np.arange(N, dtype=np.int32)
        for q, s in enumerate(which):
            if s:
                p[[2 * q, 2 * q + 1]] = p[[2 * q + 1, 2 * q]]
        out.append(p)
    return np.array(out), np.array([[1.0, 0.0]] * len(out))


def operator(n_zz):
    """Exchange within the pairs and on a ring of the other sites, and n_zz
    couplings of their own between those."""
    free = range(2 * PAIRS, N)
    exchange = [(2 * q, 2 * q + 1) for q in range(PAIRS)] + [(i, i + 1 if i + 1 < N else 2 * PAIRS) for i in free]
    zz = list(itertools.combinations(free, 2))[:n_zz]
    sites = np.array(exchange + zz, np.int32)
    local = np.zeros((len(sites), 16, 2))
    local[:len(exchange), [6, 9], 0] = 0.5
    z = np.diag([1.0, -1.0, -1.0, 1.0]).reshape(16)
    local[len(exchange):, :, 0] = np.linspace(0.1, 1.0, len(zz))[:, None] * z
    coeff = np.zeros((len(sites), 2))
    coeff[:, 0] = 1.0
    return sites, coeff, local


@pytest.mark.parametrize("dtype", [np.float32, np.complex64])
# bytes of the tables: some 98304 (masks) + 1024 + 8200 + warps + 148 per coupling
@pytest.mark.parametrize("n_zz", [400, 760, 780, 790])
def test_small_sector_with_large_tables(dtype, n_zz):
    torch, ed = gpu()
    sites, coeff, local = operator(n_zz)
    O = ed.operator_create(N, sites, coeff, local)
    B = ed.basis_build(N, 2, 0, *swaps())
    x = to_torch(ei.x_by_index(4, ed.basis_size(B), 1, True)[:, 0].real, dtype)
    try:
        got = {}
        for policy in ("slots", "term_parallel"):
            ed.kernel_policy(policy)
            got[policy] = ed.matvec(O, B, x, torch.full_like(x, float("nan"))).cpu().numpy()
    finally:
        ed.kernel_policy("auto")
    # sums of some 60 couplings and a few exchanges of O(1) numbers in single precision
    assert rel_err(got["term_parallel"], got["slots"]) < 1e-5
