"""Rounding of the slot product's row sums against the other kernels."""
import numpy as np
import pytest

import ed_inputs as ei
from gpu_util import build_pair, gpu, to_torch

pytestmark = pytest.mark.gpu


@pytest.fixture(autouse=True)
def default_kernels():
    torch, ed = gpu()
    yield
    ed.kernel_policy("auto")


ROUNDING = [
    ("ring26", 26, 13, +1, lambda: ei.ring_group(26, 0, +1), lambda: ei.heisenberg_ring(26), np.float32),
    ("ring26_k1", 26, 13, 0, lambda: ei.ring_group(26, 1), lambda: ei.xxz_ring(26, 1.0, 1.5), np.complex64),
    ("torus4x6_j1j2", 24, 12, 0, lambda: ei.torus_group(4, 6, 0, 0), lambda: ei.j1j2_torus(4, 6, 1.0, 0.5),
     np.float32),
    ("torus4x6_j1j2_k12", 24, 12, 0, lambda: ei.torus_group(4, 6, 1, 2), lambda: ei.j1j2_torus(4, 6, 1.0, 0.5),
     np.complex64),
]


@pytest.mark.parametrize("nvec", [1, 8])
@pytest.mark.parametrize("case", ROUNDING, ids=[s[0] for s in ROUNDING])
def test_rounding_error_of_the_row_sums(case, nvec):
    """The sums of a row in short chains: the rms distance of a single-precision
    product from the double-precision one is no larger than that of the kernels
    that add a row's terms as a tree or one by one (1e5 rows and more: the two
    estimates scatter by 0.3 %)."""
    torch, ed = gpu()
    name, n, n_up, z, grp, opf, dt = case
    p, c = grp()
    S = build_pair(n, n_up, z, p, c, opf(), with_oracle=False)
    x = to_torch(ei.x_by_index(17, S["dim"], nvec, True), np.complex128)
    x = (x if np.issubdtype(dt, np.complexfloating) else x.real.contiguous()).to(
        torch.complex64 if dt is np.complex64 else torch.float32)
    x64 = x.to(torch.complex128 if x.is_complex() else torch.float64)
    exact = ed.matvec(S["O"], S["B"], x64, torch.empty_like(x64), nvec)

    def rms(policy):
        ed.kernel_policy(policy)
        y = ed.matvec(S["O"], S["B"], x, torch.empty_like(x), nvec)
        return float((y.to(exact.dtype) - exact).abs().square().mean().sqrt())

    assert rms("slots") <= 1.01 * rms("term_parallel")
