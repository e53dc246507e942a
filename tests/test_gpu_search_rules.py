"""The row-per-lane kernel's choice of search on a torus (every element below 2^17
states, the table above): both sides of the line against the search over every
element, and a batch with sectors of both kinds against the single products."""
import numpy as np
import pytest

import ed_inputs as ei
from gpu_util import build_pair, gpu, to_torch

pytestmark = pytest.mark.gpu


@pytest.fixture(autouse=True)
def rowwise():
    torch, ed = gpu()
    ed.kernel_policy("rowwise")
    yield
    ed.kernel_policy("auto")
    ed.force_all_rotations(False)


@pytest.mark.parametrize("n_up", [3, 12])  # 92 and 208012 states
@pytest.mark.parametrize("kx", [0, 1])
@pytest.mark.parametrize("nvec", [1, 3])
def test_both_searches(n_up, kx, nvec):
    torch, ed = gpu()
    p, c = ei.torus_group(5, 5, kx, 0)
    S = build_pair(25, n_up, 0, p, c, ei.j1j2_torus(5, 5, 1.0, 0.5), with_oracle=False)
    x = to_torch(ei.x_by_index(6, S["dim"], nvec, True), np.complex128)
    got = ed.matvec(S["O"], S["B"], x, torch.empty_like(x), nvec)
    ed.force_all_rotations(True)
    want = ed.matvec(S["O"], S["B"], x, torch.empty_like(x), nvec)
    # the minimiser may differ by an element that fixes the minimum: characters
    # equal to their rounding
    assert float((got - want).abs().max()) <= 1e-14 * float(want.abs().max())


def test_batch_of_both_kinds():
    torch, ed = gpu()
    h = ei.j1j2_torus(5, 5, 1.0, 0.5)
    O = ed.operator_create(25, h["sites"], h["coeff"], h["local"])
    items, alone = [], []
    for n_up, kx in ((12, 0), (3, 1), (12, 2), (4, 0)):
        B = ed.basis_build(25, n_up, 0, *ei.torus_group(5, 5, kx, 0))
        x = to_torch(ei.x_by_index(n_up, ed.basis_size(B), 1, True)[:, 0], np.complex128)
        items.append((B, x, torch.full_like(x, float("nan"))))
        alone.append(ed.matvec(O, B, x, torch.empty_like(x)))
    ed.matvec_multi(O, items)
    for (_, _, y), want in zip(items, alone):
        assert torch.equal(y, want)
