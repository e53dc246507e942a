"""Basis builds and batch solves on a stream that is still busy with earlier
work: the host tables they upload are read only once the stream gets there."""
import numpy as np
import pytest

import ed_inputs as ei
from gpu_util import build_pair, gpu, to_torch

pytestmark = pytest.mark.gpu


def busy(torch):
    s = torch.cuda.Stream()
    with torch.cuda.stream(s):
        torch.cuda._sleep(100_000_000)  # some 50 ms
    return s


@pytest.mark.parametrize("n,n_up,z", [(16, 8, +1), (24, 12, 0), (32, 16, +1)])  # one cell; many at 32 sites
def test_build_behind_queued_work(n, n_up, z):
    torch, ed = gpu()
    p, c = ei.ring_group(n, 0, +1)
    S = build_pair(n, n_up, z, p, c, ei.heisenberg_ring(n), with_oracle=False)
    x = to_torch(ei.x_by_index(5, S["dim"], 1)[:, 0], np.float64)
    want = ed.matvec(S["O"], S["B"], x, torch.empty_like(x))
    s = busy(torch)
    B = ed.basis_build(n, n_up, z, p, c, stream=s)
    assert ed.basis_slots(B) == ed.basis_slots(S["B"])
    y = torch.full_like(x, float("nan"))
    s.wait_stream(torch.cuda.current_stream())
    ed.matvec(S["O"], B, x, y, stream=s)
    s.synchronize()
    assert torch.equal(y, want)


def test_batch_solve_behind_queued_work():
    torch, ed = gpu()
    h = ei.xxz_ring(12, 1.0, 1.5)
    O = ed.operator_create(12, h["sites"], h["coeff"], h["local"])
    items = []
    for k in range(12):
        p, c = ei.ring_group(12, k)
        B = ed.basis_build(12, 6, 0, p, c)
        items.append((B, to_torch(ei.x_by_index(k, ed.basis_size(B), 1, True)[:, 0], np.complex128), None))
    want = [r.e0 for r in ed.lanczos_multi(O, items, 20, ed.ED_LANCZOS_F64)]
    torch.cuda.synchronize()
    got = [r.e0 for r in ed.lanczos_multi(O, items, 20, ed.ED_LANCZOS_F64, stream=busy(torch))]
    assert got == want
