"""The slot index and the product over it, forced on small sectors (the library
builds it for large ones), against the oracle: every word width, search, type
and padding of the vector rows, sectors with weightless representatives, batches
of sectors, captured products.  Bars as in test_gpu_parity: each element is a
sum of a few dozen products of O(1) numbers, so fp64 within 1e-12 and fp32
within 2e-6 of the largest |y|."""
import numpy as np
import pytest

import ed_inputs as ei
import oracle
from gpu_util import build_pair, gpu, rel_err, to_torch
from test_gpu_parity import SECTORS

pytestmark = pytest.mark.gpu

EXTRA = [
    ("ring18_k9_p-_z-", 18, 9, -1, lambda: ei.ring_group(18, 9, -1), lambda: ei.xxz_ring(18, 1.0, 1.5)),
    ("torus6x6_nup3_k1", 36, 3, 0, lambda: ei.torus_group(6, 6, 1, 0), lambda: ei.j1j2_torus(6, 6, 1.0, 0.5)),
    ("torus4x5_k02", 20, 5, 0, lambda: ei.torus_group(4, 5, 0, 2), lambda: ei.j1j2_torus(4, 5, 1.0, 0.5)),
]
CASES = [s for s in SECTORS if s[0] not in ("ring8_empty", "ring10_noU1_xx_z-")] + EXTRA


@pytest.fixture(autouse=True)
def slots_everywhere():
    torch, ed = gpu()
    ed.kernel_policy("slots")
    yield
    ed.kernel_policy("auto")
    ed.force_generic(False)


@pytest.mark.parametrize("case", CASES, ids=[s[0] for s in CASES])
@pytest.mark.parametrize("generic", [False, True])
def test_products(case, generic):
    torch, ed = gpu()
    ed.force_generic(generic)
    name, n, n_up, z, grp, opf = case
    p, c = grp()
    S = build_pair(n, n_up, z, p, c, opf())
    present, slots, ghosts = ed.basis_slots(S["B"])
    assert present and slots >= S["dim"] + ghosts
    real = ed.basis_is_real(S["B"]) and not np.any(opf()["local"][:, :, 1])
    for nvec in (1, 3) if generic else (1, 2, 5, 8, 16):
        x = ei.x_by_index(41, S["dim"], nvec, True)
        if real:
            x = x.real.astype(np.complex128)
        want = np.stack([oracle.matvec(S["G"], S["H"], S["st"], S["nm"], x[:, v]) for v in range(nvec)], 1)
        kinds = [(np.complex128, 1e-12), (np.complex64, 2e-6)]
        if real:
            kinds += [(np.float64, 1e-12), (np.float32, 2e-6)]
        for dt, tol in kinds:
            cplx = np.issubdtype(dt, np.complexfloating)
            xt = to_torch(x if cplx else x.real, dt)
            yt = torch.full_like(xt, float("nan"))
            ed.matvec(S["O"], S["B"], xt, yt, nvec)
            got = yt.cpu().numpy()
            assert rel_err(got, want if cplx else want.real) < tol, (nvec, dt)
            again = torch.empty_like(xt)
            ed.matvec(S["O"], S["B"], xt, again, nvec)
            assert torch.equal(yt, again)


@pytest.mark.parametrize("n,lx", [(12, 0), (16, 4)])
def test_batch_equals_single_products(n, lx):
    torch, ed = gpu()
    op = ei.j1j2_torus(lx, n // lx, 1.0, 0.3) if lx else ei.xxz_ring(n, 0.7, 1.5)
    O = ed.operator_create(n, op["sites"], op["coeff"], op["local"])
    for dt, nvec in ((torch.complex128, 1), (torch.complex64, 3), (torch.complex64, 8)):
        items, alone = [], []
        for n_up, k, z in ((n // 2, 0, 1), (n // 2, 1, -1), (n // 2 + 1, 2, 0), (n // 2 + 1, 0, 0), (n // 2, 3, 1)):
            p, c = ei.torus_group(lx, n // lx, k % lx, 1) if lx else ei.ring_group(n, k)
            B = ed.basis_build(n, n_up, z, p, c)
            d = ed.basis_size(B)
            x = to_torch(ei.x_by_index(7 + k, d, nvec, True), np.complex128).to(dt)
            items.append((B, x, torch.full_like(x, float("nan"))))
            alone.append(ed.matvec(O, B, x, torch.empty_like(x), nvec))
        ed.matvec_multi(O, items, nvec)
        for (_, _, y), want in zip(items, alone):
            assert torch.equal(y, want)


def test_captured_product_replays():
    torch, ed = gpu()
    p, c = ei.ring_group(20, 0, +1)
    S = build_pair(20, 10, +1, p, c, ei.heisenberg_ring(20), with_oracle=False)
    x = to_torch(ei.x_by_index(1, S["dim"], 1)[:, 0], np.float64)
    want, y = torch.empty_like(x), torch.zeros_like(x)
    ed.matvec(S["O"], S["B"], x, want)
    torch.cuda.synchronize()
    g = torch.cuda.CUDAGraph()
    with torch.cuda.graph(g):
        ed.matvec(S["O"], S["B"], x, y)
    for _ in range(3):
        y.zero_()
        g.replay()
        torch.cuda.synchronize()
        assert torch.equal(y, want)


def test_products_on_two_streams():
    torch, ed = gpu()
    p, c = ei.ring_group(20, 3)
    S = build_pair(20, 10, 0, p, c, ei.xxz_ring(20, 1.0, 1.5), with_oracle=False)
    xs = [to_torch(ei.x_by_index(s, S["dim"], 1, True)[:, 0], np.complex128) for s in (1, 2)]
    want = [ed.matvec(S["O"], S["B"], x, torch.empty_like(x)).clone() for x in xs]
    torch.cuda.synchronize()
    streams = [torch.cuda.Stream(), torch.cuda.Stream()]
    ys = [torch.empty_like(x) for x in xs]
    for _ in range(20):
        for s, x, y in zip(streams, xs, ys):
            ed.matvec(S["O"], S["B"], x, y, stream=s)
    torch.cuda.synchronize()
    for y, w in zip(ys, want):
        assert torch.equal(y, w)
