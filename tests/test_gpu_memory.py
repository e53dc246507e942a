"""Calls that are refused the work memory they can do without give the results
they give with it, bit for bit, and so do captured products, whose graphs hold no
allocation."""
import ctypes

import numpy as np
import pytest

import ed_inputs as ei
from gpu_util import build_pair, gpu, gpu_basis_numpy, to_torch
from test_gpu_slots import CASES

pytestmark = pytest.mark.gpu


@pytest.fixture(autouse=True)
def no_limit_afterwards():
    torch, ed = gpu()
    yield
    ed.optional_memory(None)
    ed.kernel_policy("auto")
    ed.index_policy("auto")
    ed.force_generic(False)


@pytest.mark.parametrize("n,n_up,z,grp", [
    (24, 12, +1, lambda: ei.ring_group(24, 0, +1)),
    (23, 10, 0, lambda: ei.ring_group(23, 3)),
    (24, 12, -1, lambda: ei.torus_group(4, 6, 2, 3)),
], ids=["ring24", "ring23_k3", "torus4x6"])
# none of it; only arrays of a few kilobytes
@pytest.mark.parametrize("limit", [0, 1 << 14])
def test_enumeration_without_the_prefix_filter(n, n_up, z, grp, limit):
    torch, ed = gpu()
    p, c = grp()
    want = gpu_basis_numpy(ed.basis_build(n, n_up, z, p, c))
    ed.optional_memory(limit)
    B = ed.basis_build(n, n_up, z, p, c)
    got = gpu_basis_numpy(B)
    assert np.array_equal(got[0], want[0]) and np.array_equal(got[1], want[1])
    assert not ed.basis_slots(B)[0]
    assert ed.basis_count(n, n_up, z, p, c) == len(want[0])


@pytest.mark.parametrize("case", CASES, ids=[s[0] for s in CASES])
@pytest.mark.parametrize("index,generic", [("hash", False), ("bucket", False), ("hash", True)])
def test_products_without_the_copy(case, index, generic):
    torch, ed = gpu()
    ed.kernel_policy("slots")
    ed.index_policy(index)
    ed.force_generic(generic)
    name, n, n_up, z, grp, opf = case
    p, c = grp()
    S = build_pair(n, n_up, z, p, c, opf(), with_oracle=False)
    assert ed.basis_slots(S["B"])[0]
    real = ed.basis_is_real(S["B"]) and not np.any(opf()["local"][:, :, 1])
    for nvec in (1, 2, 3, 5, 8, 16):
        x = ei.x_by_index(43, S["dim"], nvec, True)
        for dt in (np.complex128, np.complex64) + ((np.float64, np.float32) if real else ()):
            xt = to_torch(x if np.issubdtype(dt, np.complexfloating) else x.real, dt)
            want, got = torch.empty_like(xt), torch.full_like(xt, float("nan"))
            ed.optional_memory(None)
            ed.matvec(S["O"], S["B"], xt, want, nvec)
            ed.optional_memory(0)
            ed.matvec(S["O"], S["B"], xt, got, nvec)
            assert torch.equal(got, want), (nvec, dt)


def sectors(ed, n, lx):
    """Sectors of a batch (basis, spin inversion or not, trivial characters or not)."""
    op = ei.j1j2_torus(lx, n // lx, 1.0, 0.3) if lx else ei.xxz_ring(n, 0.7, 1.5)
    O = ed.operator_create(n, op["sites"], op["coeff"], op["local"])
    bases = []
    for n_up, k, z in ((n // 2, 0, 1), (n // 2, 1, -1), (n // 2 + 1, 2, 0), (n // 2 + 1, 0, 0), (n // 2, 3, 1)):
        p, c = ei.torus_group(lx, n // lx, k % lx, 0) if lx else ei.ring_group(n, k)
        bases.append(ed.basis_build(n, n_up, z, p, c))
    return O, bases


# nothing; one group of two (the copies of its sectors, 137 to 546 KB); all but the largest
@pytest.mark.parametrize("limit", [0, 300_000, 500_000])
@pytest.mark.parametrize("n,lx", [(14, 0), (16, 4)])
def test_batch_without_the_copies(n, lx, limit):
    torch, ed = gpu()
    ed.kernel_policy("slots")
    O, bases = sectors(ed, n, lx)
    for dt, nvec in ((torch.complex128, 1), (torch.complex64, 3), (torch.complex64, 8)):
        xs = [to_torch(ei.x_by_index(9 + k, ed.basis_size(b), nvec, True), np.complex128).to(dt)
              for k, b in enumerate(bases)]
        want = [ed.matvec(O, b, x, torch.empty_like(x), nvec) for b, x in zip(bases, xs)]
        ys = [torch.full_like(x, float("nan")) for x in xs]
        ed.optional_memory(limit)
        ed.matvec_multi(O, list(zip(bases, xs, ys)), nvec)
        ed.optional_memory(None)
        for y, w in zip(ys, want):
            assert torch.equal(y, w)


def node_types(graph):
    rt = ctypes.CDLL("libcudart.so.13")
    g, n = ctypes.c_void_p(graph.raw_cuda_graph()), ctypes.c_size_t(0)
    assert rt.cudaGraphGetNodes(g, None, ctypes.byref(n)) == 0
    nodes = (ctypes.c_void_p * n.value)()
    assert rt.cudaGraphGetNodes(g, nodes, ctypes.byref(n)) == 0
    out = []
    for node in nodes:
        t = ctypes.c_int(-1)
        assert rt.cudaGraphNodeGetType(ctypes.c_void_p(node), ctypes.byref(t)) == 0
        out.append(t.value)
    return out


def test_captured_products_hold_no_allocation():
    torch, ed = gpu()
    O, bases = sectors(ed, 14, 0)
    xs = [to_torch(ei.x_by_index(k, ed.basis_size(b), 1, True)[:, 0], np.complex128) for k, b in enumerate(bases)]
    want = [ed.matvec(O, b, x, torch.empty_like(x)) for b, x in zip(bases, xs)]
    ys = [torch.zeros_like(x) for x in xs]
    ed.matvec_multi(O, list(zip(bases, xs, ys)))
    torch.cuda.synchronize()

    def one():
        ed.matvec(O, bases[0], xs[0], ys[0])

    def batch():
        ed.matvec_multi(O, list(zip(bases, xs, ys)))

    for call, done in ((one, 1), (batch, len(bases))):
        g = torch.cuda.CUDAGraph(keep_graph=True)
        with torch.cuda.graph(g):
            call()
        types = node_types(g)
        assert types and not {10, 11} & set(types)  # cudaGraphNodeTypeMemAlloc, MemFree
        for _ in range(2):
            for y in ys:
                y.zero_()
            g.replay()
            torch.cuda.synchronize()
            for y, w in list(zip(ys, want))[:done]:
                assert torch.equal(y, w)


@pytest.mark.parametrize("mode", ["f64", "f64_recompute", "f32_recompute", "block_f32", "block_f64", "multi"])
@pytest.mark.parametrize("graph", [0, 1])
def test_solvers_without_the_copy(mode, graph):
    torch, ed = gpu()
    n = 20
    h = ei.xxz_ring(n, 1.0, 1.5)
    O = ed.operator_create(n, h["sites"], h["coeff"], h["local"])
    p, c = ei.ring_group(n, 0, +1)
    B = ed.basis_build(n, n // 2, +1, p, c)
    x = to_torch(ei.x_by_index(2, ed.basis_size(B), 8), np.float64)
    bases = [ed.basis_build(n, n // 2 + 1, 0, *ei.ring_group(n, k)) for k in (0, 1, 10)]
    items = [(b, to_torch(ei.x_by_index(k, ed.basis_size(b), 1, True)[:, 0], np.complex128), None)
             for k, b in enumerate(bases)]

    def run():
        v = torch.empty(x.shape[0], dtype=x.dtype, device=x.device)
        if mode == "multi":
            return [r.e0 for r in ed.lanczos_multi(O, items, 20, ed.ED_LANCZOS_F64)], v.zero_()
        if mode.startswith("block"):
            m = ed.ED_LANCZOS_F32_MATVEC if mode.endswith("f32") else ed.ED_LANCZOS_F64
            return ed.lanczos_block(O, B, x, 8, 12, m, vec_out=v)[1].e0, v
        m = ed.ED_LANCZOS_F64 if mode.startswith("f64") else ed.ED_LANCZOS_F32_MATVEC
        if mode.endswith("recompute"):
            m |= ed.ED_LANCZOS_RECOMPUTE
        return ed.lanczos(O, B, x[:, 0].contiguous(), 20, m, v).e0, v

    old = ed.lanczos_graph(graph)
    try:
        want = run()
        ed.optional_memory(0)
        got = run()
    finally:
        ed.lanczos_graph(old)
    assert got[0] == want[0] and torch.equal(got[1], want[1])


def served(ed, call):
    before = ed.product_counts()
    call()
    return {k: v - before[k] for k, v in ed.product_counts().items() if v > before[k]}


def test_product_counts_name_the_kernel_that_ran():
    torch, ed = gpu()
    p, c = ei.ring_group(20, 0, +1)
    S = build_pair(20, 10, +1, p, c, ei.heisenberg_ring(20), with_oracle=False)
    x = to_torch(ei.x_by_index(1, S["dim"], 8), np.float32)
    y = torch.empty_like(x)
    x64 = x.to(torch.float64)

    def product():
        ed.matvec(S["O"], S["B"], x, y, 8)

    def block():
        ed.lanczos_block(S["O"], S["B"], x64, 8, 12, ed.ED_LANCZOS_F32_MATVEC | ed.ED_LANCZOS_VALUES_ONLY)

    def batch():
        ed.matvec_multi(S["O"], [(S["B"], x, y)], 8)

    assert served(ed, product) == served(ed, batch) == {"slot": 1}
    assert served(ed, block) == {"slot": 12}
    ed.optional_memory(0)
    assert served(ed, product) == served(ed, batch) == {"slot without copy": 1}
    assert served(ed, block) == {"slot without copy": 12}
    for policy, name in (("rowwise", "row-per-lane"), ("term_parallel", "term-parallel")):
        ed.kernel_policy(policy)
        assert served(ed, product) == {name: 1}
        assert served(ed, block) == {name: 12}


def test_small_sectors_take_one_launch():
    torch, ed = gpu()
    h = ei.heisenberg_ring(20)
    O = ed.operator_create(20, h["sites"], h["coeff"], h["local"])
    for (z, grp), one in (((+1, ei.ring_group(20, 0, +1)), True), ((0, ei.ring_group(20, 0)), True),
                          ((+1, (np.arange(20, dtype=np.int32).reshape(1, 20), np.array([[1.0, 0.0]]))), False)):
        B = ed.basis_build(20, 10, z, *grp)  # 2518, 9252, 92378 states
        x = to_torch(ei.x_by_index(3, ed.basis_size(B), 1)[:, 0], np.float64)
        y, want = torch.empty_like(x), torch.empty_like(x)
        assert served(ed, lambda: ed.matvec(O, B, x, y)) == {"slot without copy" if one else "slot": 1}
        ed.kernel_policy("slots")
        assert served(ed, lambda: ed.matvec(O, B, x, want)) == {"slot": 1}
        ed.kernel_policy("auto")
        assert torch.equal(y, want)
