"""The work this library is used for, as cases that can be timed and checked.

Six kinds of work, each through the public calls of ``paper_2308_16712_gb300.ed``:

* ``matvec``  -- y = H x in one symmetry sector (``ed.matvec``): the call every
  Krylov method, time evolution or correlation function repeats;
* ``multi``   -- y_s = H x_s in every momentum sector of a ring at once
  (``ed.matvec_multi``);
* ``build``   -- the basis of a sector and the lookup of given states in it
  (``ed.basis_build``, ``ed.basis_states``, ``ed.basis_index``): what a program
  does first, and again for each sector it looks at;
* ``lanczos`` -- the ground state of one sector (``ed.lanczos``);
* ``block``   -- block Lanczos on several vectors (``ed.lanczos_block``);
* ``spectrum`` -- the lowest energy of all sectors of a ring
  (``ed.lanczos_multi``).

The lattices are spin-1/2 rings of 16 to 38 sites and tori up to 6x6, with
translations, reflection and spin inversion; vectors in fp64, fp32, complex128
and complex64, 1 to 16 of them interleaved.  ``exact`` evaluates the same
quantities in 64 bits with plain torch, from the definition of the symmetrised
Hamiltonian (brute force over the group).
"""
from __future__ import annotations

import math

import numpy as np
import torch

import ed_inputs as ei
from paper_2308_16712_gb300 import ed

DTYPES = {"f64": torch.float64, "f32": torch.float32, "c128": torch.complex128, "c64": torch.complex64}
ESIZE = {"f64": 8, "f32": 4, "c128": 16, "c64": 8}
LOOKUPS = 4096  # states a "build" program locates in its new basis


# ----------------------------------------------------------------------------
# cases
# ----------------------------------------------------------------------------
def _ring(kind, name, n, n_up, k, parity, z, model="heisenberg", **more):
    """parity 0: translations only; z 0: no spin inversion."""
    return dict(kind=kind, name=name, lattice="ring", n=n, n_up=n_up, k=k, parity=parity, z=z, model=model, **more)


def _torus(kind, name, lx, ly, kx, ky, z, **more):
    return dict(kind=kind, name=name, lattice="torus", n=lx * ly, n_up=lx * ly // 2, lx=lx, ly=ly, kx=kx, ky=ky,
                z=z, model="j1j2", **more)


def listed():
    return [
        # the smallest call there is in earnest: the 16-site ring's ground-state
        # sector (257 states), one fp64 product -- call and launch latency
        _ring("matvec", "matvec_ring16_f64", 16, 8, 0, 1, 1, dtype="f64", nvec=1),
        # the ordinary product: the 32-site ring's ground-state sector (4.7e6
        # states), one vector in single precision
        _ring("matvec", "matvec_ring32_f32", 32, 16, 0, 1, 1, dtype="f32", nvec=1),
        # an odd ring away from half filling, complex momentum, no spin
        # inversion, three vectors: ragged in every respect, 64-bit words
        _ring("matvec", "matvec_ring33_c128x3", 33, 15, 4, 0, 0, model="xxz", dtype="c128", nvec=3),
        # plain fp64 product of a sector far larger than the caches (6.3e7)
        _ring("matvec", "matvec_ring36_f64", 36, 18, 0, 1, 1, dtype="f64", nvec=1),
        # the block product of large-scale block Lanczos: eight interleaved
        # fp32 vectors over 2.3e8 states
        _ring("matvec", "matvec_ring38_f32x8", 38, 19, 0, 1, 1, dtype="f32", nvec=8),
        # two dimensions: the 6x6 J1-J2 torus at momentum (pi/3, 0), 1.3e8 states
        _torus("matvec", "matvec_torus6x6_c128", 6, 6, 1, 0, 1, dtype="c128", nvec=1),
        # all 140 sectors (Sz 0..3, every momentum) of the 28-site XXZ ring in
        # one call, eight vectors each
        dict(kind="multi", name="multi_xxz28_c64x8", n=28, dtype="c64", nvec=8),
        # building a sector and locating product states in it
        _ring("build", "build_ring36", 36, 18, 0, 1, 1),
        # ground state of the 32-site ring, fp64, with its vector
        _ring("lanczos", "lanczos_ring32_f64", 32, 16, 0, 1, 1, mode="f64", steps=100),
        # ground state of a small sector in the mixed-precision mode: many
        # short launches
        _ring("lanczos", "lanczos_ring20_f32", 20, 10, 0, 1, 1, mode="f32", steps=50),
        # block Lanczos, the mixed-precision solver for large ground states
        _ring("block", "block_ring32_f32x8", 32, 16, 0, 1, 1, mode="f32", nvec=8, steps=24),
        # a low-energy map: the lowest level of all 100 sectors of a 20-site ring
        dict(kind="spectrum", name="spectrum_xxz20", n=20, mode="f64", steps=60),
    ]


def draw(rng):
    while True:
        case = _draw(rng)
        if case is not None:
            return case


def _draw(rng):
    kind = rng.choices(["matvec", "multi", "build", "lanczos", "block", "spectrum"], [10, 2, 3, 2, 2, 1])[0]
    if kind == "multi":
        dt = rng.choice(["c64", "c128"])
        return dict(kind=kind, n=rng.randint(16, 28), dtype=dt, nvec=rng.choice([1, 2, 4, 8] if dt == "c64" else [1, 2]))
    if kind == "spectrum":
        return dict(kind=kind, n=rng.randint(12, 20), mode="f64", steps=rng.randint(40, 60))
    if rng.random() < 0.25:
        lx, ly = rng.choice([(4, 4), (4, 5), (5, 4), (4, 6), (6, 4), (5, 5), (5, 6), (6, 5), (6, 6)])
        case = _torus(kind, "", lx, ly, rng.randrange(lx), rng.randrange(ly), rng.choice([1, -1]))
        if lx * ly % 2:
            case["z"] = 0
    else:
        n = rng.randint(16, {"matvec": 38, "build": 36}.get(kind, 32))
        half = n % 2 == 0 and rng.random() < 0.8
        k = 0 if rng.random() < 0.5 else rng.randrange(n)
        case = _ring(kind, "", n, n // 2 if half else rng.randint(n // 4, n // 2), k,
                     rng.choice([1, -1]) if 2 * k % n == 0 and rng.random() < 0.7 else 0,
                     rng.choice([1, 1, -1]) if half and rng.random() < 0.8 else 0,
                     rng.choice(["heisenberg", "xxz"]))
        if 2 * case["n_up"] != n:
            case["z"] = 0
    del case["name"]
    dim = _dim(case)
    if dim < 200:
        return None
    if kind == "matvec":
        case["dtype"] = rng.choice(["f64", "f32", "c128", "c64"] if _real(case) else ["c128", "c64"])
        case["nvec"] = rng.choice([1, 1, 2, 3, 4, 5, 8, 8, 12, 16])
        if dim * (40 + 2 * ESIZE[case["dtype"]] * case["nvec"]) > 2.4e10 or _terms(case) * (1 + case["nvec"] / 8) > 9e9:
            return None
    elif kind == "build":
        if math.comb(case["n"], case["n_up"]) > 9.1e9 or dim > 1.3e8:
            return None
    elif kind == "lanczos":
        case["mode"] = rng.choice(["f64", "f32"])
        case["steps"] = rng.randint(30, 100 if dim > 20000 else 50)
        if _terms(case) * case["steps"] > 1.2e10 or dim < 1000:
            return None
    elif kind == "block":
        if not _real(case):
            return None
        case["mode"] = rng.choice(["f64", "f32"])
        case["nvec"] = rng.choice([2, 4, 8, 16])
        case["steps"] = rng.randint(12, 24)
        if _terms(case) * case["steps"] * (1 + case["nvec"] / 8) > 8e9 or dim < 50 * case["nvec"] * case["steps"]:
            return None
    return case


# ----------------------------------------------------------------------------
# sizes
# ----------------------------------------------------------------------------
def _group(case):
    if case["lattice"] == "torus":
        return ei.torus_group(case["lx"], case["ly"], case["kx"], case["ky"])
    return ei.ring_group(case["n"], case["k"], case["parity"] or None)


def _hamiltonian(case):
    if case["model"] == "j1j2":
        return ei.j1j2_torus(case["lx"], case["ly"], 1.0, 0.5)
    if case["model"] == "xxz":
        return ei.xxz_ring(case["n"], 1.0, 1.5)
    return ei.heisenberg_ring(case["n"])


def _real(case):
    return bool(np.all(np.abs(_group(case)[1][:, 1]) < 1e-9))


def _dim(case):
    """Sector dimension: the average over the group of conj(chi) times the
    number of states the element fixes."""
    perms, chars = _group(case)
    n, n_up, total = case["n"], case["n_up"], 0.0
    for p, c in zip(perms, chars):
        seen, cycles = [False] * n, []
        for i in range(n):
            length = 0
            while not seen[i]:
                seen[i] = True
                i = int(p[i])
                length += 1
            if length:
                cycles.append(length)
        ways = [1] + [0] * n_up
        for length in cycles:
            for m in range(n_up, length - 1, -1):
                ways[m] += ways[m - length]
        total += c[0] * ways[n_up]
        if case["z"] and all(length % 2 == 0 for length in cycles):
            total += c[0] * case["z"] * 2 ** len(cycles)
    return round(total / (len(perms) * (2 if case["z"] else 1)))


def _terms(case):
    """Off-diagonal matrix elements of one product (antiparallel bonds)."""
    n, m = case["n"], case["n_up"]
    bonds = 4 * n if case["lattice"] == "torus" else n
    return _dim(case) * bonds * 2.0 * m * (n - m) / (n * (n - 1))


def _sectors(n, sz_max=3):
    """(n_up, k, z) of every sector of an n-site ring with Sz in 0..3 (1/2..7/2
    for odd n) and every momentum; spin inversion +-1 where it applies."""
    out = []
    for m in range((n + 1) // 2, min(n - 1, (n + 1) // 2 + sz_max) + 1):
        for k in range(n):
            out += [(m, k, z) for z in ((1, -1) if 2 * m == n else (0,))]
    return out


def _sector_case(n, m, k, z):
    return _ring("matvec", "", n, m, k, 0, z, "xxz")


def work(case):
    """Bytes: each row's state (8) and norm (2) and each vector element read or
    written once; a solver's step also reads and writes its Lanczos vectors.
    Operations: a multiplication and an addition per matrix element and vector."""
    if case["kind"] in ("multi", "spectrum"):
        secs = [_sector_case(case["n"], *s) for s in _sectors(case["n"])]
        dim = sum(_dim(c) for c in secs)
        nnz = dim + sum(_terms(c) for c in secs)
    else:
        dim = _dim(case)
        nnz = dim + _terms(case)
    if case["kind"] in ("matvec", "multi"):
        e, v = ESIZE[case["dtype"]], case["nvec"]
        return {"bytes": dim * (10.0 + 2 * e * v), "flops": nnz * v * (8.0 if case["dtype"][0] == "c" else 2.0)}
    if case["kind"] == "build":
        return {"bytes": dim * 10.0 + LOOKUPS * 16.0, "flops": 0.0}
    v = case.get("nvec", 1)
    cplx = case["kind"] == "spectrum" or not _real(case)
    e = 16.0 if cplx else 8.0
    return {"bytes": case["steps"] * dim * (10.0 + 5 * e * v), "flops": case["steps"] * nnz * v * (8.0 if cplx else 2.0)}


# ----------------------------------------------------------------------------
# what a program has in hand, and one pass
# ----------------------------------------------------------------------------
def _uniform(shape, dtype, seed):
    """Real and imaginary parts uniform in [-1, 1)."""
    g = torch.Generator(device="cuda").manual_seed(seed)
    out = torch.empty(shape, dtype=dtype, device="cuda")
    flat = torch.view_as_real(out) if dtype.is_complex else out
    flat.uniform_(-1.0, 1.0, generator=g)
    return out


def prepare(case, seed):
    kind = case["kind"]
    if kind in ("multi", "spectrum"):
        h = ei.xxz_ring(case["n"], 1.0, 1.5)
        op = ed.operator_create(case["n"], h["sites"], h["coeff"], h["local"])
        dtype = DTYPES[case.get("dtype", "c128")]
        v = case.get("nvec", 1)
        bases, offsets, rows = [], [], 0
        for m, k, z in _sectors(case["n"]):
            perms, chars = ei.ring_group(case["n"], k)
            bases.append(ed.basis_build(case["n"], m, z, perms, chars))
            offsets.append(rows)
            rows += (ed.basis_size(bases[-1]) + 3) // 4 * 4  # every sector's vectors start 16-byte aligned
        x = _uniform((rows, v), dtype, seed)
        dims = [ed.basis_size(b) for b in bases]
        if kind == "spectrum":
            items = [(b, x[o:o + d, 0], None) for b, o, d in zip(bases, offsets, dims)]
            return dict(case=case, op=op, x=x, items=items)
        y = torch.zeros_like(x)
        items = [(b, x[o:o + d], y[o:o + d]) for b, o, d in zip(bases, offsets, dims) if d]
        return dict(case=case, op=op, x=x, y=y, items=items)
    perms, chars = _group(case)
    if kind == "build":
        states = _random_states(case, seed)
        return dict(case=case, perms=perms, chars=chars, states=_lattice(case).least(states))
    h = _hamiltonian(case)
    op = ed.operator_create(case["n"], h["sites"], h["coeff"], h["local"])
    basis = ed.basis_build(case["n"], case["n_up"], case["z"], perms, chars)
    dim = ed.basis_size(basis)
    if kind == "matvec":
        shape = (dim,) if case["nvec"] == 1 else (dim, case["nvec"])
        x = _uniform(shape, DTYPES[case["dtype"]], seed)
        return dict(case=case, op=op, basis=basis, x=x, y=torch.empty_like(x))
    if kind == "block":
        return dict(case=case, op=op, basis=basis, x=_uniform((dim, case["nvec"]), torch.float64, seed))
    return dict(case=case, op=op, basis=basis, x=_uniform((dim,), torch.float64 if _real(case) else torch.complex128, seed))


def run(state):
    case = state["case"]
    kind = case["kind"]
    if kind == "matvec":
        return ed.matvec(state["op"], state["basis"], state["x"], state["y"], case["nvec"])
    if kind == "multi":
        ed.matvec_multi(state["op"], state["items"], case["nvec"])
        return state["y"]
    if kind == "build":
        basis = ed.basis_build(case["n"], case["n_up"], case["z"], state["perms"], state["chars"])
        states, norms = ed.basis_states(basis)
        return [states, norms, ed.basis_index(basis, state["states"])]
    if kind == "spectrum":
        return np.array([r.e0 for r in ed.lanczos_multi(state["op"], state["items"], case["steps"], ed.ED_LANCZOS_F64)])
    mode = ed.ED_LANCZOS_F64 if case["mode"] == "f64" else ed.ED_LANCZOS_F32_MATVEC
    x = state["x"]
    vec = torch.empty(x.shape[:1], dtype=x.dtype, device=x.device)
    if kind == "block":
        _, r = ed.lanczos_block(state["op"], state["basis"], x, case["nvec"], case["steps"], mode, vec_out=vec)
    else:
        r = ed.lanczos(state["op"], state["basis"], x, case["steps"], mode, vec)
    if case["mode"] == "f32":  # a vector from fp32 products is kept in single precision
        vec = vec.to(torch.complex64 if vec.is_complex() else torch.float32)
    return [r.e0, vec]


# ----------------------------------------------------------------------------
# the same in 64 bits, from the definition
# ----------------------------------------------------------------------------
class _Lattice:
    """Brute force over the group on int64 tensors of states: element (e, f) is
    the e-th lattice element in ``_group``'s order, followed by spin inversion
    if f."""

    def __init__(self, perms, n, flip, rotation):
        self.n, self.flip, self.full = n, flip, (1 << n) - 1
        # every element as a rotation of the n-bit word (by `rotation` sites a
        # step) after one of a few permutations
        self.elems = []
        index = {tuple(int(v) for v in p): e for e, p in enumerate(perms)}
        left = set(index)
        for p in list(index):
            if p in left:
                turns = []
                for r in range(0, n, rotation):
                    q = tuple((v + r) % n for v in p)
                    left.discard(q)
                    turns.append((r, index[q]))
                self.elems.append((p, turns))
        self.count = len(perms)

    def images(self, s):
        for perm, turns in self.elems:
            if all(v == i for i, v in enumerate(perm)):
                h = s
            else:
                h = torch.zeros_like(s)
                for i, v in enumerate(perm):
                    h |= ((s >> i) & 1) << v
            for r, e in turns:
                q = ((h << r) | (h >> (self.n - r))) & self.full if r else h
                yield q, e
                if self.flip:
                    yield q ^ self.full, e + self.count

    def least(self, s):
        best = s.clone()
        for q, _ in self.images(s):
            torch.minimum(best, q, out=best)
        return best

    def least_by(self, s):
        best, by = torch.full_like(s, 1 << 62), torch.zeros_like(s, dtype=torch.int16)
        for q, e in self.images(s):
            low = q < best
            best = torch.where(low, q, best)
            by[low] = e
        return best, by.to(torch.int64)

    def representatives(self, n_up):
        """Every state that is the least of its orbit, ascending."""
        n, lo = self.n, self.n // 2
        low = torch.arange(1 << lo, device="cuda")
        pop = sum((low >> i) & 1 for i in range(lo))
        by_pop = [low[pop == p] for p in range(lo + 1)]
        found = []
        high = torch.arange(1 << (n - lo), device="cuda")
        pop = sum((high >> i) & 1 for i in range(n - lo))
        for p in range(max(0, n_up - lo), min(n - lo, n_up) + 1):
            lows = by_pop[n_up - p]
            highs = high[pop == p] << lo
            step = max(1, (1 << 26) // max(1, lows.numel()))
            for h in highs.split(step):
                found.append(self._keep((h[:, None] | lows[None, :]).reshape(-1)))
        return torch.sort(torch.cat(found))[0]

    def _keep(self, s):
        for perm, turns in self.elems:
            for r, _ in turns:
                h = s
                if not all(v == i for i, v in enumerate(perm)):
                    h = torch.zeros_like(s)
                    for i, v in enumerate(perm):
                        h |= ((s >> i) & 1) << v
                q = ((h << r) | (h >> (self.n - r))) & self.full if r else h
                keep = q >= s
                if self.flip:
                    keep &= (q ^ self.full) >= s
                s = s[keep]
        return s


def _lattice(case):
    perms, _ = _group(case)
    return _Lattice(perms, case["n"], bool(case["z"]), case.get("lx", 1))


def _random_states(case, seed):
    g = torch.Generator(device="cuda").manual_seed(seed)
    order = torch.rand((LOOKUPS, case["n"]), device="cuda", generator=g).argsort(dim=1)
    bits = (order < case["n_up"]).to(torch.int64) << torch.arange(case["n"], device="cuda")
    return bits.sum(dim=1)


def _characters(case):
    c = _group(case)[1]
    c = torch.complex(torch.from_numpy(c[:, 0].copy()), torch.from_numpy(c[:, 1].copy())).cuda()
    return torch.cat([c, c * case["z"]]) if case["z"] else c


class _Sector:
    """Basis and Hamiltonian of one sector; ``reps`` as _Lattice gives them."""

    def __init__(self, case, lattice, reps):
        chi = _characters(case)
        norm = torch.zeros(reps.numel(), dtype=torch.float64, device="cuda")
        for q, e in lattice.images(reps):
            norm += torch.where(q == reps, chi[e].real, 0.0)  # the sum over the stabiliser is real
        self.keep = norm > 0.5
        self.states, self.norms = reps[self.keep], norm[self.keep].round()
        self.lattice, self.chi, self.h = lattice, chi, _hamiltonian(case)

    def bonds(self):
        for (i, j), c, m in zip(self.h["sites"].tolist(), self.h["coeff"][:, 0].tolist(), self.h["local"][:, :, 0]):
            yield i, j, c * m.reshape(4, 4)

    def diagonal(self):
        d = torch.zeros(self.states.numel(), dtype=torch.float64, device="cuda")
        for i, j, m in self.bonds():
            same = ((self.states >> i) & 1) == ((self.states >> j) & 1)
            d += torch.where(same, float(m[0, 0]), float(m[1, 1]))
        return d

    def exchanges(self):
        """(rows, columns, values) of each bond's off-diagonal elements."""
        for i, j, m in self.bonds():
            rows = torch.nonzero(((self.states >> i) & 1) != ((self.states >> j) & 1)).reshape(-1)
            other = self.states[rows] ^ ((1 << i) | (1 << j))
            best, by = self.lattice.least_by(other)
            at = torch.searchsorted(self.states, best).clamp_(max=self.states.numel() - 1)
            held = self.states[at] == best
            rows, at, by = rows[held], at[held], by[held]
            yield rows, at, float(m[1, 2]) * self.chi[by] * torch.sqrt(self.norms[at] / self.norms[rows])

    def product(self, x):
        """y = H x for x of shape (dim, nvec), complex128."""
        y = self.diagonal()[:, None] * x
        for rows, at, val in self.exchanges():
            y.index_add_(0, rows, val[:, None] * x[at])
        return y

    def matrix(self, real):
        n = self.states.numel()
        d = torch.arange(n, device="cuda")
        rows, cols, vals = [d], [d], [self.diagonal().to(torch.complex128)]
        for r, c, v in self.exchanges():
            rows.append(r)
            cols.append(c)
            vals.append(v)
        v = torch.cat(vals)
        rows, cols = torch.cat(rows), torch.cat(cols)
        order = torch.argsort(rows, stable=True)
        crow = torch.zeros(n + 1, dtype=torch.int64, device="cuda")
        crow[1:] = torch.bincount(rows, minlength=n).cumsum(0)
        v = v[order]
        return torch.sparse_csr_tensor(crow, cols[order], v.real.contiguous() if real else v, (n, n))


def _krylov(matrix, x, steps):
    """Lowest Ritz value and vector of `steps` Lanczos steps from x, each new
    vector orthogonalised against all earlier ones."""
    v = x / torch.linalg.vector_norm(x)
    vs, a, b = torch.empty((steps, x.numel()), dtype=x.dtype, device="cuda"), [], []
    for j in range(steps):
        vs[j] = v
        w = matrix @ v
        a.append(torch.vdot(v, w).real)
        done = vs[:j + 1]
        for _ in range(2):
            w = w - done.T @ (done.conj() @ w)
        b.append(torch.linalg.vector_norm(w))
        if float(b[-1]) < 1e-10:
            break
        v = w / b[-1]
    a, b = torch.stack(a).cpu(), torch.stack(b).cpu()
    t = torch.diag(a) + torch.diag(b[:len(a) - 1], 1) + torch.diag(b[:len(a) - 1], -1)
    e, y = torch.linalg.eigh(t)
    y = y[:, 0] * (1.0 if y[:, 0].sum() >= 0 else -1.0)
    return float(e[0]), (y.to(x.device).to(x.dtype)) @ vs[:len(a)]


def exact(case, seed):
    kind = case["kind"]
    if kind == "build" or case["n"] > 33:
        return None  # whole numbers; or an enumeration of many seconds
    if kind in ("multi", "spectrum"):
        st = prepare(case, seed)
        out = torch.zeros(st["x"].shape, dtype=torch.complex128, device="cuda")
        energies, start, tables = [], 0, {}
        for m, k, z in _sectors(case["n"]):
            sector = _sector_case(case["n"], m, k, z)
            if (m, bool(z)) not in tables:
                lattice = _lattice(sector)
                tables[m, bool(z)] = lattice, lattice.representatives(m)
            s = _Sector(sector, *tables[m, bool(z)])
            d = s.states.numel()
            x = st["x"][start:start + d].to(torch.complex128)
            if kind == "spectrum":
                energies.append(_krylov(s.matrix(False), x[:, 0], case["steps"])[0])
            else:
                out[start:start + d] = s.product(x)
            start += (d + 3) // 4 * 4
        return np.array(energies) if kind == "spectrum" else out
    st = prepare(case, seed)
    lattice = _lattice(case)
    s = _Sector(case, lattice, lattice.representatives(case["n_up"]))
    real = _real(case)
    if kind == "matvec":
        y = s.product(st["x"].reshape(s.states.numel(), -1).to(torch.complex128)).reshape(st["x"].shape)
        return y if st["x"].is_complex() else y.real.contiguous()
    if s.states.numel() > 6_000_000:
        return None
    if kind == "block" or case["mode"] == "f32":
        # the energy is refined in fp64, towards the sector's lowest level; the
        # vector's sign depends on the recurrence
        steps = min(s.states.numel(), 160 if s.states.numel() > 1_000_000 else 300)
        return [_krylov(s.matrix(real), st["x"].reshape(s.states.numel(), -1)[:, 0].contiguous(), steps)[0], None]
    e0, vec = _krylov(s.matrix(real), st["x"], case["steps"])
    return [e0, vec / torch.linalg.vector_norm(vec)]
