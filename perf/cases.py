"""Performance cases of the symmetry-adapted exact-diagonalization library.

Every case is one call, or one short run, that a program makes through the public entry
points: the product y = H x on device or host vectors, a Lanczos run, the energy with its
gradient, the per-class expectations, the batched product over many sectors, and the
build of a sector.  A case is a dict of plain values:

* ``op``: what runs (see the functions ``_run_*``);
* the sector: ``lattice`` ("chain", "torus" or "tilted40"), ``L`` (chain length or torus
  edge), ``sub`` (sublattices), ``up`` (up spins), ``m1``/``m2`` (momentum), ``ir`` (point
  irrep), ``J2``, ``flip`` (-1: no spin flip, else its parity);
* ``dtype`` ("f64", "f32", "c128", "c64") and the options of the op.

``exact`` restates each result in 64-bit torch: all configurations of the sector's S^z are
enumerated, every group element is applied to every one of them, and the terms of H are
summed bond by bond in fp64.
"""
from __future__ import annotations

import functools
import math

import numpy as np
import torch

import paper_1804_05028_gb300 as ed
import workloads as w
from paper_1804_05028_gb300.autograd import ground_state_energy

_DT = {"f64": torch.float64, "f32": torch.float32, "c128": torch.complex128, "c64": torch.complex64}
_BYTES = {"f64": 8, "f32": 4, "c128": 16, "c64": 8}


def _case(name, op, lattice, L, sub, up, m1=0, m2=0, ir=0, J2=0.0, flip=-1, **kw):
    c = dict(op=op, lattice=lattice, L=L, sub=sub, up=up, m1=m1, m2=m2, ir=ir, J2=J2, flip=flip, **kw)
    if name:
        c["name"] = name
    return c


def listed():
    return [
        # the smallest call: one product on the 16-site chain (D = 810), as a user's own
        # iterative solver makes it thousands of times; launch and call latency
        _case("apply_chain16_f64", "apply", "chain", 16, 2, 8, dtype="f64"),
        # an ordinary sector with complex characters: a momentum away from the symmetric
        # points (36 translations only), below half filling, 2.6e6 states
        _case("apply_sq36_k12_c128", "apply", "torus", 6, 4, 9, m1=1, m2=2, J2=0.5, dtype="c128"),
        # the 6x6 J1-J2 ground-state sector (3.2e7 states), fp32 vectors and fp64 vectors
        _case("apply_sq36_f32", "apply", "torus", 6, 4, 18, J2=0.5, dtype="f32"),
        _case("apply_sq36_f64", "apply", "torus", 6, 4, 18, J2=0.5, dtype="f64"),
        # the largest sector: 40 sites, 8.6e8 states
        _case("apply_tilted40_f32", "apply", "tilted40", 40, 4, 20, dtype="f32"),
        # one rank's share of a row-sharded product (a quarter of the rows, ragged ends)
        _case("rows_sq36_flip_f32", "rows", "torus", 6, 4, 18, J2=0.5, flip=0, dtype="f32", part=1, parts=4),
        # host vectors in and out (pinned): the call a CPU program makes
        _case("host_sq36_f32", "host", "torus", 6, 4, 18, J2=0.5, dtype="f32"),
        # mixed-precision Lanczos with its ground state on the 6x6 sector, a few steps
        _case("lanczos_sq36_mixed", "lanczos", "torus", 6, 4, 18, J2=0.5, dtype="f32", steps=4, reorth="local"),
        # a whole small diagonalization: 24-site chain, 40 steps, every vector kept and
        # reorthogonalised, ground state; many short launches
        _case("lanczos_chain24_full", "lanczos", "chain", 24, 4, 12, dtype="f64", steps=40, reorth="full"),
        # energy and gradient dE0/dJ by autograd, forward and backward (converged runs)
        _case("grad_sq36_up7", "grad", "torus", 6, 4, 7, J2=0.5, dtype="f64"),
        # all momenta and point irreps of the 5x5 torus at S^z = 1/2 .. 7/2 in one launch
        _case("batch_sq25_k4", "batch", "torus", 5, 1, 13, J2=0.3, dtype="f32", up_to=16, k=4),
        # building a sector (tables, basis, index) and taking its states to the host
        _case("build_sq36_up12", "build", "torus", 6, 4, 12, J2=0.5, dtype="f64"),
    ]


def draw(rng):
    """One more case of the same ranges; about the cost of the 6x6 sector at most."""
    op = rng.choice(["apply", "apply", "apply", "apply", "rows", "host", "expect", "lanczos", "lanczos", "grad",
                     "batch", "batch", "build"])
    if op == "batch":
        lo = rng.randint(13, 22)
        return _case(None, op, "torus", 5, 1, lo, J2=0.3, dtype="f32", up_to=min(25, lo + rng.randint(0, 2)),
                     k=rng.choice([1, 2, 4, 8]))
    small = op in ("grad", "lanczos")
    lattice = rng.choice(["chain", "torus", "torus", "tilted40"])
    m1 = m2 = ir = 0
    J2, flip = 0.0, -1
    if lattice == "chain":
        L, sub = rng.choice([(16, 2), (18, 2), (20, 2), (20, 4), (22, 2), (24, 4), (24, 3), (28, 4), (30, 3),
                             (20, 5), (20, 1), (32, 4)] if not small else [(12, 2), (16, 4), (18, 3), (20, 2), (20, 4), (24, 4)])
        up = rng.randint(L // 4, L // 2)
        m1 = rng.choice([0, 0, L // 2, rng.randint(0, L - 1)])
    elif lattice == "torus":
        L = rng.choice([4, 6, 6, 6])
        sub = 4 if L == 6 else rng.choice([4, 2, 1])
        up = rng.randint(4, 8) if L == 4 else rng.randint(5, 9) if small else rng.choice([6, 9, 11, 13, 15, 18])
        J2 = 0.5
        lim = L - 1
        m1, m2 = rng.choice([(0, 0), (0, 0), (L // 2, L // 2), (L // 2, 0), (1, 2), (rng.randint(0, lim), rng.randint(0, lim))])
    else:
        L, sub, up = 40, 4, rng.randint(4, 7) if small else rng.randint(5, 11)
    if lattice != "chain":
        c = _case(None, op, lattice, L, sub, up, m1, m2, 0, J2)
        ir = rng.randrange(_n_irreps(c))
    c = _case(None, op, lattice, L, sub, up, m1, m2, ir, J2)
    if 2 * up == _sites(c) and rng.random() < 0.4:
        c["flip"] = flip = rng.randint(0, 1)
    while _dim(c) > 4e7:                       # momenta with few point operations: lower filling
        c["up"] -= 1
        c["flip"] = -1
    real = _problem(*_sector(c)).is_real()
    c["dtype"] = rng.choice(["f64", "f32"] if real else ["c128", "c64"])
    if op == "rows":
        c["parts"] = rng.choice([2, 3, 4, 8])
        c["part"] = rng.randrange(c["parts"])
    if op == "lanczos":
        c["steps"] = rng.randint(4, 16)   # later steps of a small sector amplify rounding
        c["reorth"] = rng.choice(["local", "local", "full", "none"])
    if op == "grad":
        c["dtype"] = "f64"
    return c


# ---------------------------------------------------------------------------- sectors
def _sector(c):
    return (c["lattice"], c["L"], c["sub"], c["up"], c["m1"], c["m2"], c["ir"], c["J2"], c["flip"])


@functools.lru_cache(maxsize=64)
def _problem(lattice, L, sub, up, m1, m2, ir, J2, flip):
    if lattice == "chain":
        p = w.chain(L, sub, k=m1, n_up=up)
    elif lattice == "torus":
        p = w.square_torus(L, momentum=(m1, m2), point_irrep=ir, n_sublat=sub, J1=1.0, J2=J2, n_up=up)
    else:
        p = w.tilted_square_40(momentum=(m1, m2), point_irrep=ir, n_sublat=sub, J1=1.0, J2=J2, n_up=up)
    return w.with_spin_flip(p, flip) if flip >= 0 else p


@functools.lru_cache(maxsize=64)
def _irreps_of(lattice, L, m1, m2):
    a = ((6, 2), (-2, 6)) if lattice == "tilted40" else ((L, 0), (0, L))
    return w.n_point_irreps(*a, (m1, m2))


def _n_irreps(c):
    return _irreps_of(c["lattice"], c["L"], c["m1"], c["m2"])


@functools.lru_cache(maxsize=4)
def _sq25(up, up_to):
    return w.config_square25_sectors(J2=0.3, n_up_values=range(up, up_to + 1))


def _sites(c):
    return {"chain": c["L"], "torus": c["L"] ** 2, "tilted40": 40}[c["lattice"]]


def _dim(c):
    """The sector's dimension, as the number of configurations over the group's order."""
    return max(1.0, math.comb(_sites(c), c["up"]) / _problem(*_sector(c)).n_sym)


def _rows(c, D):
    n, r = c["parts"], c["part"]
    return D * r // n, D * (r + 1) // n


def _vector(n, dtype, seed, device="cuda"):
    """Uniform components in [-1, 1), as a Lanczos start vector has them."""
    g = torch.Generator(device=device).manual_seed(int(seed))
    dt = _DT[dtype]
    real = {torch.complex128: torch.float64, torch.complex64: torch.float32}.get(dt)
    if real is None:
        return torch.rand(n, dtype=dt, device=device, generator=g).mul_(2).sub_(1)
    x = torch.rand(2 * n, dtype=real, device=device, generator=g).mul_(2).sub_(1)
    return torch.view_as_complex(x.view(n, 2))


# ---------------------------------------------------------------------------- prepare
def _relabel(p, seed):
    """The sector with its sites renumbered inside each sublattice, as another user's
    lattice file would number them (the representatives are other integers, the dimension
    is the same)."""
    import dataclasses
    rng = np.random.RandomState(seed % (1 << 31))
    n = p.n_sites // p.n_sublat
    new = np.concatenate([X * n + rng.permutation(n) for X in range(p.n_sublat)]).astype(np.int32)
    perm = np.empty_like(p.perm)
    perm[:, new] = new[p.perm]
    return dataclasses.replace(p, bonds=new[p.bonds].astype(np.int32), perm=perm, coords=None)


def prepare(case, seed):
    op = case["op"]
    if op == "batch":
        bases = ed.build_sectors(_sq25(case["up"], case["up_to"]))
        k = case["k"]
        # one buffer per kind, each sector's block 32-byte aligned
        bufs, xs, ys = _batch_buffers(bases, [b.dim for b in bases], [b.is_real for b in bases], k, seed)
        bt = ed.Batch(bases, k=k)
        bt.set_vectors(xs, ys)
        return {"op": op, "bt": bt, "out": [b[1] for b in bufs], "keep": (bases, bufs)}
    p = _problem(*_sector(case))
    if op == "build":
        return {"op": op, "p": _relabel(p, seed)}
    B = ed.build_basis_from(p)
    st = {"op": op, "B": B, "case": case}
    D = B.dim
    if op == "grad":
        rng = np.random.RandomState(seed % (1 << 31))
        J = [1.0 + 0.05 * float(u) for u in rng.uniform(-1, 1, 1)]
        J += [case["J2"] + 0.05 * float(u) for u in rng.uniform(-1, 1, p.n_classes - 1)]
        st["J"] = torch.tensor(J, dtype=torch.float64, requires_grad=True)
        return st
    st["x"] = _vector(D, case["dtype"], seed)
    if op == "host":
        st["x"] = st["x"].cpu().pin_memory()
        st["y"] = torch.empty_like(st["x"]).pin_memory()
    elif op == "apply":
        st["y"] = torch.empty_like(st["x"])
    elif op == "rows":
        st["r"] = _rows(case, D)
        st["y"] = torch.empty(st["r"][1] - st["r"][0], dtype=st["x"].dtype, device="cuda")
    elif op == "lanczos":
        st["psi"] = torch.empty_like(st["x"])
        if case["reorth"] == "full":
            st["krylov"] = torch.empty((case["steps"] + 1) * D, dtype=st["x"].dtype, device="cuda")
        else:
            st["work"] = torch.empty(4 * D, dtype=st["x"].dtype, device="cuda")
    return st


def _batch_layout(dims, reals, k):
    """Offsets (in elements) of every sector's [dim][k] block in its kind's buffer."""
    off, n = [], {True: 0, False: 0}
    for D, r in zip(dims, reals):
        off.append(n[r])
        n[r] += (D * k + 7) // 8 * 8
    return off, n


def _batch_buffers(bases, dims, reals, k, seed):
    off, n = _batch_layout(dims, reals, k)
    g = torch.Generator(device="cuda").manual_seed(int(seed))
    bufs = []
    for real in (True, False):
        dt = torch.float32 if real else torch.complex64
        bufs.append((torch.randn(n[real], dtype=dt, device="cuda", generator=g),
                     torch.zeros(n[real], dtype=dt, device="cuda")))
    xs, ys = [], []
    for D, r, o in zip(dims, reals, off):
        X, Y = bufs[0 if r else 1]
        xs.append(X[o:o + D * k])
        ys.append(Y[o:o + D * k])
    return bufs, xs, ys


# ---------------------------------------------------------------------------- run
def run(state):
    op = state["op"]
    if op == "batch":
        state["bt"].apply()
        return state["out"]
    if op == "build":
        B = ed.build_basis_from(state["p"])
        s, t = B.export()
        B.close()
        return [s.view(np.int64), t.astype(np.int32)]
    B = state["B"]
    if op == "apply":
        return B.apply_H(state["x"], state["y"])
    if op == "rows":
        return B.apply_H_rows(state["x"], *state["r"], y=state["y"])
    if op == "host":
        return B.apply_H_host(state["x"], state["y"])
    if op == "expect":
        return B.expect_classes(state["x"])
    if op == "lanczos":
        c = state["case"]
        r = B.lanczos(dtype=state["x"].dtype, fixed_steps=c["steps"], v0=state["x"], psi=state["psi"],
                      reorth=c["reorth"], krylov=state.get("krylov"), work=state.get("work"))
        return {"E0": r["E0"], "alpha": r["alpha"], "beta": r["beta"], "psi": state["psi"]}
    J = state["J"]
    J.grad = None
    E = ground_state_energy(B, J)
    E.backward()
    return {"E": E.detach(), "grad": J.grad}


# ---------------------------------------------------------------------------- work
def _terms(p, D):
    """Exchange terms of one product: antiparallel bonds, by their mean over the sector."""
    N, u = p.n_sites, p.n_up
    return D * p.n_bonds * (2.0 * u * (N - u) / (N * (N - 1.0)) if N > 1 else 0.0)


def work(case):
    """Bytes: every row's state once, x read once and y written once per product (Lanczos:
    also one read of the previous vector, and the reorthogonalisation's reads).  Flops: a
    multiply and an add per exchange term and per diagonal entry."""
    op = case["op"]
    if op == "batch":
        b = f = 0.0
        for p in _sq25(case["up"], case["up_to"]):
            D = math.comb(25, p.n_up) / p.n_sym
            e = (4 if p.is_real() else 8) * case["k"]
            b += D * (8 + 2 * e)
            f += 2 * (D + _terms(p, D)) * case["k"] * (1 if p.is_real() else 4)
        return {"bytes": b, "flops": f}
    p = _problem(*_sector(case))
    D = _dim(case)
    e = _BYTES[case["dtype"]]
    cx = 4 if case["dtype"][0] == "c" else 1
    one_b, one_f = D * (8 + 2 * e), 2 * cx * (D + _terms(p, D))
    if op == "rows":
        n = 1.0 / case["parts"]
        return {"bytes": D * e + n * D * (8 + e), "flops": n * one_f}
    if op == "build":
        return {"bytes": D * 10, "flops": D * p.n_sym}
    if op == "lanczos":
        m = case["steps"]
        extra = m * (m + 1) // 2 * 2 if case["reorth"] == "full" else 2 * m
        n = m + 1 if case["reorth"] == "full" else 2 * m
        return {"bytes": n * one_b + extra * D * e, "flops": n * one_f + 2 * cx * extra * D}
    if op == "grad":
        return {"bytes": 150 * one_b, "flops": 150 * one_f}   # about 50 steps and 100 to the state
    return {"bytes": one_b, "flops": one_f}


def tolerance(case):
    """About four times what the path shows against ``exact``: rounding of sums of some
    hundred terms, and for Lanczos its growth over the steps."""
    op = case["op"]
    lo = case["dtype"] in ("f32", "c64")
    if op == "build":
        return "exact"
    if op == "batch":              # fp32 sums of up to 50 terms: 1.4e-7 seen
        return {"rel": 6e-7, "max": 1e-5}
    if op == "lanczos":            # fp32 vectors round once per step; fp64: 4e-15 seen
        return {"rel": 1e-6, "max": 4e-5} if lo else {"rel": 1e-11, "max": 1e-9}
    if op == "grad":               # the state is converged to a residual of 1e-10
        return {"rel": 1e-8, "max": 1e-7}
    if op == "expect":             # fp32 products of a row, summed over the rows in fp64
        return {"rel": 1e-6, "max": 1e-5} if lo else {"rel": 1e-11, "max": 1e-10}
    # one rounding to fp32 (2.6e-8 seen), or fp64 sums (6.5e-16 seen)
    return {"rel": 1e-7, "max": 2e-6} if lo else {"rel": 3e-15, "max": 1e-13}


# ---------------------------------------------------------------------------- exact
def _configs(N, k, device):
    """All N-bit integers with k ones, in increasing order (int64)."""
    row = [torch.zeros(1, dtype=torch.int64, device=device)] + [None] * k
    for n in range(1, N + 1):
        new = []
        for q in range(k + 1):
            parts = []
            if row[q] is not None:
                parts.append(row[q])
            if q and row[q - 1] is not None:
                parts.append(row[q - 1] | (1 << (n - 1)))
            # what cannot reach k ones any more is dropped
            new.append(torch.cat(parts) if parts and q + N - n >= k else None)
        row = new
    return row[k]


def _orbits(p, device):
    """Configurations, their representative, the numerator of the first minimiser's
    character, |Stab| and whether the projection survives, from every group element."""
    N = p.n_sites
    s = _configs(N, p.n_up, device)
    bits = 9
    nch = -(-N // bits)
    rep = s.clone()
    ph = torch.zeros(s.numel(), dtype=torch.int32, device=device)
    stab = torch.zeros(s.numel(), dtype=torch.int32, device=device)
    kept = torch.ones(s.numel(), dtype=torch.bool, device=device)
    best = torch.full_like(s, 1 << 62)
    chunk = [(s >> (bits * c)) & ((1 << bits) - 1) for c in range(nch)]
    for g in range(p.n_sym):
        img = np.zeros((nch, 1 << bits), np.int64)
        for b in range(N):      # bit b is label N-1-b
            to = N - 1 - int(p.perm[g, N - 1 - b])
            c, o = divmod(b, bits)
            img[c, (np.arange(1 << bits) >> o) & 1 == 1] |= 1 << to
        tab = torch.from_numpy(img).to(device)
        v = tab[0][chunk[0]]
        for c in range(1, nch):
            v |= tab[c][chunk[c]]
        if p.flip is not None and p.flip[g]:
            v ^= (1 << N) - 1
        num = int(p.phase_num[g]) % p.phase_denom
        lower = v < best
        best = torch.where(lower, v, best)
        ph[lower] = num
        same = v == s
        stab += same
        if num:
            kept &= ~same
    rep = best
    return s, rep, ph, stab, kept


_EXACT_LIMIT = 4e10     # configurations x group elements


class _Sector64:
    def __init__(self, p, device, orbits=None):
        self.p, self.device = p, device
        s, rep, ph, stab, kept = orbits or _orbits(p, device)
        sel = (rep == s) & kept
        self.basis = s[sel]
        self.t = stab[sel].to(torch.float64)
        self.D = int(self.basis.numel())
        self.s, self.rep, self.ph = s, rep, ph
        ang = 2 * math.pi * torch.arange(p.phase_denom, dtype=torch.float64, device=device) / p.phase_denom
        self.chi = torch.complex(torch.cos(ang), torch.sin(ang))

    def classes(self, x, rows=None):
        """(H_c x per class with unit exchange) for x of shape [D] or [D, k]."""
        p = self.p
        b = self.basis if rows is None else self.basis[rows[0]:rows[1]]
        t = self.t if rows is None else self.t[rows[0]:rows[1]]
        xi = x if rows is None else x[rows[0]:rows[1]]
        col = (lambda v: v) if x.dim() == 1 else (lambda v: v[:, None])
        out = [torch.zeros_like(xi) for _ in range(p.n_classes)]
        if self.D == 0:
            return out
        for (la, lb), c in zip(p.bonds, p.bond_class):
            pa, pb = p.n_sites - 1 - int(la), p.n_sites - 1 - int(lb)
            anti = (((b >> pa) ^ (b >> pb)) & 1) == 1
            out[c] += col(torch.where(anti, -0.25, 0.25).to(torch.float64) * p.Jz[c]) * xi
            r = torch.nonzero(anti).squeeze(1)
            q = torch.searchsorted(self.s, b[r] ^ ((1 << pa) | (1 << pb)))
            j = torch.searchsorted(self.basis, self.rep[q]).clamp_(max=self.D - 1)
            hit = self.basis[j] == self.rep[q]
            r, q, j = r[hit], q[hit], j[hit]
            wgt = 0.5 * torch.sqrt(self.t[j] / t[r])
            chi = self.chi[self.ph[q].long()]
            wgt = wgt * chi if x.is_complex() else wgt * chi.real
            out[c].index_add_(0, r, col(wgt) * x[j])
        return out

    def apply(self, x, J, rows=None):
        return sum(float(Jc) * h for Jc, h in zip(J, self.classes(x, rows)))

    def lanczos(self, x, J, steps, tol=0.0):
        """alpha, beta, E0 and the Ritz vector by fp64 Lanczos with every vector kept."""
        V, al, be = [x / torch.linalg.vector_norm(x)], [], []
        e = None
        for j in range(steps):
            y = self.apply(V[-1], J)
            al.append(float(torch.vdot(V[-1], y).real))
            for _ in range(2):
                K = torch.stack(V)
                y = y - K.T @ (K.conj() @ y)
            T = np.diag(al) + np.diag(be, 1) + np.diag(be, -1)
            ev, vec = np.linalg.eigh(T)
            b = float(torch.linalg.vector_norm(y))
            done = tol and b * abs(vec[-1, 0]) < tol
            e = ev[0]
            if done or j + 1 == steps or b < 1e-13:
                break
            be.append(b)
            V.append(y / b)
        z = vec[:, 0] * (1.0 if vec[:, 0].sum() >= 0 else -1.0)
        psi = sum(float(zk) * v for zk, v in zip(z, V))
        return np.array(al), np.array(be), float(e), psi / torch.linalg.vector_norm(psi)


def exact(case, seed):
    op = case["op"]
    if op == "build":
        return None
    dev = torch.device("cuda" if torch.cuda.is_available() else "cpu")
    if op == "batch":
        return _exact_batch(case, seed, dev)
    p = _problem(*_sector(case))
    if math.comb(p.n_sites, p.n_up) * float(p.n_sym) > _EXACT_LIMIT or math.comb(p.n_sites, p.n_up) > 2e8:
        return None
    S = _Sector64(p, dev)
    if op == "grad":
        rng = np.random.RandomState(seed % (1 << 31))
        J = [1.0 + 0.05 * float(u) for u in rng.uniform(-1, 1, 1)]
        J += [case["J2"] + 0.05 * float(u) for u in rng.uniform(-1, 1, p.n_classes - 1)]
        x = _vector(S.D, "f64" if p.is_real() else "c128", 7, dev)
        _, _, e, psi = S.lanczos(x, J, 400, tol=1e-11)
        g = [float(torch.vdot(psi, h).real) for h in S.classes(psi)]
        return {"E": torch.tensor(e, dtype=torch.float64), "grad": torch.tensor(g, dtype=torch.float64)}
    x = _vector(S.D, case["dtype"], seed, dev)
    x = x.to(torch.complex128 if x.is_complex() else torch.float64)
    if op == "lanczos":
        if case["steps"] > S.D // 2:
            return None
        al, be, e, psi = S.lanczos(x, p.J, case["steps"])
        return {"E0": e, "alpha": al, "beta": be, "psi": psi}
    if op == "expect":
        return np.array([float(torch.vdot(x, h).real) for h in S.classes(x)])
    return S.apply(x, p.J, _rows(case, S.D) if op == "rows" else None)


def _exact_batch(case, seed, dev):
    probs, k = _sq25(case["up"], case["up_to"]), case["k"]
    sectors = [_Sector64(p, dev) for p in probs]
    dims, reals = [S.D for S in sectors], [p.is_real() for p in probs]
    off, n = _batch_layout(dims, reals, k)
    g = torch.Generator(device=dev).manual_seed(int(seed))
    X = {r: torch.randn(n[r], dtype=torch.float32 if r else torch.complex64, device=dev, generator=g) for r in (True, False)}
    Y = {r: torch.zeros(n[r], dtype=torch.float64 if r else torch.complex128, device=dev) for r in (True, False)}
    for p, S, r, o in zip(probs, sectors, reals, off):
        if S.D:
            x = X[r][o:o + S.D * k].view(S.D, k).to(Y[r].dtype)
            Y[r][o:o + S.D * k] = S.apply(x, p.J).reshape(-1)
    return [Y[True], Y[False]]
