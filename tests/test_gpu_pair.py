"""The coset-arithmetic product (csrc/pair.cu) at the edges of what it accepts: halves made of
the split's blocks or of a colouring of the bonds, halves that are exchanged by an involution,
by other elements only or by none, spin flips (as a factor of the group and tied to other
elements), trivial, sign and complex characters, fillings whose halves hold no or all spins,
every vector type, row ranges on both sides of the size rules, each of the ways a product is
taken (asked for, so that a rule that moves does not empty a test), several streams and host
threads at once and a captured call.  Reference: the oracle's explicit matrix on small sectors,
on large ones the search kernels.  Bounds: as in test_gpu_parity, a row sums at most a few
hundred terms of size max|J| |x|, so fp64 stays near 1e-15 relative (1e-12 asked) and fp32
within a few roundings (2e-6 asked)."""
import dataclasses

import numpy as np
import pytest

import oracle
import workloads as w

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu

T = w.square_torus


def _sub(p, sel, name, **kw):
    sel = np.asarray(sel)
    return dataclasses.replace(p, perm=p.perm[sel], phase_num=p.phase_num[sel], name=name, **kw)


SECTORS = [
    w.chain(12, 2, k=5, n_up=6), w.chain(12, 4, k=6, n_up=5), w.chain(16, 4, k=3, n_up=8),
    w.chain(20, 2, k=10, n_up=9),
    w.chain(10, 2, k=0, n_up=0), w.chain(10, 2, k=0, n_up=1), w.chain(10, 2, k=5, n_up=9),
    _sub(w.chain(12, 2, k=2, n_up=6), range(0, 12, 2), "chain12_even_translations"),
    _sub(w.chain(12, 2, k=0, n_up=6), [0], "chain12_identity"),
    dataclasses.replace(w.chain(12, 2, k=2, n_up=6), flip=(np.arange(12) % 2).astype(np.uint8), name="chain12_flip_tied"),
    w.with_spin_flip(w.chain(12, 4, k=3, n_up=6), 1), w.with_spin_flip(w.chain(12, 2, k=0, n_up=6), 0),
    T(4, momentum=(0, 0), point_irrep=3, J2=0.5, n_sublat=2, n_up=7),
    T(4, momentum=(1, 0), point_irrep=1, J2=0.5, n_sublat=4, n_up=5),
    T(4, momentum=(1, 2), point_irrep=0, J2=0.5, n_sublat=4, n_up=8),
    w.with_spin_flip(T(4, momentum=(2, 2), point_irrep=1, J2=0.5, n_sublat=4, n_up=8), 1),
    T(6, momentum=(0, 0), point_irrep=1, J2=0.5, n_sublat=4, n_up=4),
    # halves that are no blocks of the split: the two colours of the nearest-neighbour bonds
    w.chain(12, 1, k=5, n_up=6), w.chain(12, 3, k=6, n_up=5), w.chain(20, 5, k=7, n_up=9),
    w.chain(16, 8, k=8, n_up=7), w.with_spin_flip(w.chain(12, 1, k=5, n_up=6), 1),
    T(4, momentum=(1, 1), point_irrep=0, J2=0.5, n_sublat=1, n_up=6),
    w.with_spin_flip(T(4, momentum=(0, 0), point_irrep=2, J2=0.5, n_sublat=1, n_up=8), 0),
    # no such halves: the search kernels
    w.chain(9, 3, k=2, n_up=4), T(3, momentum=(1, 2), point_irrep=0, J2=0.4, n_sublat=1, n_up=4),
]


def _basis(p):
    import paper_1804_05028_gb300 as ed
    return ed.build_basis_from(p)


def _vec(D, dtype, seed):
    g = torch.Generator(device="cuda").manual_seed(seed)
    return torch.randn(D, dtype=dtype, device="cuda", generator=g)


@pytest.mark.parametrize("p", SECTORS, ids=lambda p: f"{p.name}_up{p.n_up}")
def test_product_of_every_type(p):
    B = _basis(p)
    H, _, _ = oracle.hamiltonian(p)
    real = [torch.float64, torch.float32] if B.is_real else []
    for dt in real + [torch.complex128, torch.complex64]:
        x = _vec(B.dim, dt, 3)
        xd = x.cpu().to(torch.complex128).numpy()
        ref = H @ xd
        tol = (2e-6 if dt in (torch.float32, torch.complex64) else 1e-12) * max(np.abs(ref).max(), 1e-30)
        assert np.abs(B.apply_H(x).cpu().numpy() - ref).max() <= tol
        # <x|H_c|x> per class: |sum of the row shares| <= sum |x_i| |(H_c x)_i|
        got = B.expect_classes(x, Jz=p.Jz)
        for c in range(p.n_classes):
            J = [0.0] * p.n_classes
            J[c] = 1.0
            hc = oracle.hamiltonian(p.with_couplings(J, p.Jz))[0] @ xd
            scale = np.abs(xd) @ np.abs(hc) + np.abs(xd) @ np.abs(xd)
            assert abs(got[c] - np.vdot(xd, hc).real) <= (2e-6 if tol > 1e-9 * np.abs(ref).max() else 1e-12) * scale
        # the rows of a range: most of them, the fewest that coset arithmetic takes, one less
        for r0, r1 in [(B.dim // 5, B.dim - B.dim // 7), (B.dim // 2, B.dim // 2 + 16), (B.dim // 2, B.dim // 2 + 15)]:
            r1 = min(r1, B.dim)
            if r0 < r1:
                assert np.abs(B.apply_H_rows(x, r0, r1).cpu().numpy() - ref[r0:r1]).max() <= tol


def _searched(B, x, y, tol, n=48):
    """Rows of y against the search kernels, which take ranges of fewer than 16 rows and share no
    table with the coset arithmetic but the basis."""
    D, scale = B.dim, y.abs().max()
    assert B.apply_route(x.dtype, 0, 15) == "search"
    for r0 in np.linspace(0, D - 15, n).astype(np.int64).tolist():
        assert (B.apply_H_rows(x, r0, r0 + 15) - y[r0:r0 + 15]).abs().max() <= tol * scale


def _ops(p, even, odd):
    """The elements of a 6x6 group whose translation keeps the checkerboard and whose point
    operation is in `even`, or exchanges it and is in `odd`; operation of each."""
    sel, ops = [], []
    for g, name in enumerate(p.sym_names):
        op, t = name.split("+t")
        if op in (odd if sum(eval(t)) % 2 else even):
            sel.append(g)
            ops.append(op)
    return sel, ops


def _no_involution(n_up):
    """Quarter turns about plaquettes, which exchange the checkerboard halves and square to half
    turns, half turns and translations inside the halves; characters i^(quarter turns)."""
    p = T(6, momentum=(0, 0), point_irrep=0, J2=0.5, n_sublat=4, n_up=n_up)
    sel, ops = _ops(p, ("E", "C2"), ("C4", "C4^3"))
    q = _sub(p, sel, "square36_quarter_turns")
    turns = {"E": 0, "C4": 1, "C2": 2, "C4^3": 3}
    return dataclasses.replace(q, phase_denom=4, phase_num=np.array([turns[o] for o in ops], np.int32))


def _halves_kept(momentum, n_up):
    p = T(6, momentum=momentum, point_irrep=1, J2=0.5, n_sublat=4, n_up=n_up)
    return _sub(p, _ops(p, w.C4V_NAMES, ())[0], f"square36_k{momentum}_halves_kept")


# what the slot order distinguishes: characters (signs or complex), tables for two upper classes
# per slice (32 or more elements between the halves) or none, an involution that exchanges the
# halves, another exchange (a second multiplication table) or none, spin flips as a factor of the
# group or tied to its elements, halves of blocks or of colours; and the types that reach it
ALL = [torch.float64, torch.float32, torch.complex128, torch.complex64]
LARGE = [
    (T(6, momentum=(0, 0), point_irrep=1, J2=0.5, n_sublat=4, n_up=12), ALL),
    (T(6, momentum=(1, 1), point_irrep=1, J2=0.5, n_sublat=4, n_up=11), ALL[2:]),
    (T(6, momentum=(1, 2), point_irrep=0, J2=0.5, n_sublat=4, n_up=10), ALL[2:]),
    (_no_involution(11), ALL[2:]),
    (w.chain(32, 4, k=5, n_up=12), ALL[2:3]),
    (_halves_kept((0, 0), 12), ALL),
    (_halves_kept((1, 1), 10), ALL[2:]),
    (w.with_spin_flip(w.chain(32, 4, k=0, n_up=16), 1), [torch.float64, torch.complex64]),
    (w.with_spin_flip(w.chain(32, 4, k=5, n_up=16), 0), ALL[2:]),
    (dataclasses.replace(w.chain(32, 4, k=3, n_up=16), flip=(np.arange(32) % 2).astype(np.uint8), name="chain32_flip_tied"), ALL[2:]),
    (w.chain(36, 3, k=7, n_up=11), ALL[2:]),
]


@pytest.mark.parametrize("p,types", LARGE, ids=lambda v: f"{v.name}_up{v.n_up}" if hasattr(v, "n_up") else "")
def test_row_order(p, types):
    """Whole products in slot order against the search kernels on sampled rows, and against row
    ranges in basis order everywhere: the same terms summed in another order."""
    B = _basis(p)
    D = B.dim
    for dt in types:
        assert B.apply_route(dt) == "slot order" and B.apply_route(dt, classes=True) == "slot order"
        x = _vec(D, dt, 4)
        y = B.apply_H(x)
        tol = 2e-6 if dt in (torch.float32, torch.complex64) else 1e-12
        _searched(B, x, y, tol)
        cut = D // 3 + 1
        assert B.apply_route(dt, 0, cut) == "expanded"
        ref = torch.cat([B.apply_H_rows(x, 0, cut), B.apply_H_rows(x, cut, D)])
        assert (y - ref).abs().max() <= tol * ref.abs().max()
        mid = B.apply_H_rows(x, D // 2, D // 2 + 1001)      # a narrow range
        assert (y[D // 2:D // 2 + 1001] - mid).abs().max() <= tol * ref.abs().max()
        got = B.expect_classes(x)
        # blocks take the rows in any order, the sums come out the same
        assert all(np.array_equal(got, B.expect_classes(x)) for _ in range(3))
        runs = [B.lanczos(dtype=dt, fixed_steps=4) for _ in range(3)] if dt.is_complex != B.is_real else []
        assert all(np.array_equal(r["alpha"], runs[0]["alpha"]) and np.array_equal(r["beta"], runs[0]["beta"]) for r in runs)
        xd = x.to(torch.complex128)
        for c in range(p.n_classes):
            J = [0.0] * p.n_classes
            J[c] = 1.0
            hc = B.apply_H_rows(x, 0, D - 1, J=J).to(torch.complex128)
            ref_c = torch.vdot(xd[:-1], hc).real.item()
            last = B.apply_H_rows(x, D - 1, D, J=J).to(torch.complex128)
            ref_c += (xd[-1].conj() * last[0]).real.item()
            assert abs(got[c] - ref_c) <= tol * (xd.abs()[:-1] @ hc.abs()).item()
    B.close()


DIRECT = [
    T(6, momentum=(0, 0), point_irrep=1, J2=0.5, n_sublat=4, n_up=6), T(6, momentum=(1, 2), point_irrep=0, J2=0.5, n_sublat=4, n_up=6),
    w.chain(28, 4, k=5, n_up=7), w.chain(30, 3, k=15, n_up=7), w.with_spin_flip(w.chain(24, 4, k=0, n_up=12), 1),
    _sub(w.chain(28, 4, k=4, n_up=7), range(0, 28, 2), "chain28_even_translations"),
]


@pytest.mark.parametrize("p", DIRECT, ids=lambda p: f"{p.name}_up{p.n_up}")
def test_direct_rows(p):
    """Narrow ranges read x through the slots, the whole product expands it first: the same values
    summed in the same order, so the same bits (16 rows: the fewest; 17 and 33: a ragged warp)."""
    B = _basis(p)
    D = B.dim
    for dt in ([torch.float64, torch.float32] if B.is_real else []) + [torch.complex128, torch.complex64]:
        x = _vec(D, dt, 6)
        y = B.apply_H(x)
        for r0, n in [(0, 16), (D // 3, 17), (D - 33, 33), (D // 2, 66)]:
            assert torch.equal(B.apply_H_rows(x, r0, r0 + n), y[r0:r0 + n])


def test_streams_and_capture():
    p = T(6, momentum=(0, 0), point_irrep=1, J2=0.5, n_sublat=4, n_up=6)
    B = _basis(p)
    xs = [_vec(B.dim, torch.float32, s) for s in range(4)]
    ref = [B.apply_H(x).clone() for x in xs]
    ys = [torch.empty_like(x) for x in xs]
    streams = [torch.cuda.Stream() for _ in xs]
    torch.cuda.synchronize()
    for _ in range(20):
        for x, y, s in zip(xs, ys, streams):
            B.apply_H(x, y, stream=s)
    torch.cuda.synchronize()
    for y, r in zip(ys, ref):
        assert torch.equal(y, r)
    # captured once, replayed on other contents of the same buffers
    x, y = torch.empty_like(xs[0]), torch.empty_like(xs[0])
    g = torch.cuda.CUDAGraph()
    x.copy_(xs[0])
    torch.cuda.synchronize()
    with torch.cuda.graph(g):
        B.apply_H(x, y)
    for v, r in zip(xs, ref):
        x.copy_(v)
        y.zero_()
        g.replay()
        torch.cuda.synchronize()
        assert torch.equal(y, r)
    del g


def test_threads_with_other_table_sizes():
    """Two host threads whose sectors take different amounts of shared memory in one kernel: what
    one thread sets for its launch leaves the other's as it was."""
    import threading
    ps = [w.chain(8, 2, k=0, n_up=4), T(6, momentum=(0, 0), point_irrep=0, J2=0.5, n_sublat=4, n_up=4),   # coset arithmetic
          w.chain(9, 3, k=0, n_up=4), w.chain(33, 3, k=0, n_up=3)]                                        # search
    errors = []

    def work(p):
        try:
            B = _basis(p)
            x = _vec(B.dim, torch.float64, 5)
            s = torch.cuda.Stream()
            s.wait_stream(torch.cuda.default_stream())
            y, ref = torch.empty_like(x), B.apply_H(x, stream=s)
            for _ in range(3000):
                B.apply_H(x, y, stream=s)
            s.synchronize()
            assert torch.equal(y, ref)
        except Exception as e:   # noqa: BLE001 -- reported by the main thread
            errors.append(e)

    for pair in (ps[:2], ps[2:]):
        threads = [threading.Thread(target=work, args=(p,)) for p in pair]
        for t in threads:
            t.start()
        for t in threads:
            t.join()
    assert not errors, errors


def test_tables_too_wide_for_the_slot_order():
    """Third-neighbour bonds and complex characters on the 40-site cluster: the slot order would
    need 209 KB of shared memory, the rows in basis order 93; with two couplings it fits."""
    two = w.tilted_square_40(momentum=(0, 0), point_irrep=1, n_sublat=4, J2=0.5, n_up=10)
    cl = w._Cluster((6, 2), (-2, 6))
    at = {cl.key(int(x), int(y)): lab for lab, (x, y) in enumerate(two.coords)}
    third = [(lab, at[cl.key(int(x) + dx, int(y) + dy)]) for lab, (x, y) in enumerate(two.coords) for dx, dy in ((2, 0), (0, 2))]
    three = dataclasses.replace(two, bonds=np.concatenate([two.bonds, np.array(third, np.int32)]),
                                bond_class=np.concatenate([two.bond_class, np.full(len(third), 2, np.int32)]),
                                n_classes=3, J=(1.0, 0.5, 0.3), Jz=(1.0, 0.8, 0.6))
    for p, route in ((two, "slot order"), (three, "expanded")):
        B = _basis(p)
        for dt, tol in ((torch.complex64, 2e-6), (torch.complex128, 1e-12)):
            assert B.apply_route(dt) == route and B.apply_route(dt, classes=True) == route
            x = _vec(B.dim, dt, 7)
            _searched(B, x, B.apply_H(x), tol)
        B.close()


def test_product_without_scratch():
    """Where the pool has no room for x over the slots, terms read it through their indices: the
    same bits as in basis order."""
    B = _basis(w.chain(32, 4, k=0, n_up=14))          # 59 MB; builds leave up to 64 MB for the widest type in the pool
    x = _vec(B.dim, torch.float32, 8)
    y, z = torch.empty_like(x), torch.empty_like(x)
    assert B.apply_route(torch.float32) == "expanded"
    torch.cuda.synchronize()
    hold = torch.empty(torch.cuda.mem_get_info()[0] - (8 << 20), dtype=torch.uint8, device="cuda")
    B.apply_H(x, y)
    torch.cuda.synchronize()
    left = torch.cuda.mem_get_info()[0]
    del hold
    torch.cuda.empty_cache()
    assert torch.equal(B.apply_H(x, z), y) and left <= 16 << 20


def test_lanczos_beside_products_of_another_thread():
    """A product on the same basis from another thread, over another number of blocks, does not
    change how many block sums a Lanczos step adds up."""
    import threading
    B = _basis(w.chain(20, 2, k=0, n_up=10))
    x = _vec(B.dim, torch.float64, 10)
    ref = B.lanczos(fixed_steps=8, seed=2)
    stop = threading.Event()

    def narrow():
        s = torch.cuda.Stream()
        y = torch.empty(64, dtype=x.dtype, device="cuda")
        while not stop.is_set():
            B.apply_H_rows(x, 100, 164, y=y, stream=s)
        s.synchronize()

    t = threading.Thread(target=narrow)
    t.start()
    try:
        runs = [B.lanczos(fixed_steps=8, seed=2) for _ in range(400)]
    finally:
        stop.set()
        t.join()
    assert all(np.array_equal(r["alpha"], ref["alpha"]) and np.array_equal(r["beta"], ref["beta"]) for r in runs)
