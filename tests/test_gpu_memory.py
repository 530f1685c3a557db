"""Builds and products where device memory is short: a tensor takes all but a given amount first.
Out of memory is an ordinary error here, reported by the allocation."""
import contextlib
import gc

import pytest

import workloads as w

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu

MB = 1 << 20


def free_bytes():
    torch.cuda.synchronize()
    return torch.cuda.mem_get_info()[0]


@contextlib.contextmanager
def memory_left(n):
    """Leaves about n bytes of the device free (the driver hands memory out in steps of 2 MB)."""
    gc.collect()
    torch.cuda.empty_cache()
    hold = torch.empty(max(free_bytes() - n, 1), dtype=torch.uint8, device="cuda")
    try:
        yield
    finally:
        del hold
        torch.cuda.empty_cache()


def build(p, **kw):
    import paper_1804_05028_gb300 as ed
    return ed.build_basis_from(p, **kw)


def test_failed_build_gives_its_scratch_back():
    import paper_1804_05028_gb300 as ed
    p = w.config_square36()
    build(w.chain(12, 2, k=0, n_up=6)).close()      # the context's own allocations
    with memory_left(200 * MB):                     # the basis alone takes 316 MB
        left = [free_bytes()]
        for _ in range(3):
            with pytest.raises(ed.EdError) as e:
                build(p)
            assert e.value.code == 3
            left.append(free_bytes())
        assert left[0] - left[1] <= 66 * MB and left[3] >= left[1] - 2 * MB   # the shared pool keeps 64 MB


def test_pool_gives_way_to_a_build():
    """What the shared pool keeps of earlier scratch is there for a basis that needs it."""
    p = w.square_torus(6, momentum=(0, 0), point_irrep=0, J2=0.5, n_sublat=4, n_up=12)
    B = build(p, bucket_target=64)                  # an index of 10 MB beside the basis
    x = torch.rand(B.dim, dtype=torch.float32, device="cuda")
    ref, y = B.apply_H(x), torch.empty_like(x)
    basis = B.info()["basis_bytes"]
    B.close()
    build(p.with_n_up(10)).close()                  # leaves its scratch in the pool
    with memory_left(basis - 4 * MB):
        B = build(p, bucket_target=64)
        B.apply_H(x, y)
        B.close()
    assert (y - ref).abs().max() <= 2e-6 * ref.abs().max()


def test_plan_leaves_room_for_a_lanczos_run():
    """The tables of coset arithmetic (140 MB here) are not made where the run's vectors would
    then find no room: the sector is searched, as without them."""
    p = w.square_torus(6, momentum=(0, 0), point_irrep=0, J2=0.5, n_sublat=4, n_up=12)
    B = build(p)
    i = B.info()
    ref = B.lanczos(fixed_steps=3, seed=3)["E0"]
    assert B.apply_route(torch.float64) == "slot order"
    B.close()
    with memory_left(i["basis_bytes"] + i["index_bytes"] + 190 * MB):
        B = build(p)
        route = B.apply_route(torch.float64)
        e = B.lanczos(fixed_steps=3, seed=3)["E0"]
        B.close()
    assert route == "search" and abs(e - ref) <= 1e-12 * abs(ref)


def test_pool_of_a_basis_is_bounded():
    """Sixteen products in flight take sixteen times the scratch, of which two times stay."""
    p = w.square_torus(6, momentum=(0, 0), point_irrep=0, J2=0.5, n_sublat=4, n_up=12)
    B = build(p)
    x = torch.rand(B.dim, dtype=torch.float64, device="cuda")
    ys = [torch.empty_like(x) for _ in range(16)]
    streams = [torch.cuda.Stream() for _ in ys]
    B.apply_H(x, ys[0])
    before = free_bytes()
    for y, s in zip(ys, streams):
        B.apply_H(x, y, stream=s)
    held = before - free_bytes()
    assert all(torch.equal(y, ys[0]) for y in ys)
    assert held <= 2 * 8 * 2 * B.dim + 40 * MB      # slots: less than twice the states
    B.close()
