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
        before = free_bytes()
        with pytest.raises(ed.EdError) as e:
            build(p)
        assert e.value.code == 3
        assert before - free_bytes() < 4 * MB
