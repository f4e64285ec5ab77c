"""Memory kept from destroyed hierarchies goes back on request."""
import pytest

torch = pytest.importorskip("torch")
import paper_1803_02481_gb300 as bm  # noqa: E402

pytestmark = pytest.mark.gpu


def free():
    torch.cuda.synchronize()
    torch.cuda.empty_cache()
    return torch.cuda.mem_get_info()[0]


def test_release_memory_gives_back_what_is_kept():
    n = 2000
    least = 10 * 8 * n * n   # ten FP64 planes of the finest level alone
    bm.release_memory()
    k = torch.ones((n, n), device="cuda", dtype=torch.float64)
    bm.setup(k).destroy()
    bm.release_memory()      # (whatever the first setup loads stays)
    before = free()
    h = bm.setup(k)
    h.destroy()
    m = bm.setup3(torch.ones((40, 41, 42), device="cuda", dtype=torch.float64))
    kept = before - free()
    assert kept >= least
    bm.release_memory()
    assert before - free() <= kept - least   # what is in use stays
    x, _ = m.solve(torch.ones((40, 41, 42), device="cuda", dtype=torch.float64), tol=1e-6)
    m.destroy()
    bm.release_memory()
    del x
    assert abs(before - free()) <= 64 << 20
