"""Memory kept between hierarchies: handed on without a trace of its former
owner, bounded, and safe with several threads and streams."""
import threading

import pytest

torch = pytest.importorskip("torch")
import paper_1803_02481_gb300 as bm  # noqa: E402

pytestmark = pytest.mark.gpu


def problem(n, seed):
    g = torch.Generator(device="cuda")
    g.manual_seed(seed)
    k = 10.0 ** (2.0 * torch.rand((n, n), generator=g, device="cuda", dtype=torch.float64) - 1.0)
    return k, torch.rand((n, n), generator=g, device="cuda", dtype=torch.float64) - 0.5


def solve(n, seed, stream=None, **kw):
    k, b = problem(n, seed)
    torch.cuda.synchronize()
    h = bm.setup(k, bm.default_options(**kw), stream=stream)
    x = torch.zeros_like(b)
    torch.cuda.current_stream().synchronize()
    h.solve(b, x=x, tol=1e-10, stream=stream)
    h.destroy()
    return x


def test_blocks_are_bounded_and_reused_clean():
    want = solve(200, 1)
    total = torch.cuda.get_device_properties(0).total_memory
    torch.cuda.synchronize()
    before = torch.cuda.mem_get_info()[0]
    for n in (700, 201, 1500, 90, 2500, 199, 3000, 1025):
        solve(n, n)
        # the same problem in whatever block it now gets
        assert torch.equal(solve(200, 1), want)
    torch.cuda.empty_cache()
    kept = before - torch.cuda.mem_get_info()[0]
    assert kept <= total / 32 + (64 << 20)


def test_threads_and_streams():
    sizes = [63, 200, 255, 333]
    want = {n: solve(n, n) for n in sizes}
    errors = []

    def work(t):
        try:
            s = torch.cuda.Stream()
            for r in range(6):
                n = sizes[(t + r) % len(sizes)]
                if not torch.equal(solve(n, n, stream=s), want[n]):
                    errors.append((t, n))
        except Exception as e:   # a thread's exception must fail the test
            errors.append((t, repr(e)))

    threads = [threading.Thread(target=work, args=(t,)) for t in range(4)]
    for t in threads:
        t.start()
    for t in threads:
        t.join()
    assert not errors, errors
