"""Hierarchies made, solved and destroyed by several threads at once."""
import threading

import pytest

torch = pytest.importorskip("torch")
import paper_1803_02481_gb300 as bm  # noqa: E402

pytestmark = pytest.mark.gpu


def run_threads(works):
    errors = []

    def guard(work):
        try:
            work()
        except Exception as e:   # a thread's exception must fail the test
            errors.append(repr(e))

    threads = [threading.Thread(target=guard, args=(w,)) for w in works]
    for t in threads:
        t.start()
    for t in threads:
        t.join()
    assert not errors, errors[:3]


def test_destroying_leaves_other_threads_recordings_alone_3d():
    """A first solve records its cycle; hierarchies destroyed by other threads
    meanwhile must not spoil the recording."""
    k = torch.ones((9, 10, 11), device="cuda", dtype=torch.float64)
    b = torch.ones_like(k)
    torch.cuda.synchronize()

    def work():
        s = torch.cuda.Stream()
        x = torch.zeros_like(b)
        s.synchronize()
        for _ in range(60):
            h = bm.setup3(k, stream=s)
            h.solve(b, x=x, tol=1e-6, stream=s)
            h.destroy()

    run_threads([work] * 4)


def test_destroying_leaves_other_threads_recordings_alone_2d():
    """A hierarchy whose recording failed would launch its cycles one by one:
    many kernel launches in every later solve, where the recorded loop has a
    few."""
    k = torch.ones((100, 90), device="cuda", dtype=torch.float64)
    b = torch.ones_like(k)
    torch.cuda.synchronize()
    kept, done = [], threading.Event()

    def make():
        s = torch.cuda.Stream()
        x = torch.zeros_like(b)
        s.synchronize()
        try:
            for _ in range(60):
                h = bm.setup(k, stream=s)
                h.solve(b, x=x, tol=1e-10, stream=s)
                kept.append(h)
        finally:
            done.set()

    def churn():
        s = torch.cuda.Stream()
        while not done.is_set():
            bm.setup(k, stream=s).destroy()

    run_threads([make, churn, churn])
    counts = set()
    for h in kept:
        before = bm.kernel_launches()
        h.solve(b, tol=1e-10)
        counts.add(bm.kernel_launches() - before)
        h.destroy()
    assert len(counts) == 1 and max(counts) < 12, counts


@pytest.mark.parametrize("kind", ["2d", "refine", "pcg", "lines", "3d", "batch"])
def test_device_wide_waits_beside_first_solves(kind):
    """A wait for the whole device, which any part of a program may make at
    any time, is no concern of a solve that is being recorded: every first
    solve goes through and gives the same values."""
    opts = {"2d": {}, "refine": {"precision": bm.BMG_FP32_REFINE}, "pcg": {"solver": bm.BMG_SOLVER_PCG, "nu1": 1},
            "lines": {"smoother": bm.BMG_SMOOTH_ALTLINE}}.get(kind, {})
    shape = (17, 18, 19) if kind == "3d" else (63, 63) if kind == "batch" else (70, 90)
    g = torch.Generator(device="cuda")
    g.manual_seed(7)
    k = 10.0 ** torch.rand(shape, generator=g, device="cuda", dtype=torch.float64)
    b = torch.rand(shape, generator=g, device="cuda", dtype=torch.float64) - 0.5
    torch.cuda.synchronize()

    def solve(s=None):
        x = torch.zeros_like(b)
        torch.cuda.current_stream().synchronize()
        if kind == "batch":
            h = bm.Batch([k, k], bm.default_options(), stream=s)
            y = torch.zeros_like(b)
            torch.cuda.current_stream().synchronize()
            h.solve([b, b], [x, y], tol=1e-9, stream=s)
        else:
            h = (bm.setup3 if kind == "3d" else bm.setup)(k, bm.default_options(**opts), stream=s)
            h.solve(b, x=x, tol=1e-9, stream=s)
        h.destroy()
        return x

    want, done = solve(), threading.Event()

    def work():
        s = torch.cuda.Stream()
        try:
            for _ in range(40):
                assert torch.equal(solve(s), want)
        finally:
            done.set()

    def wait():
        while not done.is_set():
            torch.cuda.synchronize()

    run_threads([work, work, wait])


def test_destroy_waits_for_the_work_a_call_left():
    """The single operations return with their work under way; a hierarchy
    destroyed then keeps its memory until they are done, on either of two
    streams, whoever asks for memory next."""
    n = 2000
    g = torch.Generator(device="cuda")
    g.manual_seed(1)
    k = 10.0 ** torch.rand((n, n), generator=g, device="cuda", dtype=torch.float64)
    b = torch.rand((n, n), generator=g, device="cuda", dtype=torch.float64)
    h = bm.setup(k)
    want = h.op_relax(h.nlevels - 1, torch.zeros_like(b), b, 60)
    torch.cuda.synchronize()
    h.destroy()
    streams = [torch.cuda.Stream(), torch.cuda.Stream()]
    for s in streams * 2:
        h = bm.setup(k)
        x = torch.zeros_like(b)
        torch.cuda.synchronize()
        r = torch.empty((n // 2, n // 2), device="cuda", dtype=torch.float64)
        h.op_restrict(h.nlevels - 1, b, r, stream=streams[0])
        h.op_relax(h.nlevels - 1, x, b, 60, stream=s)
        h.destroy()
        bm.setup(k * 2.0, stream=streams[1 if s is streams[0] else 0]).destroy()
        torch.cuda.synchronize()
        assert torch.equal(x, want)
def test_setups_of_different_coarsest_sizes_at_once():
    """The coarsest factorisation takes shared memory by its size: 81 to 159
    unknowns, all above the 48 KB a kernel has without asking."""
    ks = [torch.ones((3, n), device="cuda", dtype=torch.float64) for n in (27, 35, 45, 53)]
    torch.cuda.synchronize()

    def work(turn):
        def run():
            s = torch.cuda.Stream()
            for r in range(250):
                bm.setup(ks[(r + turn) % len(ks)], stream=s).destroy()
        return run

    run_threads([work(t) for t in range(4)])


