"""Timing kernel classes (profile_set) is a switch of the whole process: a
cycle that another thread's switch overtakes keeps its values.  A level whose
legs are one kernel each holds its iterate in another buffer between the legs
than one launched an operation at a time, so the two must not meet in one
cycle."""
import threading

import pytest

torch = pytest.importorskip("torch")
import paper_1803_02481_gb300 as bm  # noqa: E402

pytestmark = pytest.mark.gpu


@pytest.fixture
def toggling():
    """A thread that turns the timing of one class on and off until the test ends."""
    stop = threading.Event()

    def work():
        while not stop.is_set():
            bm.profile_set(("fine_interp",))
            bm.profile_set(())

    t = threading.Thread(target=work)
    yield t
    stop.set()
    t.join()
    bm.profile_set(())


def problem(nx, ny):
    g = torch.Generator(device="cuda")
    g.manual_seed(nx + ny)
    k = 10.0 ** (2.0 * torch.rand((ny, nx), generator=g, device="cuda", dtype=torch.float64) - 1.0)
    return k, torch.rand((ny, nx), generator=g, device="cuda", dtype=torch.float64) - 0.5


def test_cycles_keep_their_values_while_timing_is_switched(toggling):
    k, b = problem(200, 150)
    h = bm.setup(k)
    top = h.nlevels - 1
    want = h.vcycle_from(top, b, torch.empty_like(b))
    toggling.start()
    wrong = 0
    for _ in range(2000):
        wrong += not torch.equal(h.vcycle_from(top, b, torch.empty_like(b)), want)
    h.destroy()
    assert wrong == 0


@pytest.mark.parametrize("kw", [{}, {"precision": bm.BMG_FP32_REFINE},
                                {"solver": bm.BMG_SOLVER_PCG, "nu1": 1},
                                {"solver": bm.BMG_SOLVER_PCG, "nu1": 1, "precision": bm.BMG_FP32_REFINE}])
def test_solves_keep_their_values_while_timing_is_switched(toggling, kw):
    """Each hierarchy records its solve anew."""
    k, b = problem(120, 130)
    opts = bm.default_options(**kw)

    def solve():
        h = bm.setup(k, opts)
        x, _ = h.solve(b, tol=1e-10)
        h.destroy()
        return x

    want = solve()
    toggling.start()
    wrong = sum(not torch.equal(solve(), want) for _ in range(150))
    assert wrong == 0


# one tile and less, tile edges and one beyond, even sides, long thin grids,
# sides where the tile shape changes
@pytest.mark.parametrize("nu1,nu2", [(2, 1), (1, 1), (2, 2)])
@pytest.mark.parametrize("nx,ny", [(5, 5), (8, 9), (17, 16), (33, 31), (64, 65), (127, 129), (150, 300), (3, 200),
                                   (260, 7), (513, 255), (1030, 40)])
@pytest.mark.parametrize("prec", [bm.BMG_FP64, bm.BMG_FP32_REFINE])
def test_timed_cycles_equal_untimed_ones(prec, nx, ny, nu1, nu2):
    """While a class is timed every operation is a launch of its own: one and
    two cycles of the legs, in both precisions, give the same values."""
    k, b = problem(nx, ny)
    for cycles in (1, 2):
        got = []
        for classes in ((), ("fine_interp",)):
            h = bm.setup(k, bm.default_options(nu1=nu1, nu2=nu2, precision=prec, max_cycles=cycles))
            bm.profile_set(classes)
            try:
                got.append(h.solve(b, tol=1e-300, allow_noconv=True)[0])
            finally:
                bm.profile_set(())
                h.destroy()
        assert torch.equal(*got), cycles
