"""The default level schedule: the levels of at most 300 points (100 with line
smoothing) in one block, whatever the sides; explicit choices are kept."""
import pytest

torch = pytest.importorskip("torch")
import paper_1803_02481_gb300 as bm  # noqa: E402

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("smoother,points", [(bm.BMG_SMOOTH_POINT, 300), (bm.BMG_SMOOTH_ALTLINE, 100)])
@pytest.mark.parametrize("nx,ny", [(3, 200), (17, 17), (40, 31), (255, 255), (500, 31), (700, 130)])
def test_default_threshold(nx, ny, smoother, points):
    k = torch.ones((ny, nx), device="cuda", dtype=torch.float64)
    h = bm.setup(k, bm.default_options(smoother=smoother))
    _, info = h.solve(k, tol=1e-6)
    sizes = [h.level_shape(level) for level in range(h.nlevels)]
    h.destroy()
    want = 1
    while want < len(sizes) and sizes[want][0] * sizes[want][1] <= points:
        want += 1
    assert (info.threshold, info.coarse_ctas) == (want, 1)


def test_explicit_schedules_are_kept():
    k = torch.ones((255, 255), device="cuda", dtype=torch.float64)
    for thr, ctas in ((1, -1), (3, 1), (7, 1), (4, 2), (7, -1)):
        h = bm.setup(k, bm.default_options(coarse_threshold=thr, coarse_ctas=ctas))
        _, info = h.solve(k, tol=1e-8)
        h.destroy()
        assert info.threshold == thr
        assert info.coarse_ctas == ctas if ctas > 0 else 1 <= info.coarse_ctas <= bm.max_coarse_ctas()
