"""The fused legs of a V-cycle level and the shared-memory coarse sub-cycle
against the same cycle composed of the single-operation entry points: every
value equal, on sides around the tiles' edges, even and odd, and for every
schedule threshold; the coarsest solve against a dense solve."""
import numpy as np
import pytest

torch = pytest.importorskip("torch")
import paper_1803_02481_gb300 as bm  # noqa: E402

pytestmark = pytest.mark.gpu

# one tile and less, tile edges and one beyond, even sides, long thin grids,
# a side where the legs' tile shape changes, a prescaled finest level
SIZES = [(5, 5), (8, 9), (17, 16), (33, 31), (64, 65), (127, 129), (150, 300), (3, 200), (260, 7), (513, 255),
         (1030, 40)]


def cycle(h, level, b, nu1, nu2):
    """One V(nu1, nu2) cycle from zero, an entry point per operation."""
    x = torch.zeros_like(b)
    if level == 0:
        return h.vcycle_from(0, b, x)
    h.op_relax(level, x, b, nu1)
    r = torch.empty_like(b)
    h.op_residual(level, x, b, r)
    nx, ny = h.level_shape(level - 1)
    bc = torch.empty((ny, nx), dtype=torch.float64, device="cuda")
    h.op_restrict(level, r, bc)
    h.op_interp(level, cycle(h, level - 1, bc, nu1, nu2), x)
    return h.op_relax(level, x, b, nu2, reverse=True)


@pytest.mark.parametrize("nu1,nu2", [(2, 1), (1, 1), (3, 1), (1, 0)])
@pytest.mark.parametrize("nx,ny", SIZES)
def test_cycle_equals_its_operations(nx, ny, nu1, nu2):
    g = torch.Generator(device="cuda")
    g.manual_seed(nx * 1000 + ny)

    def rand(*s):
        return torch.rand(s, generator=g, device="cuda", dtype=torch.float64)

    k = 10.0 ** (2.0 * rand(ny, nx) - 1.0)
    want = {}
    for thr in (-1, 1, 2, 3, 4):
        probe = bm.setup(k, bm.default_options())
        levels = probe.nlevels
        probe.destroy()
        if thr > levels:
            continue
        h = bm.setup(k, bm.default_options(nu1=nu1, nu2=nu2, coarse_threshold=thr))
        for level in range(1, levels):
            sx, sy = h.level_shape(level)
            if level not in want:
                b = rand(sy, sx) - 0.5
                want[level] = (b, cycle(h, level, b, nu1, nu2))
            b, x = want[level]
            assert torch.equal(h.vcycle_from(level, b, torch.empty_like(b)), x), (thr, level)
        h.destroy()


@pytest.mark.parametrize("nx,ny", [(2, 2), (3, 3), (70, 2), (2, 300), (35, 3), (17, 16)])
def test_coarsest_solve_matches_dense(nx, ny):
    rng = np.random.default_rng(5)
    h = bm.setup(torch.from_numpy(10.0 ** rng.uniform(-1, 1, (ny, nx))).cuda())
    sx, sy = h.level_shape(0)
    st = h.level_stencil(0)
    n = sx * sy
    a = np.zeros((n, n))
    for j in range(sy):
        for i in range(sx):
            q = j * sx + i
            a[q, q] = st["C"][j, i]
            for name, di, dj in (("W", -1, 0), ("S", 0, -1), ("SW", -1, -1), ("NW", -1, 1)):
                if 0 <= i + di < sx and 0 <= j + dj < sy:
                    p = (j + dj) * sx + i + di
                    a[q, p] = a[p, q] = -st[name][j, i]
    b = rng.uniform(-1, 1, (sy, sx))
    x = h.vcycle_from(0, torch.from_numpy(b).cuda(), torch.empty((sy, sx), dtype=torch.float64, device="cuda"))
    h.destroy()
    want = np.linalg.solve(a, b.ravel())
    # forward error of a product with an inverse from a Cholesky factor, and of
    # the dense solve it is compared with: both n kappa eps at most
    tol = 2 * n * np.linalg.cond(a) * np.finfo(float).eps * np.linalg.norm(want)
    assert np.linalg.norm(x.cpu().numpy().ravel() - want) <= tol


@pytest.mark.parametrize("smoother", [bm.BMG_SMOOTH_XLINE, bm.BMG_SMOOTH_YLINE, bm.BMG_SMOOTH_ALTLINE])
@pytest.mark.parametrize("nx,ny", [(2, 9), (15, 16), (16, 15), (17, 33), (31, 300), (257, 47), (530, 560), (560, 530)])
def test_line_sweep_solves_its_last_lines(nx, ny, smoother):
    """Line lengths below, at and above one block of 16, several groups of
    separators, levels on both sides of the one-kernel step's size: after a
    sweep the lines of the colour solved last have zero residual.  A line's
    solve is backward stable up to a small factor, so its residual is within
    64 eps of the terms of its equations (the 9-point diagonal bound
    2 C |x|)."""
    rng = np.random.default_rng(nx + ny)
    h = bm.setup(torch.from_numpy(10.0 ** rng.uniform(-1, 1, (ny, nx))).cuda(),
                 bm.default_options(smoother=smoother))
    top = h.nlevels - 1
    for level in {top, max(1, top - 1)} if top else {0}:
        if level == 0:
            continue
        sx, sy = h.level_shape(level)
        b = torch.from_numpy(rng.uniform(-1, 1, (sy, sx))).cuda()
        x = torch.from_numpy(rng.uniform(-1, 1, (sy, sx))).cuda()
        scale = (2.0 * torch.from_numpy(h.level_stencil(level)["C"]).cuda()).max()
        for reverse in (False, True):
            h.op_relax(level, x, b, 1, reverse=reverse)
            r = h.op_residual(level, x, b, torch.empty_like(b)).abs()
            # forward: x-lines then y-lines, odd lines first; reverse: the whole turned
            rows = smoother == bm.BMG_SMOOTH_XLINE or (smoother == bm.BMG_SMOOTH_ALTLINE and reverse)
            first = 0 if reverse else 1      # 0-based index of the colour solved last
            last = r[first::2] if rows else r[:, first::2]
            if last.numel():
                assert last.max() <= 64 * np.finfo(float).eps * scale * x.abs().max() + 1e-15
    h.destroy()
