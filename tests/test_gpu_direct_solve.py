"""Solves that are one coarsest solve and nothing else (a side of at most
three points has one level) on nearly singular operators: three walls without
flux and a fourth with a small exchange coefficient.  Substitution with the
Cholesky factor is backward stable: |b - A x| <= (3 n + 1) u |L||L^T||x|
elementwise (Higham, Accuracy and Stability of Numerical Algorithms, theorem
10.4), whatever the condition; the product with an inverse is not."""
import numpy as np
import pytest

from oracle import boxmg3d_oracle as O3
from oracle import boxmg_oracle as O

torch = pytest.importorskip("torch")
import paper_1803_02481_gb300 as bm  # noqa: E402

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("beta", [1.0, 1e-4, 1e-8])
@pytest.mark.parametrize("nx,ny", [(3, 40), (40, 3), (2, 70), (3, 3)])
def test_one_level_solve_is_backward_stable(nx, ny, beta):
    rng = np.random.default_rng(nx + ny)
    k = 10.0 ** rng.uniform(-0.5, 0.5, (ny, nx))
    bc = (0.0, 0.0, 0.0, beta) if ny > nx else (0.0, beta, 0.0, 0.0)
    b = rng.uniform(-1, 1, (ny, nx))
    b -= b.mean()
    st = O.assemble_fv5(k, bc=bc)
    h = bm.setup(torch.from_numpy(k).cuda(), bm.default_options(bc_beta=bc, max_cycles=1))
    assert h.nlevels == 1
    bt = torch.from_numpy(b).cuda()
    xs = [h.solve(bt, tol=1e-300, allow_noconv=True)[0], h.vcycle_from(0, bt, torch.empty_like(bt))]
    h.destroy()
    n = nx * ny
    lo = np.abs(O.cholesky(O.stencil_to_csr(st).toarray()))
    for x in (x.cpu().numpy() for x in xs):
        # the solve's bound, and 7 u of the terms for evaluating the residual
        terms = (lo @ (lo.T @ np.abs(x.ravel()))).reshape(b.shape) + np.abs(b)
        assert (np.abs(O.residual(st, x, b)) <= (3 * n + 8) * 2.0 ** -53 * terms).all()


@pytest.mark.parametrize("kw", [{}, {"coarse_ctas": 2}, {"smoother": bm.BMG_SMOOTH_ALTLINE},
                                {"precision": bm.BMG_FP32_REFINE}, {"solver": bm.BMG_SOLVER_PCG, "nu1": 1}])
@pytest.mark.parametrize("nx,ny", [(31, 31), (70, 9), (9, 150)])
def test_cycles_with_a_substituted_coarsest_solve(nx, ny, kw):
    """The same walls on several levels (9 to 37 coarsest unknowns, too near to
    singular for the inverse), in every kernel of the coarsest levels.  The
    stop test's residual and the oracle's differ by rounding, 20 u |A||x| / |b|
    < 1e-14, against the 5 % allowed; with PCG by the recursion too."""
    rng = np.random.default_rng(nx + ny)
    k = 10.0 ** rng.uniform(-0.5, 0.5, (ny, nx))
    bc = (0.0, 0.0, 0.0, 1e-6)
    b = rng.uniform(-1, 1, (ny, nx))
    b -= b.mean()
    h = bm.setup(torch.from_numpy(k).cuda(), bm.default_options(bc_beta=bc, **kw))
    assert h.nlevels > 1
    a = h.coarse_factor()
    a = a @ a.T
    assert (np.diag(a) * np.diag(np.linalg.inv(a))).max() > 1e3
    x, _ = h.solve(torch.from_numpy(b).cuda(), tol=1e-10)
    h.destroy()
    r = O.residual(O.assemble_fv5(k, bc=bc), x.cpu().numpy(), b)
    assert np.linalg.norm(r) <= 1.05e-10 * np.linalg.norm(b)


@pytest.mark.parametrize("prec,tol", [(bm.BMG_FP64, 1e-13), (bm.BMG_FP32_REFINE, 1e-6)])
@pytest.mark.parametrize("nx,ny,nz", [(3, 6, 5), (2, 2, 2), (17, 3, 4)])
def test_one_level_solve_3d(nx, ny, nz, prec, tol):
    """One cycle is the solution (in FP32 to its rounding, 6e-8 of the entries
    of a well conditioned system)."""
    rng = np.random.default_rng(nx * ny * nz)
    b = rng.uniform(-1, 1, (nz, ny, nx))
    k = 10.0 ** rng.uniform(-0.5, 0.5, (nz, ny, nx))
    h = bm.setup3(torch.from_numpy(k).cuda(), bm.default_options(max_cycles=1, precision=prec))
    assert h.nlevels == 1
    x, _ = h.solve(torch.from_numpy(b).cuda(), tol=0.0, allow_noconv=True)
    h.destroy()
    want = np.linalg.solve(O3.assemble_fv7(k).toarray(), b.ravel())
    assert np.abs(x.cpu().numpy().ravel() - want).max() <= tol * np.abs(want).max()


@pytest.mark.parametrize("kw", [{}, {"precision": bm.BMG_FP32_REFINE}, {"solver": bm.BMG_SOLVER_PCG, "nu1": 1},
                                {"solver": bm.BMG_SOLVER_PCG, "nu1": 1, "precision": bm.BMG_FP32_REFINE}])
@pytest.mark.parametrize("nx,ny", [(500, 31), (31, 500), (3, 33), (3, 32)])
def test_sub_cycle_with_nothing_to_stage(nx, ny, kw):
    """A coarsest level of more than 96 unknowns (186, 99) with no other level
    in the sub-cycle, and one of exactly 96: the stop test is met.  Bound as
    above."""
    rng = np.random.default_rng(nx + ny)
    k = 10.0 ** rng.uniform(-0.5, 0.5, (ny, nx))
    b = rng.uniform(-1, 1, (ny, nx))
    h = bm.setup(torch.from_numpy(k).cuda(), bm.default_options(**kw))
    x, info = h.solve(torch.from_numpy(b).cuda(), tol=1e-10)
    h.destroy()
    assert info.threshold == 1
    r = O.residual(O.assemble_fv5(k), x.cpu().numpy(), b)
    assert np.linalg.norm(r) <= 1.05e-10 * np.linalg.norm(b)
