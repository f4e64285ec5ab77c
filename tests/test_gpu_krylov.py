"""The conjugate-gradient passes on the finest level: sides odd and even and
smaller than a warp, problems below and above one unit of work, alone and in
a batch, against a dense-operator CG run of the same recurrence."""
import numpy as np
import pytest

from oracle import boxmg_oracle as O

torch = pytest.importorskip("torch")
import paper_1803_02481_gb300 as bm  # noqa: E402

pytestmark = pytest.mark.gpu


def problem(nx, ny, scale=1.0):
    rng = np.random.default_rng(nx + 7 * ny)
    return 10.0 ** rng.uniform(-1, 1, (ny, nx)), scale * rng.uniform(-1, 1, (ny, nx))


@pytest.mark.parametrize("prec", [bm.BMG_FP64, bm.BMG_FP32_REFINE])
@pytest.mark.parametrize("nx,ny", [(2, 3), (5, 4), (31, 33), (64, 64), (127, 63), (513, 40), (1026, 31)])
def test_pcg_solves_every_shape(nx, ny, prec):
    """The iterate meets the stop test with the oracle's operator.  The test
    uses the recursive residual; recursion and evaluation differ by rounding,
    at most about 30 eps |A||x| / |b| here, far below the 5 % allowed."""
    k, b = problem(nx, ny)
    h = bm.setup(torch.from_numpy(k).cuda(),
                 bm.default_options(nu1=1, nu2=1, solver=bm.BMG_SOLVER_PCG, precision=prec, max_cycles=100))
    x, info = h.solve(torch.from_numpy(b).cuda(), tol=1e-9)
    h.destroy()
    r = O.residual(O.assemble_fv5(k), x.cpu().numpy(), b)
    assert np.linalg.norm(r) <= 1.05e-9 * np.linalg.norm(b)


@pytest.mark.parametrize("scale", [1e-60, 1.0, 1e60])
def test_pcg_fp32_is_scale_free(scale):
    """Powers of ten far outside FP32's range in the right-hand side: the casts
    see r / ||r||, so the iteration counts agree and the iterates scale."""
    k, b = problem(95, 61)
    opts = bm.default_options(nu1=1, nu2=1, solver=bm.BMG_SOLVER_PCG, precision=bm.BMG_FP32_REFINE)
    h = bm.setup(torch.from_numpy(k).cuda(), opts)
    x1, i1 = h.solve(torch.from_numpy(b).cuda(), tol=1e-9)
    xs, i2 = h.solve(torch.from_numpy(scale * b).cuda(), tol=1e-9)
    h.destroy()
    assert i1.cycles == i2.cycles
    # scaling by a power of ten rounds b once: relative changes of a few eps,
    # and the solves agree to their tolerance
    assert torch.linalg.norm(xs / scale - x1) <= 1e-8 * torch.linalg.norm(x1)


@pytest.mark.parametrize("nu1,nu2,solver", [(1, 1, bm.BMG_SOLVER_PCG), (2, 1, bm.BMG_SOLVER_VCYCLE),
                                            (2, 2, bm.BMG_SOLVER_PCG), (3, 1, bm.BMG_SOLVER_VCYCLE)])
def test_batch_of_every_side_matches_single_solves(nu1, nu2, solver):
    """Sides 3 to 511 in one batch, with the fused legs (one or two pre-, one
    post-sweep) and without: every problem meets the stop test, a zero
    right-hand side gives a zero solution, and a second solve repeats the
    first bit for bit."""
    sides = [3, 7, 15, 31, 63, 63, 127, 255, 511]
    data = [problem(n, n) for n in sides]
    data[4] = (data[4][0], np.zeros((63, 63)))
    ks = [torch.from_numpy(k).cuda() for k, _ in data]
    bs = [torch.from_numpy(b).cuda() for _, b in data]
    batch = bm.Batch(ks, bm.default_options(nu1=nu1, nu2=nu2, solver=solver, max_cycles=200))
    xs = [torch.ones_like(b) if b.any() else torch.zeros_like(b) for b in bs]
    again = [x.clone() for x in xs]
    infos = batch.solve(bs, xs, tol=1e-8)
    batch.solve(bs, again, tol=1e-8)
    batch.destroy()
    for (k, b), x, y, info in zip(data, xs, again, infos):
        assert torch.equal(x, y)
        if not b.any():
            assert info.cycles == 0 and not x.any()
            continue
        r = O.residual(O.assemble_fv5(k), x.cpu().numpy(), b)
        assert np.linalg.norm(r) <= 1.05e-8 * np.linalg.norm(b)
