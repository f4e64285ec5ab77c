"""Options of the batched solver: the r/C interpolation term is left out of
the batched cycle on every level, those of the coarse kernel included."""
import pytest

torch = pytest.importorskip("torch")
import paper_1803_02481_gb300 as bm  # noqa: E402

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("nu1,nu2", [(2, 1), (2, 2)])
def test_batch_cycles_leave_out_the_residual_term(nu1, nu2):
    """Values and cycle counts do not depend on interp_residual_term."""
    g = torch.Generator(device="cuda")
    g.manual_seed(3)
    sides = [7, 15, 31, 63, 127]
    ks = [10.0 ** (2.0 * torch.rand((n, n), generator=g, device="cuda", dtype=torch.float64) - 1.0) for n in sides]
    bs = [torch.rand((n, n), generator=g, device="cuda", dtype=torch.float64) - 0.5 for n in sides]
    out = []
    for term in (0, 1):
        batch = bm.Batch(ks, bm.default_options(nu1=nu1, nu2=nu2, interp_residual_term=term))
        xs = [torch.zeros_like(b) for b in bs]
        infos = batch.solve(bs, xs, tol=1e-9)
        batch.destroy()
        out.append((xs, [i.cycles for i in infos]))
    assert out[0][1] == out[1][1]
    for n, x0, x1 in zip(sides, out[0][0], out[1][0]):
        assert torch.equal(x0, x1), n
