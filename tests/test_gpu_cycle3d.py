"""3D V-cycles against the oracle's, cycle by cycle: sides of both parities
(the finest restriction takes the residual of one colour only, whose points
change with the parities of the sides), one and several blocks along a row,
with and without pre- and post-smoothing.  The coarse correction carries a
residual's rounding, u |A| |x|, to at most cond(A) u of x, 10^-10 here; bound
as for the solves of test_gpu_parity3d, 1e-9 of max|x|."""
import numpy as np
import pytest

from oracle import boxmg3d_oracle as O3

torch = pytest.importorskip("torch")
import paper_1803_02481_gb300 as bm  # noqa: E402

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("nu1,nu2", [(2, 1), (1, 1), (3, 0), (0, 2)])
@pytest.mark.parametrize("nx,ny,nz", [(4, 4, 4), (5, 8, 7), (8, 5, 6), (16, 15, 9), (260, 5, 4), (33, 16, 17)])
def test_3d_cycles_match_oracle(nx, ny, nz, nu1, nu2):
    rng = np.random.default_rng(nx + ny * nz)
    k = 10.0 ** rng.uniform(-1, 1, (nz, ny, nx))
    b = rng.uniform(-1, 1, (nz, ny, nx))
    ho = O3.setup(k, nu1=nu1, nu2=nu2)
    for cycles in (1, 2, 3):
        x = np.asarray(O3.solve(ho, b, tol=1e-300, max_cycles=cycles).x).reshape(b.shape)
        h = bm.setup3(torch.from_numpy(k).cuda(), bm.default_options(nu1=nu1, nu2=nu2, max_cycles=cycles))
        got, info = h.solve(torch.from_numpy(b).cuda(), tol=1e-300, allow_noconv=True)
        h.destroy()
        assert info.cycles == cycles
        assert np.abs(got.cpu().numpy() - x).max() <= 1e-9 * np.abs(x).max(), cycles
