"""3D setup at the edges of its blocks: assembly tiles of 32 x 8 cells and
columns of 16 layers, Galerkin blocks of 64 coarse points, sides of both
parities, a wide contrast (divisions by very different denominators).  The
assembled level is exact and the weights are within 1e-12, as in the setup
test of test_gpu_parity3d.  A Galerkin entry is a sum of at most 27 inner sums
of at most 27 products on either side, so GPU and oracle (on the same P)
differ by at most 2 (27 + 27 + 2) u times the entry of |P|^T |A| |P|; on 10^10
contrasts that is far more than 1e-12 of the diagonal."""
import numpy as np
import pytest

from oracle import boxmg3d_oracle as O3

torch = pytest.importorskip("torch")
import paper_1803_02481_gb300 as bm  # noqa: E402
from tests.test_gpu_parity3d import interp_to_csr, stencil_to_csr  # noqa: E402

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("decades", [1.0, 5.0])
@pytest.mark.parametrize("nx,ny,nz", [(32, 8, 16), (33, 9, 17), (31, 7, 15), (4, 16, 33), (130, 4, 5), (65, 10, 4)])
def test_3d_setup_matches_oracle_at_block_edges(nx, ny, nz, decades):
    k = 10.0 ** np.random.default_rng(nx * ny + nz).uniform(-decades, decades, (nz, ny, nx))
    h = bm.setup3(torch.from_numpy(k).cuda())
    ho = O3.setup(k)
    top = h.nlevels - 1
    assert abs(stencil_to_csr(h.level_stencil(top), (nx, ny, nz)) - ho.levels[-1].a).max() == 0
    for level in range(top, 0, -1):
        shape, coarse = h.level_shape(level), h.level_shape(level - 1)
        a = stencil_to_csr(h.level_stencil(level), shape)
        p = interp_to_csr(h.level_interp(level), shape)
        assert abs(p - O3.interpolation(a, shape)).max() <= 1e-12
        err = abs(stencil_to_csr(h.level_stencil(level - 1), coarse) - O3.galerkin(a, p, coarse))
        bound = 2 * 56 * 2.0 ** -53 * (abs(p).T @ abs(a) @ abs(p))
        assert (err - bound).max() <= 0
    h.destroy()
