"""2D setup at the edges of its blocks: assembly tiles of 32 x 8 cells, weight
tiles of 32 x 8 coarse indices, sides of both parities, with and without
anisotropy, and a jump of 10^35 > 2^100 (quotients outside the range of the
shared reciprocals).  Every level is compared with the oracle's operations on
the GPU's own operator: the assembled level is exact, the weights are within
1e-12 as in test_gpu_parity.  A weight is a quotient of sums of non-negative
terms by a denominator formed in the same order on both sides, so GPU and
oracle differ by at most 8 u of it; a Galerkin entry is a sum of at most 9
inner sums of at most 9 products, hence at most (2 (9 + 9 + 2) + 2 8 + 8) u
times the entry of |P|^T |A| |P|."""
import numpy as np
import pytest

from oracle import boxmg_oracle as O
from tests.parity_helpers import interp_planes, nine_from_five

torch = pytest.importorskip("torch")
import paper_1803_02481_gb300 as bm  # noqa: E402

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("jump,r,aspect", [(1.0, 1.0, 1.0), (1e-35, 1.0, 1.0), (1.0, 4.0, 0.5)])
@pytest.mark.parametrize("nx,ny", [(2, 2), (3, 9), (32, 8), (31, 7), (33, 9), (63, 15), (64, 16), (65, 17), (66, 18),
                                   (130, 35), (7, 200)])
def test_setup_matches_oracle_at_block_edges(nx, ny, jump, r, aspect):
    k = 10.0 ** np.random.default_rng(nx * ny).uniform(-1.0, 1.0, (ny, nx))
    k[:, nx // 2:] *= jump
    h = bm.setup(torch.from_numpy(k).cuda(), bm.default_options(aniso_r=r, cell_aspect=aspect))
    top = h.nlevels - 1
    fine = O.assemble_fv5(k, r, aspect)
    for d in ("C", "W", "S"):
        assert np.array_equal(h.level_stencil(top)[d], fine[d]), d
    for level in range(top, 0, -1):
        st = nine_from_five(h.level_stencil(level))
        sy, sx = st["C"].shape
        p = O.interpolation(st)
        planes, valid = interp_planes(p, sx, sy)
        got = h.level_interp(level)
        for q, name in enumerate(("XW", "XE", "YS", "YN", "CSW", "CSE", "CNW", "CNE")):
            assert np.abs(got[name] - planes[q])[valid[q]].max(initial=0.0) <= 1e-12, (level, name)
        want = O.stencil_to_csr(O.galerkin(st, p))
        coarse = O.stencil_to_csr(nine_from_five(h.level_stencil(level - 1)))
        bound = 64 * 2.0 ** -53 * (abs(p).T @ abs(O.stencil_to_csr(st)) @ abs(p))
        assert (abs(coarse - want) - bound).max() <= 0, level
    h.destroy()
