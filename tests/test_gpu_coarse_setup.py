"""pr_coarse_create at the edges of its tiles: grids around multiples of the
warp, of the 64-column tile and of the rows a CTA takes, few and many
squarings (the band of the squared matrix narrower and wider than the grid)."""
import numpy as np
import pytest

from oracle import oracle
from paper_1912_09240_gb300 import build as b

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("bins", [3, 17, 31, 33, 63, 65, 129, 333, 513, 601, 1300])
@pytest.mark.parametrize("kind,dT", [(oracle.MODEL_OU, 1e-4), (oracle.MODEL_DOUBLE_WELL, 0.1),
                                     (oracle.MODEL_ADVECTION, 0.2)])
def test_propagator_matches_oracle(bins, kind, dT):
    import torch
    from paper_1912_09240_gb300 import _lib as L
    b.build()
    par = dict(lam=0.5, beta=1.5, eps=0.7)
    h = L.pr_coarse_create(L.Model(kind, 1, **par), L.Grid(bins, -3.0, 2.5), dT)
    P = torch.empty(bins, bins, dtype=torch.float64, device="cuda")
    L.pr_coarse_matrix(h, P)
    torch.cuda.synchronize()
    L.pr_coarse_destroy(h)
    want = oracle.coarse_propagator(oracle.Model(kind, 1, **par), oracle.Grid(bins, -3.0, 2.5), dT)
    # the bound of the other propagator tests: both exponentials within 1e-12
    assert np.max(np.abs(P.cpu().numpy() - want)) <= 1e-12
