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


@pytest.mark.parametrize("bins", [700, 1024])
def test_a_handle_holds_its_matrix_alone(bins):
    """Device memory of eight handles: the matrix each, rounded up to the allocator's 2 MiB."""
    import torch
    from paper_1912_09240_gb300 import _lib as L
    b.build()
    make = lambda: L.pr_coarse_create(L.Model(L.PR_MODEL_OU, 1, 0.5, 1.5, 0.7), L.Grid(bins, -3.0, 2.5), 0.1)
    L.pr_coarse_destroy(make())
    torch.cuda.synchronize()
    before = torch.cuda.mem_get_info()[0]
    handles = [make() for _ in range(8)]
    torch.cuda.synchronize()
    held = before - torch.cuda.mem_get_info()[0]
    for h in handles:
        L.pr_coarse_destroy(h)
    assert held <= 8 * (8 * bins * bins + (2 << 20))
