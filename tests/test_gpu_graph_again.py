"""A graph-replayed solver started again: iteration 0 of the second run is
enqueued on the side streams while the graphs of the first run exist, and the
replay must come after it."""
import numpy as np
import pytest

torch = pytest.importorskip("torch")

import workloads

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("chunk", [0, 3, 5])
def test_runs_repeat(chunk):
    from paper_1912_09240_gb300 import build as b
    b.build()
    from paper_1912_09240_gb300 import _lib as L
    from paper_1912_09240_gb300.parareal import PararealSolver
    w = workloads.DOUBLE_WELL.scaled(N=200_000, K=17, T=17 * 0.01, dt=1e-4, bins=200)
    model = L.Model(w.kind, w.fast_dim, w.lam, w.beta, w.eps, w.tau_x)
    x0, y0 = workloads.initial_ensemble(w)
    x0, y0 = (torch.tensor(v, dtype=torch.float32, device="cuda") for v in (x0, y0))
    ref = None
    for graph in (False, True):
        s = PararealSolver(model, L.Grid(w.bins, w.lo, w.hi), w.N, w.K, w.steps, w.step_dt, rng=L.Rng(w.seed, 0),
                           chunk=chunk, graph=graph)
        for _ in range(3):
            s.set_initial(x0, y0)
            for _ in range(3):
                s.iterate()
            rho = s.rho.cpu().numpy()
            ref = rho if ref is None else ref
            np.testing.assert_array_equal(rho, ref)
        s.close()
