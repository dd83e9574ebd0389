"""Resampling where its fast forms end: weights on both sides of 2^-40 and 2^-9
(the fixed point's usual range), ranges of particles per CTA just below and
above the staged ones, particle counts around a CTA's outputs."""
import numpy as np
import pytest

from oracle import oracle
from paper_1912_09240_gb300 import build as b

pytestmark = pytest.mark.gpu


def _weights(kind, n):
    r = np.random.default_rng(n)
    w = {"uniform": lambda: np.full(n, 1.0),
         "spread": lambda: np.exp2(r.uniform(-60, 0, n)),
         "heavy": lambda: r.pareto(1.1, n),
         "sparse": lambda: (r.random(n) < 0.3) * r.random(n),
         "ramp": lambda: np.linspace(0.01, 2.0, n),
         "dyadic": lambda: np.exp2(-np.floor(r.uniform(5, 45, n)))}[kind]()
    return w / max(w.sum(), 1e-300) if kind != "dyadic" else w / 2.0 ** np.ceil(np.log2(w.sum()))


@pytest.mark.parametrize("kind", ["uniform", "spread", "heavy", "sparse", "ramp", "dyadic"])
@pytest.mark.parametrize("n", [2, 2047, 2049, 5003, 70001])
@pytest.mark.parametrize("mode", [0, 1])
def test_indices_and_weighted_cdf(kind, n, mode):
    import torch
    from paper_1912_09240_gb300 import _lib as L
    b.build()
    w = np.stack([_weights(kind, n), _weights(kind, n)[::-1]])
    x = np.random.default_rng(3).normal(0, 1, (2, n)).astype(np.float32)
    gw, gx = torch.tensor(w.copy(), device="cuda"), torch.tensor(x, device="cuda")
    idx = torch.empty(2, n, dtype=torch.int32, device="cuda")
    xo = torch.empty_like(gx)
    ws = torch.empty(L.pr_resample_workspace(n, 2), dtype=torch.uint8, device="cuda")
    L.pr_resample(L.PR_F32, 1, gx, None, False, gw, n, 2, 3, mode, L.Rng(5, 9), idx, xo, None, ws)
    want = oracle.resample(w, mode, 5, 3, problem=9)
    got = idx.cpu().numpy().view(np.uint32)
    np.testing.assert_array_equal(got, want)
    np.testing.assert_array_equal(xo.cpu().numpy(), np.take_along_axis(x, want.astype(np.int64), 1))
    cdf = torch.empty(2, 101, dtype=torch.float64, device="cuda")
    wr = torch.empty(L.pr_restrict_weighted_workspace(2, 100), dtype=torch.uint8, device="cuda")
    L.pr_restrict_weighted(L.PR_F32, gx, False, gw, n, 2, L.Grid(100, -3.0, 3.0), cdf, wr)
    np.testing.assert_array_equal(cdf.cpu().numpy(),
                                  oracle.restrict_weighted(x.astype(np.float64), w, oracle.Grid(100, -3.0, 3.0)))


@pytest.mark.parametrize("kind", ["sorted", "runs", "one"])
@pytest.mark.parametrize("n", [4866, 9730, 300007])
@pytest.mark.parametrize("mode", [0, 1])
def test_ranges_longer_than_the_staged_one(kind, n, mode):
    """A CTA's outputs spread over up to all particles: ascending weights of five decades, zero weights
    but for short runs, and one particle that holds nearly all; the ranges of the smaller sizes are just
    above one, two and four times the staged one."""
    import torch
    from paper_1912_09240_gb300 import _lib as L
    b.build()
    r = np.random.default_rng(n)
    w = {"sorted": lambda: np.sort(np.exp(2.5 * r.normal(0, 1, n))),
         "runs": lambda: ((np.arange(n) % 1000) < 3) * r.random(n) + (np.arange(n) == n - 1),
         "one": lambda: np.where(np.arange(n) == n // 3, 1e6, 1e-3 * r.random(n))}[kind]()
    w = np.stack([w / w.sum(), (w / w.sum())[::-1]])
    x = r.normal(0, 1, (2, n))
    gw, gx = torch.tensor(w.copy(), device="cuda"), torch.tensor(x, device="cuda")
    idx = torch.empty(2, n, dtype=torch.int32, device="cuda")
    xo = torch.empty_like(gx)
    ws = torch.empty(L.pr_resample_workspace(n, 2), dtype=torch.uint8, device="cuda")
    L.pr_resample(L.PR_F64, 1, gx, None, False, gw, n, 2, 3, mode, L.Rng(5, 9), idx, xo, None, ws)
    want = oracle.resample(w, mode, 5, 3, problem=9)
    np.testing.assert_array_equal(idx.cpu().numpy().view(np.uint32), want)
    np.testing.assert_array_equal(xo.cpu().numpy(), np.take_along_axis(x, want.astype(np.int64), 1))
