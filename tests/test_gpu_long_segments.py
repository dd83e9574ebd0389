"""The quantile iterator where its monotone repair pools long stretches of
knots (advected, narrowed and noisy states against each other): bit for bit
the oracle's, and knots that are already in order left alone."""
import math

import numpy as np
import pytest

from oracle import oracle
from paper_1912_09240_gb300 import build as b

pytestmark = pytest.mark.gpu


def _gauss(bins, mean, sd):
    e = np.linspace(-3.0, 3.0, bins + 1)
    c = np.array([0.5 * (1 + math.erf((v - mean) / (sd * math.sqrt(2)))) for v in e])
    return (c - c[0]) / (c[-1] - c[0])


def _empirical(bins, mean, sd, n, seed):
    x = np.random.default_rng(seed).normal(mean, sd, (1, n))
    return oracle.restrict(x, oracle.Grid(bins, -3.0, 3.0))[1][0]


CASES = {
    "advected": lambda i: (_gauss(i, 0.9, 0.5), _gauss(i, -0.2, 0.4), _gauss(i, 0.1, 0.9)),
    "narrowed": lambda i: (_gauss(i, 0.0, 0.2), _gauss(i, 0.1, 0.9), _gauss(i, 0.0, 1.2)),
    "sampled": lambda i: (_gauss(i, 0.2, 0.6), _empirical(i, 0.25, 0.6, 500, 1), _empirical(i, 0.2, 0.62, 700, 2)),
    "noise": lambda i: (_gauss(i, 0.2, 0.6), _gauss(i, 0.2, 0.6),
                        np.clip(_gauss(i, 0.2, 0.6) * (1 - 1e-13), 0.0, 1.0)),
    "in_order": lambda i: (_gauss(i, 0.3, 0.5), _gauss(i, 0.0, 0.5), _gauss(i, 0.3, 0.5)),
}


@pytest.mark.parametrize("name", sorted(CASES))
@pytest.mark.parametrize("bins", [5, 63, 64, 288, 600, 1024])
@pytest.mark.parametrize("qmode", [0, 1])
def test_long_pooled_segments(name, bins, qmode):
    import torch
    from paper_1912_09240_gb300 import _lib as L
    b.build()
    t = [torch.tensor(v, dtype=torch.float64, device="cuda").reshape(1, -1) for v in CASES[name](bins)]
    for v in t:
        v[:, -1] = 1.0
    out = torch.empty_like(t[0])
    st = torch.empty(1, dtype=torch.int32, device="cuda")
    L.pr_iterate(L.PR_ITER_QUANTILE, qmode, L.Grid(bins, -3.0, 3.0), 1, *t, out, st)
    want = oracle.iterate(oracle.Grid(bins, -3.0, 3.0), *(v.cpu().numpy()[0] for v in t), oracle.ITER_QUANTILE, qmode)
    assert int(st.item()) == 0
    np.testing.assert_array_equal(out.cpu().numpy()[0], want)
    # the same states through the sweep, on one CTA and on clusters of 2, 4 and 8
    h = L.pr_coarse_create(L.Model(L.PR_MODEL_DOUBLE_WELL, 1, 0.5, 3.0, 0.01), L.Grid(bins, -3.0, 3.0), 0.1)
    try:
        got = []
        for ctas in (1, 2, 4, 8):
            L.pr_set_update_cluster(ctas)
            rho = torch.empty(3, bins + 1, dtype=torch.float64, device="cuda")
            L.pr_parareal_update(h, L.PR_ITER_QUANTILE, qmode, 2, t[0][0], torch.cat([t[1], t[0]]),
                                 torch.cat([t[2], t[1]]), rho, st)
            got.append(rho)
        assert all(torch.equal(got[0], g) for g in got[1:])
    finally:
        L.pr_set_update_cluster(8)
        L.pr_coarse_destroy(h)


@pytest.mark.parametrize("bins", [5, 64, 300, 512, 1024])
@pytest.mark.parametrize("n", [1, 200, 500])
def test_many_states_at_once(bins, n):
    """One, two and more states per SM (and as few as the shared memory allows): each as if alone."""
    import torch
    from paper_1912_09240_gb300 import _lib as L
    b.build()
    names = sorted(CASES)
    rows = [np.stack([np.asarray(CASES[names[k % len(names)]](bins)[f]) for k in range(n)]) for f in range(3)]
    t = [torch.tensor(r, device="cuda") for r in rows]
    for v in t:
        v[:, -1] = 1.0
    st = torch.empty(1, dtype=torch.int32, device="cuda")
    for iterator in (0, 1, 3):
        out = torch.empty_like(t[0])
        L.pr_iterate(iterator, 0, L.Grid(bins, -3.0, 3.0), n, *t, out, st)
        assert int(st.item()) == 0
        for k in range(min(n, len(names))):
            one = torch.empty(1, bins + 1, dtype=torch.float64, device="cuda")
            L.pr_iterate(iterator, 0, L.Grid(bins, -3.0, 3.0), 1, *(v[k:k + 1].clone() for v in t), one, st)
            same = out[k::len(names)]
            assert torch.equal(same, one.expand_as(same))
