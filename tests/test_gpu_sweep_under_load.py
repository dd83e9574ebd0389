"""The clusters that run the serial sweep and the coarse step give the bits of
one CTA while fine kernels share the chip with them, so that the CTAs of a
cluster start at different times and drift apart."""
import numpy as np
import pytest

torch = pytest.importorskip("torch")

from oracle import oracle
from paper_1912_09240_gb300 import build as b

pytestmark = pytest.mark.gpu

K = 17


@pytest.fixture(scope="module")
def L():
    b.build()
    from paper_1912_09240_gb300 import _lib
    yield _lib
    _lib.pr_set_update_cluster(8)


class Load:
    """Fine kernels on a stream of their own, short CTAs with a matching table beside the sweep's."""

    def __init__(self, L, n=1 << 18, slices=2):
        self.L, self.n, self.slices = L, n, slices
        self.stream = torch.cuda.Stream()
        self.x = torch.randn(slices, n, device="cuda")
        self.y = torch.randn(slices, 1, n, device="cuda")
        self.out = torch.empty_like(self.x), torch.empty_like(self.y)
        self.grid = L.Grid(256, -4.0, 4.0)
        self.cdf = torch.linspace(0, 1, 257, dtype=torch.float64, device="cuda").repeat(slices, 1)
        torch.cuda.synchronize()

    def __call__(self, times):
        m = self.L.Model(self.L.PR_MODEL_DOUBLE_WELL, 1, 0.5, 1.0, 0.1)
        with torch.cuda.stream(self.stream):
            for _ in range(times):
                self.L.pr_fine_propagate(m, self.L.PR_F32, self.L.Rng(1, 0), self.x, self.y, False, *self.out, self.n,
                                         0, self.slices, 100, 1e-3, self.grid, self.cdf, self.cdf)


def _states(bins, n, seed):
    x = np.random.default_rng(seed).normal(0.0, 0.7, (n, 3000)) + np.linspace(-0.5, 0.5, n)[:, None]
    return torch.tensor(oracle.restrict(x, oracle.Grid(bins, -3.0, 3.0))[1], device="cuda")


@pytest.mark.parametrize("bins", [64, 200, 256, 257, 512])
@pytest.mark.parametrize("iterator", [0, 1, 2, 3, 4])
def test_sweep(L, bins, iterator):
    load = Load(L)
    h = L.pr_coarse_create(L.Model(L.PR_MODEL_DOUBLE_WELL, 1, 0.5, 3.0, 0.01), L.Grid(bins, -3.0, 3.0), 0.05)
    c0, fs, cs = _states(bins, 1, 1), _states(bins, K, 2), _states(bins, K, 3)
    st = torch.zeros(1, dtype=torch.int32, device="cuda")
    for qmode in ((0, 1) if iterator == 0 else (0,)):
        def sweep(ctas, out):
            L.pr_set_update_cluster(ctas)
            L.pr_parareal_update(h, iterator, qmode, K, c0[0], fs, cs, out, st)

        want = torch.empty(K + 1, bins + 1, dtype=torch.float64, device="cuda")
        sweep(1, want)
        got = torch.zeros(50, K + 1, bins + 1, dtype=torch.float64, device="cuda")
        torch.cuda.synchronize()
        for r in range(50):
            load(3)
            sweep((8, 4, 8, 2)[r % 4], got[r])
        torch.cuda.synchronize()
        assert int(st.item()) == 0
        assert all(torch.equal(want, g) for g in got)
    L.pr_coarse_destroy(h)


@pytest.mark.parametrize("bins", [64, 256, 257, 600])
def test_coarse_step(L, bins):
    load = Load(L)
    h = L.pr_coarse_create(L.Model(L.PR_MODEL_DOUBLE_WELL, 1, 0.5, 3.0, 0.01), L.Grid(bins, -3.0, 3.0), 0.05)
    states = _states(bins, 400, 4)
    want = torch.empty_like(states)
    L.pr_coarse_fp(h, states, want, 400)        # one CTA each
    torch.cuda.synchronize()
    for n in (1, 19, 38, 76, 152):              # clusters of 8, 8, 8, 4 and 2 CTAs
        got = torch.zeros(20, n, bins + 1, dtype=torch.float64, device="cuda")
        torch.cuda.synchronize()
        for r in range(20):
            load(2)
            L.pr_coarse_fp(h, states[:n].contiguous(), got[r], n)
        torch.cuda.synchronize()
        assert all(torch.equal(want[:n], g) for g in got)
    L.pr_coarse_destroy(h)
