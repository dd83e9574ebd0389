"""The ends of the number range in the coarse step and the iterators.  Their
comparisons run on the integer units and in binary32: with infinities and NaNs
they decide as the floating comparisons do, whatever the sign bit of a NaN, so
that a NaN reaches the caller's status, and on grids whose knots are below
binary32's range as the binary64 products do."""
import math

import numpy as np
import pytest

torch = pytest.importorskip("torch")

from oracle import oracle
from paper_1912_09240_gb300 import build as b

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def L():
    b.build()
    from paper_1912_09240_gb300 import _lib
    return _lib


def _gauss(bins, mean, sd):
    e = np.linspace(-3.0, 3.0, bins + 1)
    c = np.array([0.5 * (1 + math.erf((v - mean) / (sd * math.sqrt(2)))) for v in e])
    return (c - c[0]) / (c[-1] - c[0])


def _iterate(L, grid, qmode, rows):
    t = [torch.tensor(v, dtype=torch.float64, device="cuda").reshape(1, -1) for v in rows]
    out, st = torch.empty_like(t[0]), torch.zeros(1, dtype=torch.int32, device="cuda")
    L.pr_iterate(L.PR_ITER_QUANTILE, qmode, grid, 1, *t, out, st)
    return out.cpu().numpy()[0], int(st.item())


@pytest.mark.parametrize("lo", [-1.7e308, 1.6e308])
@pytest.mark.parametrize("qmode", [0, 1])
@pytest.mark.parametrize("bins", [40, 300])
def test_pooled_sums_beyond_the_number_range(L, lo, qmode, bins):
    """Edges near the end of the number range: the sums of pooled knots are infinite and the
    interpolation between them not a number, which the result must show where the oracle's does."""
    hi = lo + 1e299
    rows = (_gauss(bins, 0.9, 0.5), _gauss(bins, -0.2, 0.4), _gauss(bins, 0.1, 0.9))
    got, _ = _iterate(L, L.Grid(bins, lo, hi), qmode, rows)
    with np.errstate(all="ignore"):
        want = oracle.iterate(oracle.Grid(bins, lo, hi), *rows, oracle.ITER_QUANTILE, qmode)
    # (not the values: segments are pooled apart, and an infinite sum would reach across them)
    assert np.isnan(got).any() == np.isnan(want).any()


@pytest.mark.parametrize("sign", [1.0, -1.0])
@pytest.mark.parametrize("row", [0, 1, 2])
def test_nan_in_a_cdf(L, sign, row):
    """A NaN level interpolates to NaN or drops out of the order; the status says so in any case."""
    rows = [_gauss(64, m, 0.5) for m in (0.2, 0.0, 0.1)]
    rows[row][10] = math.copysign(math.nan, sign)
    got, st = _iterate(L, L.Grid(64, -3.0, 3.0), 0, rows)
    assert st != 0
    assert np.all(np.isnan(got) | ((got >= 0.0) & (got <= 1.0)))


@pytest.mark.parametrize("bins", [40, 200, 300])
@pytest.mark.parametrize("last", [math.inf, -math.inf, math.nan, -math.nan])
def test_coarse_step_of_what_is_no_cdf(L, bins, last):
    """The last entry of the CDF, and so the last mass, infinite or NaN: rows whose sum is not above
    the tail's bound (a NaN among them) count as empty, and the quotient inf / inf as one."""
    grid = L.Grid(bins, -3.0, 3.0)
    h = L.pr_coarse_create(L.Model(L.PR_MODEL_DOUBLE_WELL, 1, 0.5, 3.0, 0.01), grid, 0.05)
    P = torch.empty(bins, bins, dtype=torch.float64, device="cuda")
    L.pr_coarse_matrix(h, P)
    c = _gauss(bins, 0.2, 0.5)
    c[-1] = last
    t = torch.tensor(c, dtype=torch.float64, device="cuda").reshape(1, -1)
    out = torch.empty_like(t)
    L.pr_coarse_fp(h, t, out, 1)
    got = out.cpu().numpy()[0]
    L.pr_coarse_destroy(h)
    want = np.zeros(bins + 1)
    full = P.cpu().numpy()[:, -1] * last == np.inf
    if full.any():
        want[1 + np.argmax(full):] = 1.0
    want[-1] = 1.0
    np.testing.assert_array_equal(got, want)


@pytest.mark.parametrize("scale", [1e-30, 1e-36, 1e-40, 1e-42, 1e-44, 1e-46, 1e-60, 1e-300])
@pytest.mark.parametrize("qmode", [0, 1])
@pytest.mark.parametrize("bins", [64, 300, 700])
def test_pooled_knots_below_the_range_of_binary32(L, scale, qmode, bins):
    """Bit for bit the oracle's pooling, as on grids of ordinary size."""
    lo, hi = -3.0 * scale, 3.0 * scale
    for rows in ((_gauss(bins, 0.9, 0.5), _gauss(bins, -0.2, 0.4), _gauss(bins, 0.1, 0.9)),
                 (_gauss(bins, 0.0, 0.2), _gauss(bins, 0.1, 0.9), _gauss(bins, 0.0, 1.2))):
        got, st = _iterate(L, L.Grid(bins, lo, hi), qmode, rows)
        assert st == 0
        want = oracle.iterate(oracle.Grid(bins, lo, hi), *rows, oracle.ITER_QUANTILE, qmode)
        np.testing.assert_array_equal(got, want)
