"""Binary64 restriction and matching bit for bit where the bin from binary32
arithmetic must give way to the exact comparisons: particles on the edges and a
few units either side, outside the grid, at the ends of the number range; grids
far from zero, tiny and huge ones."""
import numpy as np
import pytest

torch = pytest.importorskip("torch")

pytestmark = pytest.mark.gpu

GRIDS = [(1, 0.0, 1.0), (7, -1e-20, 3e-20), (64, -1e25, 1e25), (50, 0.0, 1e-290), (300, -3.0, 3.0), (333, 100.0, 101.0),
         (1500, 0.0, 600.0), (2000, -0.7, 5.3), (4096, 1e6, 1e6 + 1.0), (4096, -3.0, 3.0)]


def _particles(og, rng):
    e = og.edges()
    h = (og.hi - og.lo) / og.bins
    near = [e]
    for d in (1, 2, 3):
        up, down = e, e
        for _ in range(d):
            up, down = np.nextafter(up, np.inf), np.nextafter(down, -np.inf)
        near += [up, down]
    for rel in (2.0 ** -24, 2.0 ** -20, 2.0 ** -12, 1e-3, 0.02, 0.5):
        near += [e + rel * h, e - rel * h]
    far = [0.0, -0.0, 5e-324, -5e-324, 1e-310, 1e-40, -1e-40, 1e39, -1e39, 1e300, -1e300, og.lo - 1.0, og.hi + 1.0]
    return np.concatenate(near + [rng.uniform(og.lo - h, og.hi + h, 20_001), far])


@pytest.mark.parametrize("bins,lo,hi", GRIDS)
def test_bit_for_bit(orc, bins, lo, hi):
    from paper_1912_09240_gb300 import build as b
    b.build()
    from paper_1912_09240_gb300 import _lib as L
    og, rng = orc.Grid(bins, lo, hi), np.random.default_rng(bins)
    x = np.stack([_particles(og, rng), _particles(og, rng)])
    n = x.shape[1]
    counts, cp = orc.restrict(x, og)
    gx, grid = torch.tensor(x, device="cuda"), L.Grid(bins, lo, hi)
    gc = torch.empty(2, bins, dtype=torch.int32, device="cuda")
    gcdf = torch.empty(2, bins + 1, dtype=torch.float64, device="cuda")
    L.pr_restrict(L.PR_F64, gx, n, 2, grid, gc, gcdf)
    torch.cuda.synchronize()
    np.testing.assert_array_equal(gc.cpu().numpy(), counts.astype(np.int32))
    np.testing.assert_array_equal(gcdf.cpu().numpy(), cp)
    _, ct = orc.restrict(np.clip(x[::-1] * 0.9 + 0.05 * (lo + hi), lo, hi), og)
    out = torch.empty_like(gx)
    L.pr_match(L.PR_F64, gx, out, n, 2, grid, gcdf, torch.tensor(ct, device="cuda"))
    torch.cuda.synchronize()
    np.testing.assert_array_equal(out.cpu().numpy(), orc.match(x, og, cp, ct))
