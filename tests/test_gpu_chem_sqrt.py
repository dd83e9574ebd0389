"""The binary64 amplitudes of the chemical system, sqrt(max(., 0)): one step from
states that put their arguments at both ends of the square root's range and
beyond them (where the library's function takes over), at zero and below it."""
import numpy as np
import pytest

torch = pytest.importorskip("torch")

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def L():
    from paper_1912_09240_gb300 import build as b
    b.build()
    from paper_1912_09240_gb300 import _lib
    return _lib


@pytest.mark.parametrize("scale", [0.0, 1e-300, 1e-40, 2.0 ** -96, 1e-20, 1e-3, 1.0, 1e3, 1e12, 1e29, 1e33, 1e60])
@pytest.mark.parametrize("sign", [1.0, -1.0])
def test_one_step_over_the_range_of_the_amplitudes(L, orc, scale, sign):
    """The tolerance is 16 units of 2^-53 of the absolute terms (eight operations
    in a term at most, and the two sides' normals)."""
    n, dt, tau, eps = 4096, 1e-3, 25.0, 2.5e-2
    big = scale > 1.0
    # the slow amplitude scales with x and y, the fast one with k0 where y is small
    rates = (0.0 if scale == 0.0 else min(scale, 1e3), 1.0, 3.0 if not big else 1.0, 1.0 if not big else 0.0, 2.0, 0.5)
    rng = np.random.default_rng(5)
    x = sign * scale * rng.uniform(0.5, 2.0, (1, n))
    y = sign * scale * rng.uniform(0.5, 2.0, (1, 1, n))
    gm, om = L.Model(4, 1, 0.0, 1.0, eps, tau, rates), orc.Model(4, 1, eps=eps, tau_x=tau, rates=rates)
    gx, gy = torch.tensor(x, device="cuda"), torch.tensor(y, device="cuda")
    L.pr_fine_propagate(gm, L.PR_F64, L.Rng(7, 3), gx, gy, False, gx, gy, n, 5, 1, 1, dt)
    torch.cuda.synchronize()
    ox, oy = orc.fine_propagate(om, 7, x, y, 5, 1, dt, problem=3)
    k, ya, xa = rates, np.abs(y[:, 0]), np.abs(x)
    ax, ay = dt / tau, dt / eps
    vx = ax * (k[4] * ya + k[5] * xa)
    poly = k[0] + (k[1] + k[2] + 2 * k[3]) * ya + (k[2] + 3 * k[3]) * ya ** 2 + k[3] * ya ** 3
    z = 7.0   # |normal| <= sqrt(2 ln 2^33) = 6.77
    u = 16 * 2.0 ** -53
    assert np.all(np.abs(gx.cpu().numpy() - ox) <= u * (xa + vx + z * np.sqrt(vx)))
    # the polynomial under the fast square root may cancel: an error d of it changes sqrt(v) by at most
    # d / sqrt(v), and by at most sqrt(d)
    y0 = y[:, 0]
    v = np.maximum(ay * (k[0] + (k[1] - k[2] + 2 * k[3]) * y0 + (k[2] - 3 * k[3]) * y0 ** 2 + k[3] * y0 ** 3), 0.0)
    d = u * ay * poly
    with np.errstate(divide="ignore", invalid="ignore"):
        amp = np.minimum(np.sqrt(d), np.where(v > 0, d / np.sqrt(v), np.inf))
    assert np.all(np.abs(gy.cpu().numpy()[:, 0] - oy[:, 0]) <= u * (ya + ay * poly + z * np.sqrt(v)) + z * amp)
