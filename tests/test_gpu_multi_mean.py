"""The mean of the fast components in the binary64 kernel, without a division
where the quotient's exponent allows: every dimension, and sums of any scale."""
import numpy as np
import pytest

torch = pytest.importorskip("torch")

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("d", [2, 3, 5, 7, 11, 13, 16])
@pytest.mark.parametrize("scale", [0.0, 1e-305, 1e-280, 1.0, 1e20, 1e280])
def test_one_step(orc, d, scale):
    """From x = 0 one step moves x by dt (1 - lambda) mean(y) or so and the noise; 16 units of
    2^-53 of these terms (d additions, five products, the two sides' normals)."""
    from paper_1912_09240_gb300 import build as b
    b.build()
    from paper_1912_09240_gb300 import _lib as L
    n, dt, lam, beta, eps = 1000, 1e-4, 0.5, 3.0, 1e-3
    rng = np.random.default_rng(d)
    x, y = np.zeros((1, n)), scale * rng.uniform(0.5, 2.0, (1, d, n))
    gm = L.Model(L.PR_MODEL_DW_MULTI, d, lam, beta, eps)
    gx, gy = torch.tensor(x, device="cuda"), torch.tensor(y, device="cuda")
    L.pr_fine_propagate(gm, L.PR_F64, L.Rng(7, 3), gx, gy, False, gx, gy, n, 2, 1, 1, dt)
    torch.cuda.synchronize()
    ox, oy = orc.fine_propagate(orc.Model(L.PR_MODEL_DW_MULTI, d, lam, beta, eps), 7, x, y, 2, 1, dt, problem=3)
    u = 16 * 2.0 ** -53
    noise = 7.0 * np.sqrt(2.0 * dt / beta)
    assert np.all(np.abs(gx.cpu().numpy() - ox) <= u * (dt * y.mean(axis=1) + noise))
    assert np.all(np.abs(gy.cpu().numpy() - oy) <= u * (y * (1 + dt / eps) + 7.0 * np.sqrt(2.0 * dt / eps)))
