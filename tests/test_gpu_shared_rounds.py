"""The binary32 kernels with the Philox rounds split into the part all
particles of a step share (made 32 at a time per warp) and the particles' own:
step counts around the chunks of 32 pairs and of 8, 16 and 32 steps, slice
lengths that the chunks straddle, particle counts that leave part of a warp."""
import numpy as np
import pytest

from oracle import oracle
from paper_1912_09240_gb300 import build as b

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def L():
    b.build()
    from paper_1912_09240_gb300 import _lib
    return _lib


# binary32 paths against the binary64 oracle: the bound of the other per-particle tests
TOL = 2e-3


@pytest.mark.parametrize("d", [1, 2, 3, 4, 7, 11, 15, 16])
@pytest.mark.parametrize("steps", [1, 2, 7, 8, 9, 31, 33, 63, 64, 65, 66, 130])
@pytest.mark.parametrize("n", [1, 33, 5003])
def test_steps_around_the_chunks(L, d, steps, n):
    import torch
    rng = np.random.default_rng(n + d)
    x, y = rng.normal(-1, 0.3, (2, n)), rng.normal(0, 1, (2, d, n))
    kind = L.PR_MODEL_DOUBLE_WELL if d == 1 else L.PR_MODEL_DW_MULTI
    gx, gy = (torch.tensor(v, dtype=torch.float32, device="cuda") for v in (x, y))
    x, y = gx.double().cpu().numpy(), gy.double().cpu().numpy()
    L.pr_fine_propagate(L.Model(kind, d, 0.5, 3.0, 0.01), L.PR_F32, L.Rng((9 << 32) + 5, 3), gx, gy, False, gx, gy, n,
                        4, 2, steps, 1e-4)
    ids = np.unique(np.concatenate([np.arange(min(n, 40)), n - 1 - np.arange(min(n, 40))])).astype(np.uint32)
    xo, yo = oracle.fine_propagate(oracle.Model(1 if d == 1 else 2, d, 0.5, 3.0, 0.01), (9 << 32) + 5, x[:, ids],
                                   y[:, :, ids], 4, steps, 1e-4, problem=3, ids=ids)
    for got, want in ((gx.cpu().numpy()[:, ids], xo), (gy.cpu().numpy()[:, :, ids], yo)):
        assert np.all(np.abs(got - want) <= TOL * np.maximum(np.abs(want), 1.0))


@pytest.mark.parametrize("n", [1, 31, 127, 129, 1000])
@pytest.mark.parametrize("slices,steps,ckpt", [(1, 64, 64), (3, 22, 20), (5, 10, 4), (2, 66, 34), (40, 2, 30), (7, 62, 100)])
def test_adjoint_chunks_straddle_slices(L, n, slices, steps, ckpt):
    """The reverse walk (even steps and checkpoints) against the tangent-linear."""
    import torch
    rng = np.random.default_rng(7)
    x0, y0 = (torch.tensor(rng.normal(1, 0.3, n), dtype=torch.float32, device="cuda") for _ in range(2))
    m = (1.0, 1.0, 0.1)
    grad = torch.empty(n, 3, dtype=torch.float64, device="cuda")
    xb, yb = (torch.empty(n, dtype=torch.float64, device="cuda") for _ in range(2))
    xT = torch.empty(n, dtype=torch.float32, device="cuda")
    ws = torch.empty(L.pr_fine_adjoint_workspace(n, slices, steps, ckpt), dtype=torch.uint8, device="cuda")
    L.pr_fine_adjoint(L.Model(L.PR_MODEL_OU, 1, *m), L.Rng(11, 2), x0, y0, n, 3, slices, steps, 1e-4, ckpt, xT, None,
                      None, None, grad, xb, yb, ws)
    X, _, DX, _ = oracle.fine_tangent(oracle.Model(0, 1, *m), 11, x0.double().cpu().numpy(), y0.double().cpu().numpy(),
                                      3, slices, steps, 1e-4, problem=2)
    got = np.concatenate([grad.cpu().numpy(), xb.cpu().numpy()[:, None], yb.cpu().numpy()[:, None]], 1)
    scale = np.maximum(np.abs(DX), np.sqrt((DX ** 2).mean(0)))
    assert np.all(np.abs(got - DX) <= TOL * scale)
    assert np.all(np.abs(xT.cpu().numpy() - X) <= TOL * np.maximum(np.abs(X), 1.0))
    # and the ensemble sum with seeds is the contracted per-particle result
    seed = torch.tensor(rng.normal(0, 1, n), dtype=torch.float64, device="cuda")
    total = torch.empty(3, dtype=torch.float64, device="cuda")
    L.pr_fine_adjoint(L.Model(L.PR_MODEL_OU, 1, *m), L.Rng(11, 2), x0, y0, n, 3, slices, steps, 1e-4, ckpt, None, None,
                      seed, None, total, None, None, ws)
    want = (seed.cpu().numpy()[:, None] * DX[:, :3])
    assert np.all(np.abs(total.cpu().numpy() - want.sum(0)) <= TOL * np.abs(want).sum(0))


@pytest.mark.parametrize("d", [2, 3, 4, 7, 8, 12, 14, 15, 16])
@pytest.mark.parametrize("steps", [1, 3, 4, 6, 9, 34])
def test_small_launches_take_whole_blocks(d, steps):
    """The multi-component kernel draws whole blocks in launches of up to two warps per sub-partition and
    shared rounds beyond: the first particles of a large ensemble end where they do in a small one."""
    import torch
    from paper_1912_09240_gb300 import _lib as L
    from paper_1912_09240_gb300 import build as b
    b.build()
    n = 150_001                                   # two CTAs of 512 threads per SM
    g = torch.Generator(device="cuda").manual_seed(d)
    x = torch.randn(1, n, generator=g, device="cuda")
    y = torch.randn(1, d, n, generator=g, device="cuda")
    model = L.Model(L.PR_MODEL_DW_MULTI, d, 0.5, 1.0, 0.1)

    def run(k):
        xi, yi = (v[..., :k].clone(memory_format=torch.contiguous_format) for v in (x, y))   # (propagated in place)
        L.pr_fine_propagate(model, L.PR_F32, L.Rng(9, 2), xi, yi, False, xi, yi, k, 4, 1, steps, 1e-3)
        return xi, yi

    full = run(n)
    for k in (1, 63, 4097, 20_000):
        part = run(k)
        assert torch.equal(part[0], full[0][:, :k]) and torch.equal(part[1], full[1][:, :, :k])
