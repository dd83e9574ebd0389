"""The binary64 amplitudes of the chemical system, sqrt(max(., 0)): one step from
states that put their arguments at both ends of the square root's range and
beyond them (where the library's function takes over), at zero and below it."""
import ctypes
import subprocess

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


ROOTS = r"""
#include "pr_common.cuh"
__global__ void roots(const double* v, double* s, int n)
{
    const int i = blockIdx.x * blockDim.x + threadIdx.x;
    if (i < n) s[i] = pr::sqrt_clamped_f64(v[i]);
}
extern "C" int run(const void* v, void* s, int n)
{
    roots<<<(n + 255) / 256, 256>>>((const double*)v, (double*)s, n);
    return (int)cudaDeviceSynchronize();
}
"""


@pytest.mark.parametrize("kind", ["all exponents", "near one", "short significands", "squares", "edges"])
def test_root_is_correctly_rounded(tmp_path, kind):
    """The root itself against the host's, bit for bit: every exponent, significands with runs of zeros or
    ones at their end, squares and their neighbours, zeros, subnormals, negative numbers, infinity, NaN.
    Left out: 4^k (1 - 2^-53), whose root is 2^-55 of a unit from a midpoint."""
    from paper_1912_09240_gb300 import build as b
    n = 1 << 21
    r = np.random.default_rng(7)
    bits = r.integers(0, 0x7FF0 << 48, n, dtype=np.uint64)
    ones = (np.uint64(1) << r.integers(0, 53, n).astype(np.uint64)) - np.uint64(1)
    if kind == "near one":
        bits = (bits & np.uint64((1 << 52) - 1)) | (r.integers(1020, 1027, n).astype(np.uint64) << np.uint64(52))
    if kind == "short significands":
        bits = np.where(r.random(n) < 0.5, bits & ~ones, bits | ones)
    v = bits.view(np.float64)
    if kind == "squares":
        root = r.integers(1, 1 << 26, n).astype(np.float64) * np.exp2(r.integers(-30, 30, n))
        v = (root * root).view(np.int64) + r.integers(-2, 3, n)
        v = v.view(np.float64)
    if kind == "edges":
        v = np.array([0.0, -0.0, 5e-324, 2.2e-308, 2.0 ** -1022, np.nextafter(2.0 ** -1022, 0), -1.0, -5e-324, -1e308,
                      1.0, 2.0, 4.0, np.nextafter(1.0, 2), np.nextafter(2.0, 3), np.nextafter(2.0, 1), 1.7e308,
                      np.inf, -np.inf, np.nan, -np.nan])
    v = v[(v.view(np.uint64) & np.uint64((1 << 53) - 1)) != np.uint64((1 << 52) - 1)]
    (tmp_path / "r.cu").write_text(ROOTS)
    so = str(tmp_path / "r.so")
    subprocess.check_call([b.nvcc(), *b.ARCH, "-O3", "-std=c++17", "-shared", "-Xcompiler", "-fPIC", "-I", b.CSRC,
                           "-o", so, str(tmp_path / "r.cu")])
    gv = torch.tensor(v, device="cuda")
    gs = torch.empty_like(gv)
    torch.cuda.synchronize()
    assert ctypes.CDLL(so).run(ctypes.c_void_p(gv.data_ptr()), ctypes.c_void_p(gs.data_ptr()), v.size) == 0
    with np.errstate(invalid="ignore"):
        want = np.sqrt(np.fmax(v, 0.0))
    np.testing.assert_array_equal(gs.cpu().numpy(), np.where(want == 0.0, 0.0, want))
