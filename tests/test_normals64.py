"""Binary64 normals from integer arithmetic (csrc/normal64.cuh, normal_tables.py).

On the CPU the header is compiled for the host and compared with long double
arithmetic; on the GPU one Euler-Maruyama step from the origin gives the
normals themselves, and the two placements of the tables give the same bits.
"""
import ctypes
import os
import subprocess

import numpy as np
import pytest

from paper_1912_09240_gb300 import build as b, normal_tables

SRC = r"""
#include <cstdint>
#define PR_TABLE_STORAGE alignas(16) static const
#include "normal_tables.h"
#include "normal64.cuh"
extern "C" void normals(const uint32_t* w0, const uint32_t* w1, long n, uint64_t* z0, uint64_t* z1)
{
    const pr::NormalTables t = pr::normal_tables_at(pr::kNormalTables);
    for (long i = 0; i < n; ++i) pr::box_muller_fixed(w0[i], w1[i], t, z0[i], z1[i]);
}
"""


def _words(kind):
    k = np.arange(1 << 16, dtype=np.uint64)
    if kind == "random":
        r = np.random.default_rng(0)
        return r.integers(0, 1 << 32, (2, 1 << 18), dtype=np.uint64).astype(np.uint32)
    ends = {"low": k, "high": (1 << 23) - 1 - k, "half": (1 << 22) - (1 << 15) + k,
            "segments": (k % 46 << 17) + (k // 46) - 700}[kind] % (1 << 23)
    r = np.random.default_rng(1).integers(0, 1 << 9, (2, 1 << 16), dtype=np.uint64)
    # ends of the range in the radius word, and the same in the angle word
    return np.stack([(ends << 9) | r[0], (ends[::-1] << 9) | r[1]]).astype(np.uint32)


@pytest.mark.parametrize("kind", ["random", "low", "high", "half", "segments"])
def test_normals_against_long_double(tmp_path, kind):
    if np.finfo(np.longdouble).eps > 2.0 ** -63:
        pytest.skip("long double is binary64 here")
    normal_tables.write(str(tmp_path / "normal_tables.h"))
    (tmp_path / "n.cpp").write_text(SRC)
    so = str(tmp_path / "n.so")
    subprocess.check_call(["g++", "-O2", "-std=c++17", "-shared", "-fPIC", "-I", str(tmp_path), "-I", b.CSRC, "-o", so,
                           str(tmp_path / "n.cpp")])
    w0, w1 = (np.ascontiguousarray(w) for w in _words(kind))
    z = np.empty((2, w0.size))
    p = lambda a: a.ctypes.data_as(ctypes.c_void_p)
    ctypes.CDLL(so).normals(p(w0), p(w1), ctypes.c_long(w0.size), p(z[0]), p(z[1]))
    m = (2 * (w0 >> 9).astype(np.int64) + 1)
    two24 = np.longdouble(1 << 24)
    r = np.sqrt(-2 * np.where(m > (1 << 23), np.log1p(-(two24 - m) / two24), np.log(m / two24)))
    # the angle from the nearest quarter turn: exact reduction, then |a| <= pi / 4
    a = (2 * (w1 >> 9).astype(np.int64) + 1)
    q = (a + (1 << 21)) >> 22
    x = (a - (q << 22)).astype(np.longdouble) * (np.longdouble(2) * np.arccos(np.longdouble(-1)) / two24)
    c, s = np.cos(x), np.sin(x)
    cos = np.choose(q & 3, [c, -s, -c, s])
    sin = np.choose(q & 3, [s, c, -s, -c])
    for got, want in ((z[0], r * cos), (z[1], r * sin)):
        err = np.abs(got.astype(np.longdouble) - want)
        # the fixed-point pair within 2^-56 (radius 2^-57.3, angle 2^-59.5 times r < 5.8), the encoding half an ulp
        assert np.all(err <= 2.0 ** -56 + 0.5 * np.spacing(np.abs(got)) * 1.001)


def _all_words(kind):
    """Every radius with one angle, or every angle with one radius (of which the words' upper 23 bits count)."""
    k = (np.arange(1 << 23, dtype=np.uint64) << 9).astype(np.uint32)
    one = np.full(k.size, {"angles": 0x12345600, "angles, u near 1": 0xFFFFFE00, "radii": 0x02345600}[kind], np.uint32)
    return (k, one) if kind == "radii" else (one, k)


@pytest.mark.parametrize("kind", ["angles", "angles, u near 1", "radii"])
def test_relative_error_at_every_size(tmp_path, kind):
    """The error relative to the normal, however small it is: half an ulp of the rounding (2^-53 at most)
    and the fixed-point pair's: the sine at node 0, n times a series that is off by a unit of 2^31.4 in a
    term of 2^-23.3, 2^-54.7; the product of radius and sine, two units of 2^57.6, 2^-56.6; radius, cosine
    and the other nodes' sines below 2^-58 each.  2^-54 covers the sum."""
    if np.finfo(np.longdouble).eps > 2.0 ** -63:
        pytest.skip("long double is binary64 here")
    normal_tables.write(str(tmp_path / "normal_tables.h"))
    (tmp_path / "n.cpp").write_text(SRC)
    so = str(tmp_path / "n.so")
    subprocess.check_call(["g++", "-O2", "-std=c++17", "-shared", "-fPIC", "-I", str(tmp_path), "-I", b.CSRC, "-o", so,
                           str(tmp_path / "n.cpp")])
    w0, w1 = _all_words(kind)
    z = np.empty((2, w0.size))
    p = lambda a: a.ctypes.data_as(ctypes.c_void_p)
    ctypes.CDLL(so).normals(p(w0), p(w1), ctypes.c_long(w0.size), p(z[0]), p(z[1]))
    two24 = np.longdouble(1 << 24)
    for lo in range(0, w0.size, 1 << 20):     # in parts: long doubles take 16 bytes each
        part = slice(lo, lo + (1 << 20))
        m = (2 * (w0[part] >> 9).astype(np.int64) + 1)
        r = np.sqrt(-2 * np.where(m > (1 << 23), np.log1p(-(two24 - m) / two24), np.log(m / two24)))
        a = (2 * (w1[part] >> 9).astype(np.int64) + 1)
        q = (a + (1 << 21)) >> 22
        x = (a - (q << 22)).astype(np.longdouble) * (np.longdouble(2) * np.arccos(np.longdouble(-1)) / two24)
        c, s = np.cos(x), np.sin(x)
        for got, want in ((z[0, part], r * np.choose(q & 3, [c, -s, -c, s])),
                          (z[1, part], r * np.choose(q & 3, [s, c, -s, -c]))):
            assert np.all(np.abs(got.astype(np.longdouble) - want) <= (2.0 ** -53 + 2.0 ** -54) * np.abs(want))


def _step(bins, match, d, n, steps, eps=0.1, x0=None, y0=None):
    import torch
    from paper_1912_09240_gb300 import _lib as L
    kind = L.PR_MODEL_OU if d == 1 else L.PR_MODEL_DW_MULTI
    model, grid = L.Model(kind, d, 1.0, 1.0, eps), L.Grid(bins, -4.0, 4.0)
    dev = "cuda"
    x = torch.zeros(1, n, dtype=torch.float64, device=dev) if x0 is None else x0.clone()
    y = torch.zeros(1, d, n, dtype=torch.float64, device=dev) if y0 is None else y0.clone()
    cdf = torch.linspace(0.0, 1.0, bins + 1, dtype=torch.float64, device=dev).reshape(1, -1)
    counts = torch.empty(1, bins, dtype=torch.int32, device=dev)
    L.pr_fine_propagate(model, L.PR_F64, L.Rng(17, 3), x, y, False, x, y, n, 5, 1, steps, 1e-3, grid,
                        cdf if match else None, cdf if match else None, None, None, counts, None)
    torch.cuda.synchronize()
    return x, y, counts


@pytest.mark.gpu
@pytest.mark.parametrize("d", [1, 2, 3, 4, 16])
@pytest.mark.parametrize("n", [1, 129, 5003])
def test_one_step_gives_the_normals(d, n):
    from oracle import oracle
    b.build()
    x, y, _ = _step(64, False, d, n, 1)
    sx, sy = np.sqrt(2.0 * 1e-3), np.sqrt(2.0 / 0.1 * 1e-3)
    got = np.concatenate([x.cpu().numpy() / sx, y.cpu().numpy()[0] / sy])
    want = np.stack([oracle.step_normals(17, 3, p, 5, 0, 1 + d) for p in range(min(n, 200))], 1)
    # both sides within an ulp or two of the exact normal (|z| < 5.8: 2^-50), the products round once more
    assert np.max(np.abs(got[:, :want.shape[1]] - want)) <= 2.0 ** -48


@pytest.mark.gpu
@pytest.mark.parametrize("d", [1, 3])
@pytest.mark.parametrize("n", [700, 1 << 17, (1 << 20) + 37])
def test_tables_in_shared_memory_or_not(d, n):
    """The tables beside the histograms (shared memory) and, at 4096 bins with a matching that maps
    every particle onto itself, through L1; and runs too short for the copy."""
    import torch
    b.build()
    g = torch.Generator(device="cuda").manual_seed(3)
    x0 = torch.randn(1, n, generator=g, device="cuda", dtype=torch.float64)
    y0 = torch.randn(1, d, n, generator=g, device="cuda", dtype=torch.float64)
    a = _step(100, False, d, n, 17, x0=x0, y0=y0)
    c = _step(4096, True, d, n, 17, x0=x0, y0=y0)
    assert torch.equal(a[0], c[0]) and torch.equal(a[1], c[1])
    assert int(a[2].sum()) == n and int(c[2].sum()) == n
    # a short run ends where the same steps of the longer one's binary64 oracle path do
    from oracle import oracle
    m = oracle.Model(0 if d == 1 else 2, d, 1.0, 1.0, 0.1)
    ids = np.unique(np.concatenate([np.arange(min(n, 50)), n - 1 - np.arange(min(n, 50))])).astype(np.uint32)
    s = _step(100, False, d, n, 7, x0=x0, y0=y0)
    for steps, got in ((7, s), (17, a)):
        xo, _ = oracle.fine_propagate(m, 17, x0.cpu().numpy()[:, ids], y0.cpu().numpy()[:, :, ids], 5, steps, 1e-3,
                                      problem=3, ids=ids)
        assert np.max(np.abs(xo - got[0].cpu().numpy()[:, ids])) <= 1e-12
