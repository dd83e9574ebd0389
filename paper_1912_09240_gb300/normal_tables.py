"""Fixed-point tables of the binary64 normals, written as a C header at build time.

The binary64 kernels take their Box-Muller normals r cos(theta), r sin(theta)
from integer arithmetic (csrc/normal64.cuh): the radius r(u) = sqrt(-2 ln u)
from piecewise polynomials, the angle, reflected into an eighth of a turn, from
cosines and sines at equidistant nodes and the angle-addition formulas.
Everything here is computed with ``decimal`` and integers, so the header is the
same on every machine.

Radius: u = M 2^-24 with M an odd 24-bit integer.  For M < 2^23 the variable
is M, otherwise 2^24 - M (r is smooth in the logarithm of both; near u = 1 it
behaves like sqrt(2 (1 - u))).  Each binade 2^e <= M' < 2^(e+1) is cut into 32
equal segments, and on each r is the polynomial of degree 7 through its
Chebyshev points (relative error below 2^-60), as coefficients in sigma = tau / 2,
tau in [0, 1) the place in the segment, in units of 2^-(60 + shift): the shift of
the binade (``radius_shift``) puts r between 2^61 and 2^63 units, so that a small
radius keeps as many bits as a large one.
"""
from __future__ import annotations

import decimal
import os

D = decimal.Decimal
SEG_BITS = 5
DEGREE = 7
BINADES = 23
TAIL_SHIFT = 8        # c5..c7 are kept in units of 2^(TAIL_SHIFT - 60 - shift)
NODE_BITS = 10        # nodes per eighth of a turn: 2^10


def _pi(prec: int) -> D:
    """Machin's formula."""
    def arctan_inv(q: int, one: int) -> int:
        t = s = one // q
        k, sign = 3, -1
        while t:
            t //= q * q
            s += sign * (t // k)
            k, sign = k + 2, -sign
        return s
    one = 10 ** (prec + 10)
    return D(4 * (4 * arctan_inv(5, one) - arctan_inv(239, one))) / one


def _cos_sin(x: D) -> tuple:
    """Taylor series (|x| < 2)."""
    c, s, t, k = D(1), x, x, 1
    eps = D(10) ** -45
    u = D(1)
    while abs(t) > eps:
        u = -t * x / (k + 1)
        c += u
        t = u * x / (k + 2)
        s += t
        k += 2
    return c, s


def _chebyshev(n: int):
    """The Chebyshev points on [0, 1] and the rows turning values there into
    monomial coefficients."""
    pi = _pi(40)
    pts = [(1 - _cos_sin(pi * (2 * k + 1) / (2 * n))[0]) / 2 for k in range(n)]
    rows = []
    for k in range(n):   # Lagrange basis polynomial k, expanded
        poly, den = [D(1)], D(1)
        for j in range(n):
            if j != k:
                poly = [(poly[i - 1] if i else D(0)) - (poly[i] * pts[j] if i < len(poly) else D(0))
                        for i in range(len(poly) + 1)]
                den *= pts[k] - pts[j]
        rows.append([c / den for c in poly])
    return pts, rows


def _rint(v: D) -> int:
    return int(v.to_integral_value(rounding=decimal.ROUND_HALF_EVEN))


def radius_shift(side: int, e: int) -> int:
    """r 2^(60 + shift) is at least 2^61 and below 2^63 on the binade 2^e of u (side 0) or 1 - u (side 1)."""
    return (26 - e) >> 1 if side else int(e >= 13)


def radius_table():
    """[segment][DEGREE + 1] integers: c_k 2^k 2^(60 + shift) (k <= 4), the rest in units of 2^(TAIL_SHIFT - 60 - shift)."""
    n = DEGREE + 1
    pts, rows = _chebyshev(n)
    out = []
    segs = 1 << SEG_BITS
    for side in range(2):
        for e in range(BINADES):
            for g in range(segs):
                vals = []
                for p in pts:
                    m = D(2) ** (e - 24) * (1 + (g + p) / segs)   # u or 1 - u
                    vals.append((-2 * (1 - m if side else m).ln()).sqrt())
                coef = [sum(rows[k][i] * vals[k] for k in range(n)) for i in range(n)]
                one = 60 + radius_shift(side, e)
                assert all(2 ** 60 < v * 2 ** one < 2 ** 63 for v in vals)
                scaled = [c * 2 ** (one + i - (TAIL_SHIFT if i > 4 else 0)) for i, c in enumerate(coef)]
                out.append([_rint(c) for c in scaled])
    return out


def node_table():
    """[node](cos 2^63, sin 2^(62 + z)) of node pi/4 / 2^NODE_BITS, z the zeros in front of its number in
    NODE_BITS bits: an angle between this node and the next has them in front of it too."""
    pi = _pi(40)
    return [tuple(_rint(v * 2 ** k) for v, k in zip(_cos_sin(pi / 4 * i / (1 << NODE_BITS)),
                                                    (63, 62 + NODE_BITS - i.bit_length())))
            for i in range(1 << NODE_BITS)]


def header() -> str:
    with decimal.localcontext() as ctx:
        ctx.prec = 42
        rad, nodes = radius_table(), node_table()
        d = 2 * _pi(40) / 2 ** 24                      # the angle of one unit
        consts = {
            "kSin1": _rint(d * 2 ** 84), "kSin3": _rint(d ** 3 / 6 * 2 ** 98),
            "kSin5": _rint(d ** 5 / 120 * 2 ** 144),
            "kCos2": _rint(d ** 2 / 2 * 2 ** 97), "kCos4": _rint(d ** 4 / 24 * 2 ** 119),
        }
    for c in rad:
        assert all(abs(v) < 2 ** 63 for v in c[:5]) and all(abs(v) < 2 ** 31 for v in c[5:])
    u64 = lambda v: "0x%xull" % (v & (2 ** 64 - 1))
    u32 = lambda v: v & (2 ** 32 - 1)
    lines = ["// Written by normal_tables.py at build time.", "#pragma once", "namespace pr {"]
    lines += ["constexpr unsigned long long %s = %s;" % (k, u64(v)) for k, v in consts.items()]
    lines += ["constexpr int kSegBits = %d;" % SEG_BITS, "constexpr int kRadiusSegments = %d;" % len(rad), "constexpr int kTailShift = %d;" % TAIL_SHIFT,
              "constexpr int kNodes = %d;" % len(nodes),
              "// per segment: c0 c1 | c2 c3 | c4, c5 + 2^32 c6; then c7 of every segment"]
    words = [u64(w) for c in rad for w in (*c[:5], u32(c[5]) | (u32(c[6]) << 32))]
    words += [u64(w) for n in nodes for w in n]
    c7 = [u32(c[7]) for c in rad]
    words += [u64(a | (b << 32)) for a, b in zip(c7[::2], c7[1::2])]
    lines.append("PR_TABLE_STORAGE unsigned long long kNormalTables[%d] = {" % len(words))
    lines += [",".join(words[i:i + 8]) + "," for i in range(0, len(words), 8)]
    lines += ["};", "}  // namespace pr", ""]
    return "\n".join(lines)


def write(path: str) -> str:
    tmp = path + f".tmp{os.getpid()}"
    with open(tmp, "w") as f:
        f.write(header())
    os.replace(tmp, path)
    return path


if __name__ == "__main__":
    import sys
    print(write(sys.argv[1]))
