"""The serial sweep on a cluster of CTAs: what an exchange stores into the other
CTAs' shared memory must overlap nothing that they may still be using, that is,
nothing that is used between the cluster barrier before it and its own (the
CTAs run apart in between).  The places are taken from the device code's own
layout, compiled for the host."""
import subprocess

import pytest

from paper_1912_09240_gb300 import build as b

# what carve_jq lays out, as (name, element count, element size) per field
SRC = r"""
#include <cstdio>
#include <cstdlib>
#include "coarse_dev.cuh"
int main(int argc, char** argv)
{
    for (int i = 1; i < argc; ++i) {
        const int I = atoi(argv[i]), M = 3 * (I + 1);
        alignas(16) static unsigned char base[1 << 18];
        const pr::JqSmem j = pr::carve_jq(base, I);
        auto show = [&](const char* name, const void* p, size_t bytes) {
            printf("%d %s %ld %zu\n", I, name, (long)((const unsigned char*)p - base), bytes);
        };
        show("all", base, pr::jq_smem_bytes(I));
        show("levels", j.levels, 8 * (size_t)M);
        show("mass", j.mass, 8 * (size_t)I);
        show("mp", j.mp, 8 * (size_t)I);
        show("counted", j.counted, 8 * (size_t)M);
        show("kq", j.kq, 16 * (size_t)M);
        show("below", j.below, 8 * (size_t)M);
        show("per", j.per, 4 * (size_t)((M + 31) / 32));
        show("bsum", j.bsum, 16 * (size_t)M);
        show("wsum", j.wsum, 8 * (size_t)pr::kWsum);
        show("edges", j.edges, 8 * (size_t)(I + 1));
        show("flag", j.flag, 16);
    }
}
"""
BINS = [1, 5, 63, 64, 200, 256, 257, 288, 512, 1023, 1024]


@pytest.fixture(scope="module")
def layout(tmp_path_factory):
    d = tmp_path_factory.mktemp("layout")
    (d / "l.cu").write_text(SRC)
    subprocess.check_call([b.nvcc(), *b.ARCH, "-std=c++17", "-I", b.CSRC, "-o", str(d / "l"), str(d / "l.cu")])
    out = {}
    for line in subprocess.check_output([str(d / "l"), *map(str, BINS)], text=True).splitlines():
        bins, name, at, size = line.split()
        out.setdefault(int(bins), {})[name] = (int(at), int(at) + int(size))
    return out


def _apart(places, target, others):
    lo, hi = places[target]
    assert lo % 8 == 0 and places["all"][0] <= lo and hi <= places["all"][1]
    for o in others:
        assert hi <= places[o][0] or places[o][1] <= lo, (target, o)


@pytest.mark.parametrize("bins", BINS)
def test_counts_exchanged_beside_the_coarse_step(layout, bins):
    """share(mp) .. share(counted): the coarse step's scan and division, the edges and the status flag."""
    _apart(layout[bins], "counted", ["mass", "mp", "wsum", "edges", "flag"])


@pytest.mark.parametrize("bins", BINS)
def test_knots_exchanged_beside_the_levels(layout, bins):
    """share(counted) .. share(kq): merge, compaction and quantiles (which read `below`, not their own knots)."""
    _apart(layout[bins], "kq", ["counted", "below", "per", "levels", "bsum", "wsum", "edges", "flag"])
    _apart(layout[bins], "below", ["counted", "per", "levels", "bsum", "wsum", "edges", "flag"])
    # the group counts fit the scratch that they stand in
    p = layout[bins]
    assert p["wsum"][0] <= p["per"][0] and p["per"][1] <= p["wsum"][1]
