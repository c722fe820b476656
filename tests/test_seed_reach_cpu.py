"""CPU check of the bounds the Voronoi assignment narrows its seed lists with
(csrc/reach.h): least and largest distance of a seed to an interval of sites, against
the distances to every site of it; and of the rule that leaves lattices of small grains
to the kernel of single sites, against the lists of seeds thrown at random.  The header
is compiled by itself for the host."""
import os
import subprocess

import numpy as np
import pytest

CSRC = os.path.join(os.path.dirname(os.path.dirname(os.path.abspath(__file__))), "paper_1007_3509_gb300", "csrc")

MAIN = """
#include <stdio.h>
#include "reach.h"
int main(int argc, char** argv) {
    int near, s, b, len, L;
    if (argc > 1) {
        int dim, e[3];
        long long G;
        while (scanf("%d %d %d %d %lld", &dim, e, e + 1, e + 2, &G) == 5)
            printf("%d %d\\n", (int)hp::assign_by_bricks(dim, e, G), (int)hp::brick_lists(dim, e, G).seeds);
        return 0;
    }
    while (scanf("%d %d %d %d %d", &near, &s, &b, &len, &L) == 5) {
        const hp::Reach r = near ? hp::reach_near(s, b, len) : hp::reach(s, b, len, L);
        printf("%d %d\\n", r.lo, r.hi);
    }
}
"""


@pytest.fixture(scope="module")
def bounds(tmp_path_factory):
    d = tmp_path_factory.mktemp("reach")
    src, exe = str(d / "main.cpp"), str(d / "main")
    open(src, "w").write(MAIN)
    subprocess.run(["g++", "-std=c++17", "-O1", "-I", CSRC, "-o", exe, src], check=True)

    def run(rows, *args):
        text = "\n".join(" ".join(map(str, r)) for r in rows)
        out = subprocess.run([exe, *args], input=text, capture_output=True, text=True, check=True).stdout
        return np.array(out.split(), dtype=np.int64).reshape(-1, 2)
    return run


def test_folded_bounds_are_the_extreme_distances(bounds):
    rows, want = [], []
    for L in (1, 2, 6, 16, 50):
        for b in range(0, L, max(1, L // 5)):
            for ln in sorted({0, 1, 7, 31, L - 1}):
                if b + ln >= L:
                    continue
                for s in range(L):
                    d = np.abs(np.arange(b, b + ln + 1) - s)
                    d = np.minimum(d, L - d)
                    rows.append((0, s, b, ln, L))
                    want.append((d.min(), d.max()))
    np.testing.assert_array_equal(bounds(rows), want)


def test_near_image_bounds_are_the_extreme_distances(bounds):
    """A looser upper bound gives the same tessellation from lists several times as long."""
    rows, want = [], []
    for ln in (0, 1, 3, 7, 31, 63):
        for b in (0, 8, 40):
            for s in range(b - 50, b + ln + 51):
                d = np.abs(np.arange(b, b + ln + 1) - s)
                rows.append((1, s, b, ln, 0))
                want.append((d.min(), d.max()))
    np.testing.assert_array_equal(bounds(rows), want)


def _list_lengths(L, G, ext, rng):
    """Seeds within reach of a few whole bricks: those no further from the brick than the
    least over the seeds of the largest distance to it."""
    pos = np.stack([rng.integers(0, v, G) for v in L], 1)
    out = []
    for _ in range(6):
        lo2, hi2 = np.zeros(G), np.zeros(G)
        for d, (l, e) in enumerate(zip(L, ext)):
            b = rng.integers(0, max(1, l // e)) * e
            t = np.abs(np.arange(b, min(b + e, l))[:, None] - np.arange(l)[None, :])
            t = np.minimum(t, l - t)
            lo2 += t.min(0)[pos[:, d]].astype(float) ** 2
            hi2 += t.max(0)[pos[:, d]].astype(float) ** 2
        out.append(int((lo2 <= hi2.min()).sum()))
    return np.mean(out)


@pytest.mark.parametrize("L,sizes", [
    ((128, 128, 128), (3, 8, 24, 48, 64, 110, 150, 300, 2000)), ((200, 96, 130), (6, 40, 150, 400)),
    ((512, 512, 8), (6, 16, 48, 300)), ((30, 30, 30), (3, 24, 80, 300)), ((1024, 1024), (3, 8, 10, 16, 24, 100)),
    ((256, 256), (3, 10, 32, 200)), ((34, 900), (3, 60))])
def test_lists_that_overflow_are_left_to_single_sites(bounds, L, sizes):
    rng = np.random.default_rng(11)
    ext = (32, 8, 8) if len(L) == 3 else (64, 32)
    for v in sizes:
        G = int(np.prod(L)) // v
        (bricks, est), = bounds([(len(L), *L, *(1,) * (3 - len(L)), G)], "rule")
        n = _list_lengths(L, G, ext, rng)
        if n > 20:
            assert 0.85 < est / n < 1.5, (L, v, est, n)
        if n > 1024:
            assert not bricks, (L, v, n)
        if v >= 100:
            assert bricks, (L, v, n)


def test_axes_too_long_for_32_bit_distances(bounds):
    assert bounds([(2, 32770, 4, 1, 40), (3, 4, 4, 40000, 40), (2, 32768, 64, 1, 40)], "rule")[:, 0].tolist() == [0, 0, 1]
