"""CPU check of the bounds the Voronoi assignment narrows its seed lists with
(csrc/reach.h): least and largest distance of a seed to an interval of sites, against
the distances to every site of it.  The header is compiled by itself for the host."""
import os
import subprocess

import numpy as np
import pytest

CSRC = os.path.join(os.path.dirname(os.path.dirname(os.path.abspath(__file__))), "paper_1007_3509_gb300", "csrc")

MAIN = """
#include <stdio.h>
#include "reach.h"
int main() {
    int near, s, b, len, L;
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

    def run(rows):
        text = "\n".join(" ".join(map(str, r)) for r in rows)
        out = subprocess.run([exe], input=text, capture_output=True, text=True, check=True).stdout
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
