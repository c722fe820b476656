"""CPU check of the rules that choose among kernels and their splits (csrc/routes.h),
compiled by themselves for the host."""
import os
import subprocess

import pytest

CSRC = os.path.join(os.path.dirname(os.path.dirname(os.path.abspath(__file__))), "paper_1007_3509_gb300", "csrc")


@pytest.fixture(scope="module")
def ask(tmp_path_factory):
    """ask(expression, ...): the expressions evaluated with the header's functions."""
    d = tmp_path_factory.mktemp("routes")

    def run(*exprs):
        src, exe = str(d / "main.cpp"), str(d / "main")
        open(src, "w").write("#include <stdio.h>\n#include \"routes.h\"\nusing namespace hp;\nint main() {\n" +
                             "".join(f'printf("%g\\n", (double)({e}));\n' for e in exprs) + "}\n")
        subprocess.run(["g++", "-std=c++17", "-I", CSRC, "-o", exe, src], check=True)
        return [float(v) for v in subprocess.run([exe], capture_output=True, text=True, check=True).stdout.split()]
    return run


def _lean_windows(x, y, z):
    return -(-x // 56) * -(-y // 28) * (z // 2)


def test_few_windows_take_eight_warps(ask):
    """Lattices with material points that four warps a window swept slower than eight."""
    small = [(32, 32, 32), (44, 76, 32), (48, 48, 48), (56, 56, 56), (76, 64, 40), (112, 112, 112), (126, 90, 76)]
    large = [(126, 90, 78), (128, 128, 64), (128, 128, 128), (1024, 1024, 1024)]
    got = ask(*(f"lean_warps({_lean_windows(*L)})" for L in small + large))
    assert got == [8] * len(small) + [4] * len(large)


def test_a_scant_second_wave_takes_eight_warps(ask):
    """Ensembles without material points whose four-warp windows (seven an SM) just overflow
    one wave: 64^3, 128^3 and 64^3 were slower so than they had been with eight warps."""
    got = ask(*(f"lean_warps({w}, 7)" for w in (456, 576, 960, 1064, 1065, 1152, 1344, 1440, 1536, 1920, 6400)))
    assert got == [8, 4, 4, 4, 8, 8, 8, 8, 4, 4, 4]
    assert ask("lean_warps(1344)", "lean_warps(1344, 0)") == [4, 4]


def test_tall_tiles_where_short_ones_need_a_second_wave(ask):
    """Lattices of 2.3 to 4.2 million sites that the short tiles swept slower."""
    tall = [(8, 1362, 2300), (8, 1190, 3500), (8, 3002, 1000), (8, 1702, 1702), (8, 2046, 1500), (8, 1502, 2000),
            (8, 1800, 1800), (8, 2044, 2044), (8, 2402, 1100), (8, 4096, 4096),
            (4, 1702, 1702), (4, 3002, 1000), (4, 1502, 2000), (4, 1362, 2300), (4, 1922, 1960)]
    short = [(8, 1502, 1502), (8, 1022, 2300), (8, 1202, 1202), (8, 3002, 700), (8, 500, 500),
             (4, 1602, 1700), (4, 962, 2800), (4, 2046, 2046), (4, 2402, 2402), (4, 1800, 1800), (4, 2048, 2048), (4, 4096, 4096)]
    got = ask(*(f"tall_tiles({n}, {x}, {y}, false)" for n, x, y in tall + short))
    assert got == [1] * len(tall) + [0] * len(short)
    # with material points, by sites alone
    assert ask("tall_tiles(8, 1702, 1702, true)", "tall_tiles(8, 2048, 2048, true)", "tall_tiles(4, 3002, 3002, true)") == [0, 1, 0]


def test_one_lattice_on_a_cluster_by_its_shape(ask):
    """Long or wide strips that the cluster kernel swept slower than one launch per colour."""
    cluster = [(4, 64, 64), (4, 128, 128), (4, 126, 130), (4, 256, 64), (4, 190, 86), (8, 64, 64), (8, 128, 128), (8, 128, 256),
               (8, 256, 256), (8, 220, 220), (8, 512, 64), (8, 64, 512), (8, 120, 240)]
    colour = [(4, 128, 200), (4, 120, 240), (4, 64, 256), (4, 512, 32), (4, 1024, 16), (4, 2048, 8), (4, 16, 1024), (4, 8, 2000),
              (8, 512, 128), (8, 300, 200), (8, 180, 360), (8, 64, 1000), (8, 2000, 30), (8, 2048, 16), (8, 1022, 64),
              (8, 16, 4000), (8, 32, 2000)]
    got = ask(*(f"one_resident({n}, {x}, {y}, res_cluster(8, {y}))" for n, x, y in cluster + colour))
    assert got == [1] * len(cluster) + [0] * len(colour)


def _ensemble_us(ask, nbr, shapes, sharing=1):
    tiles = "[] { TileCost t; " + "".join(f"t.add({x}, {y}); " for x, y in shapes) + f"return t.us({nbr}, true); }}()"
    return ask(tiles, *(f"res_us({nbr}, {x}, {y}, 8, {sharing})" for x, y in shapes))


def test_ensembles_estimate_the_longest_member_and_the_tiles(ask):
    """Measured us per MCS (50-site grains, kT = 1) of one wave of clusters and of the tiles."""
    for nbr, shapes, cluster, tiles in [
            (8, [(600, 600)] + [(64, 64)] * 7, 33.0, 17.7), (8, [(400, 1000)] + [(64, 64)] * 14, 38.9, 18.6),
            (8, [(2048, 64)] * 8, 28.1, 16.2), (8, [(500, 500)] * 8, 20.7, 22.7), (8, [(300, 300)] * 8, 11.1, 14.2),
            (8, [(200, 200)] * 8, 7.0, 12.4), (8, [(64, 1000)] * 8, 13.4, 19.9), (4, [(600, 600)] * 8, 30.0, 23.8),
            (4, [(256, 256)] * 8, 6.8, 11.4), (4, [(2048, 64)] * 8, 16.0, 12.6), (4, [(400, 1000)] + [(64, 64)] * 14, 37.0, 15.7)]:
        t, *m = _ensemble_us(ask, nbr, shapes)
        assert abs(max(m) / cluster - 1) < 0.2 and abs(t / tiles - 1) < 0.3, (nbr, shapes[0], t, max(m))
        assert (max(m) <= 1.07 * t) == (cluster <= tiles), (nbr, shapes[0], t, max(m))


def test_narrow_lattices_go_per_colour(ask):
    """Lattices that a window of 128 columns goes through several times over."""
    def rule(n, x, y, tables=0, mp=0):
        return f"per_colour_2d({n}, {x}, {x * y}LL, {tables}, {mp})"
    colour = [rule(4, 16, 8000, 1), rule(4, 16, 60000, 1), rule(4, 100, 4000, 1), rule(4, 16, 60000), rule(4, 126, 8000, 0, 1),
              rule(8, 16, 60000), rule(8, 16, 60000, 1), rule(8, 64, 20000, 0, 1), rule(4, 700, 700), rule(8, 2000, 30)]
    tiles = [rule(4, 128, 2000, 1), rule(4, 360, 360, 1), rule(4, 1024, 1024), rule(8, 100, 4000, 1), rule(8, 128, 600),
             rule(8, 128, 128, 0, 1), rule(8, 256, 256, 1)]
    assert ask(*colour, *tiles) == [1] * len(colour) + [0] * len(tiles)


def test_small_lattices_are_counted_by_many_warps(ask):
    """A share of 2048 sites left a 500^2 lattice to 123 warps, one after the other's step."""
    sizes = [64 ** 2, 250 ** 2, 500 ** 2, 1116 ** 2, 1116 * 1118, 2000 ** 2, 4096 ** 2, 1024 ** 3]
    assert ask(*(f"counts_seg({n}LL)" for n in sizes)) == [128, 128, 128, 256, 256, 512, 2048, 2048]
