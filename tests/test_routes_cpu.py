"""CPU check of the rules that choose among the sweep kernels (csrc/routes.h), compiled by
themselves for the host."""
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
