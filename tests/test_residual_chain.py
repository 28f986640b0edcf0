"""The rule by which the kernels of a residual start in each other's tails (residual_chain.h, host C++ alone)."""
import os
import shutil
import subprocess

import pytest

CSRC = os.path.join(os.path.dirname(os.path.dirname(os.path.abspath(__file__))), "paper_1807_01151_gb300", "csrc")


@pytest.fixture(scope="module")
def chains(tmp_path_factory):
    gxx = shutil.which("g++")
    if gxx is None:
        pytest.skip("no C++ compiler")
    d = tmp_path_factory.mktemp("rule")
    src, exe = d / "rule.cpp", d / "rule"
    src.write_text('#include <cstdio>\n#include <cstdlib>\n#include "residual_chain.h"\nint main(int, char** v) {\n'
                   'std::printf("%d\\n", (int)emg::residual_chains(std::atoi(v[1]), std::atoi(v[2]), std::atoll(v[3]), '
                   'std::atoll(v[4])));\n}\n')
    subprocess.run([gxx, "-std=c++17", "-Wall", "-I", CSRC, str(src), "-o", str(exe)], check=True)

    def rule(dim, n1, n2, p):
        e = n1 * n2 if dim == 2 else 6 * n1 * n1 * n2
        f = 2 * e + n1 if dim == 2 else 3 * e + 6 * n1 * n1
        out = subprocess.run([str(exe)] + [str(x) for x in (dim, p, e, f * (p + 2) ** (dim - 1))],
                             capture_output=True, text=True, check=True)
        return bool(int(out.stdout))
    return rule


@pytest.mark.parametrize("case", [(2, 32, 16, 0), (2, 110, 55, 0), (3, 10, 12, 0), (2, 32, 16, 1), (2, 32, 16, 2), (2, 24, 10, 3),
                                  (2, 45, 21, 4), (3, 3, 4, 1), (2, 181, 80, 3), (2, 150, 70, 4), (2, 256, 128, 2)])
def test_chained_where_it_was_measured_faster(chains, case):
    assert chains(*case)


@pytest.mark.parametrize("case", [(2, 128, 64, 0), (2, 256, 128, 0), (2, 90, 45, 2), (2, 128, 64, 2), (2, 90, 45, 3), (2, 110, 50, 3),
                                  (2, 128, 64, 3), (2, 110, 50, 4), (3, 6, 9, 1), (3, 5, 6, 2), (3, 5, 7, 3),
                                  (3, 6, 9, 3), (3, 4, 6, 4), (3, 5, 7, 4)])
def test_apart_where_chaining_was_measured_slower(chains, case):
    assert not chains(*case)
