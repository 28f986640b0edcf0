"""The rule that shares the Krylov rows out over thread blocks (arnoldi_blocks.h, host C++ alone)."""
import os
import shutil
import subprocess

import pytest

CSRC = os.path.join(os.path.dirname(os.path.dirname(os.path.abspath(__file__))), "paper_1807_01151_gb300", "csrc")


@pytest.fixture(scope="module")
def blocks(tmp_path_factory):
    gxx = shutil.which("g++")
    if gxx is None:
        pytest.skip("no C++ compiler")
    d = tmp_path_factory.mktemp("rule")
    src, exe = d / "rule.cpp", d / "rule"
    src.write_text('#include <cstdio>\n#include <cstdlib>\n#include "arnoldi_blocks.h"\nint main(int, char** v) {\n'
                   'std::printf("%lld\\n", (long long)emg::arnoldi_blocks(std::atoll(v[1]), std::atoi(v[2]), 152, '
                   'std::atoi(v[3]), 320));\n}\n')
    subprocess.run([gxx, "-std=c++17", "-Wall", "-I", CSRC, str(src), "-o", str(exe)], check=True)
    return lambda rows, f32, per_sm=2: int(subprocess.run([str(exe), str(rows), str(int(f32)), str(per_sm)],
                                                          capture_output=True, text=True, check=True).stdout)


@pytest.mark.parametrize("rows", [29185, 30720, 33280, 36400, 38912])
def test_float64_rows_between_192_and_256_a_block_take_256(blocks, rows):
    """One block an SM as long as 256 rows a block allow it: a second one on every SM costs more."""
    assert blocks(rows, False) == -(-rows // 256) <= 152


@pytest.mark.parametrize("f32", [False, True])
@pytest.mark.parametrize("per_sm", [1, 2, 3])
def test_blocks_are_resident_and_hold_every_row(blocks, f32, per_sm):
    """Every block co-resident (a cooperative launch), at most the partials' room, at least one."""
    for rows in (1, 127, 128, 129, 2560, 10240, 10241, 19456, 19457, 29184, 29185, 38912, 38913, 40960, 64000, 10 ** 7):
        n = blocks(rows, f32, per_sm)
        assert 1 <= n <= min(152 * min(per_sm, 2), 320)
        if n < 152 * min(per_sm, 2):
            assert -(-rows // n) <= 256
