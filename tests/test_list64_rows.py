"""When the buffers of the FP64 lists are allocated, on the CPU (a program compiled
against the rule in forces.cuh): once per growth of the units; neither a size beyond
the limit nor a size that could not be had is tried again at every evaluation (each
try would wait for the stream and drop the steps' graph); rows that are there stay."""
import os
import shutil
import subprocess

import pytest

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))
CSRC = os.path.join(ROOT, "paper_2510_21230_gb300", "csrc")

PROGRAM = r"""
#include <cstdio>
#include <cstdlib>
#include "forces.cuh"
int main(int, char** a)
{
    std::printf("%lld\n", atm3::list64_rows_wanted(atoll(a[1]), atoll(a[2]), atoll(a[3]), atoi(a[4])));
}
"""


@pytest.fixture(scope="module")
def wanted(tmp_path_factory):
    nvcc = os.path.join(os.environ.get("CUDA_HOME", "/usr/local/cuda"), "bin", "nvcc")
    if not os.path.exists(nvcc):
        nvcc = shutil.which("nvcc")
    if nvcc is None:
        pytest.skip("no nvcc")
    d = tmp_path_factory.mktemp("rows")
    (d / "rows.cu").write_text(PROGRAM)
    subprocess.run([nvcc, "-std=c++17", "-I", CSRC, "-I", os.path.join(ROOT, "include"), str(d / "rows.cu"),
                    "-o", str(d / "rows")], check=True, capture_output=True)
    return lambda *a: int(subprocess.run([str(d / "rows"), *map(str, a)], check=True, capture_output=True,
                                         text=True).stdout)


def test_rows_hold_the_unit_and_the_graph_headroom(wanted):
    for mcap in (1, 7, 8, 63, 64, 270, 576):
        s = wanted(1000, 0, 0, mcap)
        assert s % 8 == 0 and mcap + max(8, mcap // 8) <= s
        assert wanted(1000, s, 0, mcap + max(8, mcap // 8)) == 0     # (graph steps' capacity)
        assert wanted(1000, s, 0, s + 1) > s


def test_beyond_the_limit_nothing_is_tried(wanted):
    s = wanted(1000, 0, 0, 270)
    n = (16 << 30) // (16 * s)
    assert wanted(n, 0, 0, 270) == s
    assert wanted(n + 1, 0, 0, 270) == 0
    assert wanted(n + 1, 100, 0, 270) == 0                           # the smaller rows stay


def test_what_could_not_be_had_is_not_tried_again(wanted):
    s = wanted(1000, 0, 0, 270)
    assert wanted(1000, 0, s, 270) == 0
    assert wanted(1000, 0, s, 576) == 0
    assert 0 < wanted(1000, 0, s, 100) < s                           # (smaller units later)
