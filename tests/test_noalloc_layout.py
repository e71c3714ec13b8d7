"""The scratch array of the allocation-free entry point, on the CPU: a program
compiled against its layout prints where a call's arrays lie.  What a call must
find at zero (status word, occupancy maxima, cell counts, replica ids, kinetic
energies) has to be inside the one range that the call clears, without overlaps and
inside the array, for any size; the call itself clears that range before its first
kernel.  No device is used."""
import os
import re
import shutil
import subprocess

import pytest

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))
CSRC = os.path.join(ROOT, "paper_2510_21230_gb300", "csrc")

PROGRAM = r"""
#include <cstdio>
#include "noalloc_layout.cuh"
using namespace atm3;
int main()
{
    const long long sizes[][2] = {{0, 27}, {1, 27}, {500, 64}, {5003, 343}, {32768, 32768}};
    for (auto& s : sizes) {
        const NaZero Z = na_zero(s[0], s[1]);
        std::printf("%lld %lld %zu %zu %zu %zu %zu %zu %zu %zu %zu %zu\n", s[0], s[1], NA.res, NA.zero, Z.status,
                    Z.maxocc, Z.count, Z.rep_of_cell, Z.rep_of_mol, Z.ke, Z.end, NA.total);
    }
}
"""


@pytest.fixture(scope="module")
def layouts(tmp_path_factory):
    nvcc = os.path.join(os.environ.get("CUDA_HOME", "/usr/local/cuda"), "bin", "nvcc")
    if not os.path.exists(nvcc):
        nvcc = shutil.which("nvcc")
    if nvcc is None:
        pytest.skip("no nvcc")
    d = tmp_path_factory.mktemp("layout")
    (d / "layout.cu").write_text(PROGRAM)
    subprocess.run([nvcc, "-std=c++17", "-I", CSRC, "-I", os.path.join(ROOT, "include"),
                    str(d / "layout.cu"), "-o", str(d / "layout")], check=True, capture_output=True)
    out = subprocess.run([str(d / "layout")], check=True, capture_output=True, text=True).stdout
    return [tuple(map(int, line.split())) for line in out.splitlines()]


def test_what_starts_at_zero_is_inside_the_cleared_range(layouts):
    assert len(layouts) == 5
    for n, ncell, res, zero, status, maxocc, count, roc, rom, ke, end, total in layouts:
        assert zero == status and res < zero
        spans = [(status, 4), (maxocc, 4 * 7), (count, 4 * ncell), (roc, 4 * ncell), (rom, 4 * n), (ke, 8 * n)]
        at = zero
        for begin, size in spans:
            assert begin >= at and begin % 256 == 0
            at = begin + size
        assert at <= end <= total


def test_the_range_is_cleared_before_the_first_kernel():
    with open(os.path.join(CSRC, "noalloc.cu")) as f:
        src = f.read()
    clear = re.search(r"cudaMemsetAsync\(base \+ NA\.zero, 0, Z\.end - NA\.zero, st\)", src)
    assert clear and clear.start() < src.index("launch_cell_counts(")
    for name in ("count", "rep_of_cell", "rep_of_mol", "ke", "status", "maxocc"):
        assert re.search(r"\b%s = reinterpret_cast<\w+\*>\(base \+ Z\.%s\)" % (name, name), src), name
