"""When the product rule takes its kernel, and with how many warps (the rule in
forces.cu, asked on the CPU through the built library): four-warp CTAs for small units,
whose sixteen idle in vapours; never one warp beside a large table; not 3c01 in FP64 with
units of a few molecules, where the owner kernel is the faster one."""
import os
import shutil
import subprocess

import pytest

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))
PKG = os.path.join(ROOT, "paper_2510_21230_gb300")

PROGRAM = r"""
#include <cstdio>
#include <cstdlib>
#include "forces.cuh"
int main(int, char** a)
{
    atm3::ForceJob j{};
    double x = 0.0;
    j.x = &x;
    j.trunc = 1;
    j.trav = atoi(a[1]);
    j.prec = atoi(a[2]);
    j.mcap = atoi(a[3]);
    j.b.ncell = atoll(a[4]);
    j.b.ntot = 8000;
    j.optin = 232448;
    j.sms = 152;
    const atm3::ProdLaunch l = atm3::atm_prod_plan(j);
    std::printf("%d %d\n", l.warps, l.smem);
}
"""
T = {"3c01": 0, "3c18": 1, "3c08": 2, "3c08a": 4}


@pytest.fixture(scope="module")
def plan(tmp_path_factory):
    nvcc = os.path.join(os.environ.get("CUDA_HOME", "/usr/local/cuda"), "bin", "nvcc")
    if not os.path.exists(nvcc):
        nvcc = shutil.which("nvcc")
    if nvcc is None:
        pytest.skip("no nvcc")
    from paper_2510_21230_gb300 import build
    lib = build.build()
    d = tmp_path_factory.mktemp("prod")
    (d / "plan.cu").write_text(PROGRAM)
    subprocess.run([nvcc, "-std=c++17", "-I", os.path.join(PKG, "csrc"), "-I", os.path.join(ROOT, "include"),
                    str(d / "plan.cu"), lib, "-Xlinker", "-rpath", "-Xlinker", PKG, "-o", str(d / "plan")],
                   check=True, capture_output=True)
    return lambda trav, prec, mcap, ncell=10000: tuple(map(int, subprocess.run(
        [str(d / "plan"), str(T[trav]), "0" if prec == "fp64" else "1", str(mcap), str(ncell)], check=True,
        capture_output=True, text=True).stdout.split()))


@pytest.mark.parametrize("trav", ["3c01", "3c18", "3c08", "3c08a"])
def test_small_units_take_four_warps(plan, trav):
    for mcap in (1, 14, 64):
        assert plan(trav, "fp32c", mcap)[0] == 4
        if trav != "3c01":
            assert plan(trav, "fp64", mcap)[0] == 4
        assert plan(trav, "fp32c", 120)[0] > 4


def test_owner_fp64_only_with_units_of_some_size(plan):
    assert plan("3c01", "fp64", 32)[0] == 0 and plan("3c01", "fp64", 47)[0] == 0
    assert plan("3c01", "fp64", 61)[0] == 4


def test_two_warps_beside_the_largest_table(plan):
    assert plan("3c08", "fp64", 217, 27)[0] > 0
    for mcap in (226, 230, 236, 260):
        assert plan("3c08", "fp64", mcap, 27)[0] == 0
    assert plan("3c08", "fp32c", 260, 27)[0] > 0
