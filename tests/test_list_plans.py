"""The plans of the forward lists (forces.cu, asked on the CPU through the built library):
a plan that is not taken promises no LJ force either (its callers leave the LJ kernel out
for one that does), whatever kept it from being taken."""
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
    static uint2 list[1];
    atm3::List64Args l{};
    l.list = list;
    l.stride = 1 << 20;
    atm3::ForceJob j{};
    j.prec = atoi(a[1]);
    j.trav = atoi(a[2]);
    j.mcap_fwd = atoi(a[3]);
    j.optin = atoi(a[4]);
    j.lj = atoi(a[5]);
    j.lj_apart = !j.lj;
    j.l64 = &l;
    j.whole = true;
    j.b.ncell = 343;
    j.b.ntot = 5000;
    j.sms = 152;
    const atm3::FwdLaunch f = j.prec ? atm3::atm_fwd_plan(j) : atm3::atm_list64_plan(j);
    std::printf("%d %d\n", f.use ? 1 : 0, f.lj);
}
"""


@pytest.fixture(scope="module")
def plan(tmp_path_factory):
    nvcc = os.path.join(os.environ.get("CUDA_HOME", "/usr/local/cuda"), "bin", "nvcc")
    if not os.path.exists(nvcc):
        nvcc = shutil.which("nvcc")
    if nvcc is None:
        pytest.skip("no nvcc")
    from paper_2510_21230_gb300 import build
    lib = build.build()
    d = tmp_path_factory.mktemp("lists")
    (d / "plan.cu").write_text(PROGRAM)
    subprocess.run([nvcc, "-std=c++17", "-I", os.path.join(PKG, "csrc"), "-I", os.path.join(ROOT, "include"),
                    str(d / "plan.cu"), lib, "-Xlinker", "-rpath", "-Xlinker", PKG, "-o", str(d / "plan")],
                   check=True, capture_output=True)
    return lambda *a: tuple(map(int, subprocess.run([str(d / "plan"), *map(str, a)], check=True, capture_output=True,
                                                    text=True).stdout.split()))


@pytest.mark.parametrize("prec", [0, 1])
@pytest.mark.parametrize("trav", [0, 1, 2])
@pytest.mark.parametrize("lj", [0, 1])
def test_lists_that_are_not_taken_give_no_lj(plan, prec, trav, lj):
    if trav == 0 and lj:
        return  # (steps of 3c01 keep LJ apart)
    assert plan(prec, trav, 250, 232448, lj) == (1, 1 if lj else 2)
    assert plan(prec, trav, 60000, 232448, lj) == (0, 0)
    if prec:
        assert plan(prec, trav, 250, 6000, lj) == (0, 0)     # (a device with little shared memory)
