"""The pair rule from forward lists (atm_fwd.cuh, atm_list64.cu) where it can go wrong:
three to many cells per axis and runs of cells with every remainder, lists of a
few rows, around the 32 a warp holds, beyond the rows met one by one, and
beyond the warp's row table; molecules at equal heights (a layer's order is by
height); systems of few cells (several CTAs per cell) and of many (runs).
Counts are exact against the oracle's decisions in the same precision, forces
and energies within the 2e-5 (FP32C) and 1e-10 (FP64) of every parity test.
(FP64 lists need cells of at most 32 molecules: the densest case takes the
block kernel there.)"""
import numpy as np
import pytest

import oracle

pytestmark = pytest.mark.gpu

RC, NU = 2.5, 0.073


@pytest.fixture(scope="module")
def atm3():
    import torch
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_2510_21230_gb300 import atm3 as m, build
    build.build()
    return m


def lattice(cells, rho, seed, flat=False):
    """A jittered simple cubic lattice at density rho in a box of that many
    cells per axis; flat: the layers of the lattice keep one height each."""
    box = np.array(cells) * RC * 1.013
    per = np.maximum(1, np.floor(box * rho ** (1.0 / 3.0)).astype(int))
    rng = np.random.default_rng(seed)
    g = np.stack(np.meshgrid(*[np.arange(k) for k in per], indexing="ij"), -1).reshape(-1, 3)
    x = (g + 0.5 + rng.uniform(-0.1, 0.1, g.shape) * ([1, 1, 0] if flat else 1)) * (box / per)
    return box, np.ascontiguousarray(x.T[:, rng.permutation(len(x))])


@pytest.mark.parametrize("prec,rtol", [("fp32c", 2e-5), ("fp64", 1e-10)])
@pytest.mark.parametrize("trav", ["3c01", "3c18", "3c08"])
@pytest.mark.parametrize("cells,rho,flat", [
    ((3, 3, 3), 0.8, False), ((4, 3, 5), 0.05, False), ((5, 4, 3), 0.8, True),
    ((3, 5, 4), 1.05, False), ((6, 3, 3), 1.2, False), ((7, 4, 3), 1.5, True),
    ((4, 4, 4), 2.6, False), ((31, 20, 20), 0.1, False), ((6, 34, 30), 0.3, True)])
def test_against_oracle(atm3, trav, cells, rho, flat, prec, rtol):
    box, x = lattice(cells, rho, seed=sum(cells), flat=flat)
    n = x.shape[1]
    prm = oracle.params(box, RC, NU)
    orc = "fp32" if prec == "fp32c" else prec
    ref, lj = oracle.atm_cells(prm, x, trav, "pair", orc), oracle.lj_cells(prm, x, orc)
    with atm3.AtmSystem(box, n, rc=RC, nu=NU) as s:
        s.set_state(x)
        s.build_cells()
        apart = s.compute_forces(trav, "pair", prec)
        f = {w: s.get_forces(w) for w in ("lj", "atm", "total")}
        inside = s.step(0, trav, "pair", prec)
        f["step"] = s.get_forces("total")
        runs = [apart, inside]
        if prec == "fp32c":  # (the deterministic FP64 sums are the block kernel's)
            s.set_deterministic(True)
            runs.append(s.compute_forces(trav, "pair", prec))
            f["det"] = s.get_forces("atm")
    for r in runs:
        for k in ("n_cand3", "n_int3"):
            assert r[k] == ref[k], k
        for k in ("n_cand2", "n_int2"):
            assert r[k] == lj[k], k
        assert r["e3"] == pytest.approx(ref["e3"], rel=rtol)
        assert r["w3"] == pytest.approx(ref["w3"], rel=rtol)
        assert r["e2"] == pytest.approx(lj["e2"], rel=rtol)
        assert r["w2"] == pytest.approx(lj["w2"], rel=rtol, abs=rtol * abs(lj["e2"]))
    want = {"lj": lj["f"], "atm": ref["f"], "det": ref["f"], "total": lj["f"] + ref["f"],
            "step": lj["f"] + ref["f"]}
    for w, got in f.items():
        scale = np.sqrt(np.mean(want[w] ** 2))
        assert np.all(np.abs(got - want[w]) <= rtol * (np.abs(want[w]) + scale)), w
