"""The product rule outside the deterministic mode (atm_prod.cuh) where it can go
wrong: three to many cells per axis, units of a few rows and of several words of
32 rows (both sides of a whole word, with remainders), two molecules closer than
any distance cut helps, molecules of one height, and a box of few units.
Counts are exact against the oracle's decisions in the same precision, forces and
energies within the 2e-5 (FP32C) and 1e-10 (FP64) of every parity test."""
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
@pytest.mark.parametrize("trav", ["3c01", "3c18", "3c08", "3c08a"])
@pytest.mark.parametrize("cells,rho,flat", [
    ((3, 3, 3), 0.8, False), ((4, 3, 5), 0.05, False), ((5, 4, 3), 0.25, True),
    ((3, 5, 4), 1.05, False), ((9, 3, 4), 0.01, False), ((7, 4, 3), 0.6, True)])
def test_against_oracle(atm3, trav, cells, rho, flat, prec, rtol):
    box, x = lattice(cells, rho, seed=sum(cells), flat=flat)
    n = x.shape[1]
    prm = oracle.params(box, RC, NU)
    ref = oracle.atm_cells(prm, x, trav, "product", "fp32" if prec == "fp32c" else prec)
    with atm3.AtmSystem(box, n, rc=RC, nu=NU) as s:
        s.set_state(x)
        s.build_cells()
        got = s.compute_forces(trav, "product", prec)
        f = s.get_forces("atm")
    for k in ("n_cand3", "n_int3"):
        assert got[k] == ref[k], k
    assert got["e3"] == pytest.approx(ref["e3"], rel=rtol)
    assert got["w3"] == pytest.approx(ref["w3"], rel=rtol)
    scale = np.sqrt(np.mean(ref["f"] ** 2))
    assert np.all(np.abs(f - ref["f"]) <= rtol * (np.abs(ref["f"]) + scale))


@pytest.mark.parametrize("prec", ["fp32c", "fp64"])
@pytest.mark.parametrize("gap", [0.2, 1e-2])
def test_a_close_pair(atm3, gap, prec):
    """The least distance bounds the rows: with a pair this close nothing is cut,
    and the counts are still the oracle's."""
    box, x = lattice((5, 4, 6), 0.3, seed=9)
    x[:, 1] = x[:, 0] + np.array([gap, 0.0, 0.0])
    x = np.mod(x, box[:, None])
    prm = oracle.params(box, RC, NU)
    for trav in ("3c01", "3c18", "3c08", "3c08a"):
        ref = oracle.atm_cells(prm, x, trav, "product", "fp32" if prec == "fp32c" else prec)
        with atm3.AtmSystem(box, x.shape[1], rc=RC, nu=NU) as s:
            s.set_state(x)
            s.build_cells()
            got = s.compute_forces(trav, "product", prec)
        assert (got["n_cand3"], got["n_int3"]) == (ref["n_cand3"], ref["n_int3"]), trav
