"""The LJ kernel of the evaluations that do not take it inside the lists or units
(k_lj_owner) where it can go wrong: neighbourhoods of a few molecules, of more than
one tile of 512, cells of one to many more than the 16 molecules a CTA takes at a
time, sparse systems with empty cells.  Counts are exact against the oracle's
decisions in the same precision, forces and sums within 2e-5 (FP32C) and 1e-10
(FP64) as in every parity test."""
import numpy as np
import pytest

import oracle

pytestmark = pytest.mark.gpu

RC, NU = 2.5, 0.073


def lattice(cells, rho, seed):
    box = np.array(cells) * RC * 1.013
    per = np.maximum(1, np.floor(box * rho ** (1.0 / 3.0)).astype(int))
    rng = np.random.default_rng(seed)
    g = np.stack(np.meshgrid(*[np.arange(k) for k in per], indexing="ij"), -1).reshape(-1, 3)
    x = (g + 0.5 + rng.uniform(-0.1, 0.1, g.shape)) * (box / per)
    return box, np.ascontiguousarray(x.T[:, rng.permutation(len(x))])


@pytest.mark.parametrize("prec,rtol", [("fp32c", 2e-5), ("fp64", 1e-10)])
@pytest.mark.parametrize("cells,rho", [((3, 3, 3), 0.02), ((5, 3, 4), 0.8), ((3, 4, 3), 1.25), ((4, 3, 3), 4.0),
                                       ((9, 8, 7), 0.004)])
def test_lj_apart_equals_the_oracle(cells, rho, prec, rtol):
    import torch
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_2510_21230_gb300 import atm3, build
    build.build()
    box, x = lattice(cells, rho, seed=sum(cells))
    lj = oracle.lj_cells(oracle.params(box, RC, NU), x, "fp32" if prec == "fp32c" else prec)
    with atm3.AtmSystem(box, x.shape[1], rc=RC, nu=NU) as s:
        s.set_state(x)
        s.build_cells()
        got = s.compute_forces("3c08a", "pair", prec)
        f = s.get_forces("lj")
    assert (got["n_cand2"], got["n_int2"]) == (lj["n_cand2"], lj["n_int2"])
    assert got["e2"] == pytest.approx(lj["e2"], rel=rtol)
    assert got["w2"] == pytest.approx(lj["w2"], rel=rtol, abs=rtol * abs(lj["e2"]))
    scale = np.sqrt(np.mean(lj["f"] ** 2))
    assert np.all(np.abs(f - lj["f"]) <= rtol * (np.abs(lj["f"]) + scale))
