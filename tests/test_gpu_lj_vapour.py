"""The LJ kernel where most cells are empty (a CTA then takes several): molecules scattered
over 8,000 to 64,000 cells, alone, in parts of a domain and as replicas of a batch, against
the oracle as in every parity test; and a vapour's evaluation does not pay for its cells."""
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


def pairs(cells, n, seed):
    """n molecules on random sites of a jittered lattice (1.27 apart), mostly two by two."""
    rng = np.random.default_rng(seed)
    box, per = np.full(3, cells * RC * 1.013), 2 * cells
    sites = []
    seen = set()
    while len(sites) < n:
        a = rng.integers(0, per, 3)
        for b in (a, (a + [1, 0, 0]) % per):
            if tuple(b) not in seen:
                seen.add(tuple(b))
                sites.append(b)
    g = np.array(sites[:n])
    return box, np.ascontiguousarray(((g + 0.5 + rng.uniform(-0.1, 0.1, g.shape)) * (box / per)).T)


def close(f, want, rtol):
    assert np.all(np.abs(f - want) <= rtol * (np.abs(want) + np.sqrt(np.mean(want ** 2))))


@pytest.mark.parametrize("prec,rtol", [("fp32c", 2e-5), ("fp64", 1e-10)])
@pytest.mark.parametrize("cells,n", [(20, 61), (20, 4001), (40, 500), (20, 7999)])
def test_against_oracle(atm3, cells, n, prec, rtol):
    box, x = pairs(cells, n, cells + n)
    prm = oracle.params(box, RC, NU)
    lj = oracle.lj_cells(prm, x, "fp32" if prec == "fp32c" else prec)
    with atm3.AtmSystem(box, n, rc=RC, nu=NU) as s:
        s.set_state(x)
        s.build_cells()
        got = s.compute_forces("3c08a", "pair", prec)
        f = s.get_forces("lj")
        assert (got["n_cand2"], got["n_int2"]) == (lj["n_cand2"], lj["n_int2"])
        assert got["e2"] == pytest.approx(lj["e2"], rel=rtol)
        close(f, lj["f"], rtol)
        # two parts of a domain add up to the whole
        f2, c2, i2 = np.zeros_like(f), 0, 0
        for lo, hi in ((0, 7), (7, cells)):
            s.set_owned_layers(lo, hi)
            r = s.compute_forces("3c08a", "pair", prec)
            f2, c2, i2 = f2 + s.get_forces("lj"), c2 + r["n_cand2"], i2 + r["n_int2"]
    assert (c2, i2) == (lj["n_cand2"], lj["n_int2"])
    close(f2, lj["f"], rtol)


def test_replicas(atm3):
    sys = [pairs(c, n, n) for c, n in ((20, 50), (12, 300), (15, 41))]
    with atm3.AtmSystem([b for b, _ in sys], [x.shape[1] for _, x in sys], rc=RC, nu=NU) as s:
        s.set_state(np.concatenate([x for _, x in sys], axis=1))
        s.build_cells()
        s.compute_forces("3c08a", "pair", "fp64")
        f, res, at = s.get_forces("lj"), s.results(), 0
    for (box, x), r in zip(sys, res):
        lj = oracle.lj_cells(oracle.params(box, RC, NU), x)
        assert (r["n_cand2"], r["n_int2"]) == (lj["n_cand2"], lj["n_int2"])
        close(f[:, at:at + x.shape[1]], lj["f"], 1e-10)
        at += x.shape[1]


def test_a_vapour_does_not_pay_for_its_cells(atm3):
    """20 molecules in a million cells: LJ took 870 us with a CTA for every cell."""
    box, x = pairs(100, 20, 3)
    with atm3.AtmSystem(box, 20, rc=RC, nu=NU) as s:
        s.set_state(x)
        s.build_cells()
        s.set_profiling(True)
        for _ in range(12):
            s.compute_forces("3c08a", "pair", "fp64")
        p = s.get_profile()
    print(p)
    assert p["ms_lj"] / 12 < 0.2
