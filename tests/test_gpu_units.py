"""FP64 evaluations in units far from 1 (lengths in metres, say: r_c of 1e-9).  The
kernels test in FP32 first, where squares and products of six lengths may leave its
range; what FP32 cannot decide is decided in FP64, so every scale gives the oracle's
counts, forces and energies within the 1e-10 of every parity test.  Lengths are
scaled by a power of two, nu by its ninth power, which is exact: counts and energies
are the oracle's at scale 1, forces those divided by the scale.  (The triplet terms'
own q^5, a fifteenth power, bounds the scales at 2^+-65; cells, LJ and the pair
histogram go on.)"""
import numpy as np
import pytest

import oracle

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def atm3():
    import torch
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_2510_21230_gb300 import atm3 as m, build
    build.build()
    return m


def system(exp):
    s = 2.0 ** exp
    rng = np.random.default_rng(11)
    box = np.array([4, 3, 5]) * 2.5 * 1.013
    per = np.floor(box * 0.6 ** (1.0 / 3.0)).astype(int)
    g = np.stack(np.meshgrid(*[np.arange(k) for k in per], indexing="ij"), -1).reshape(-1, 3)
    x = (g + 0.5 + rng.uniform(-0.1, 0.1, g.shape)) * (box / per)
    return box * s, np.ascontiguousarray(x.T[:, rng.permutation(len(x))]) * s, 2.5 * s, s


def close(got, want, rtol=1e-10):
    scale = np.sqrt(np.mean((want / np.abs(want).max()) ** 2)) * np.abs(want).max()
    assert np.all(np.abs(got - want) <= rtol * (np.abs(want) + scale))


@pytest.mark.parametrize("trav,trunc", [("3c08", "pair"), ("3c01", "pair"), ("3c08", "product"),
                                        ("3c01", "product"), ("3c18", "product"), ("3c08a", "product")])
@pytest.mark.parametrize("exp", [-65, -30, 20, 65])
def test_triplets(atm3, exp, trav, trunc):
    b1, x1, r1, _ = system(0)
    box, x, rc, s = system(exp)
    nu = 0.073 * s ** 9
    prm = oracle.params(b1, r1, 0.073)
    ref, lj = oracle.atm_cells(prm, x1, trav, trunc, "fp64"), oracle.lj_cells(prm, x1, "fp64")
    with atm3.AtmSystem(box, x.shape[1], rc=rc, nu=nu, lj_sigma=s) as c:
        c.set_state(x)
        c.build_cells()
        got = c.compute_forces(trav, trunc, "fp64")
        f, f2 = c.get_forces("atm"), c.get_forces("lj")
    assert (got["n_cand3"], got["n_int3"]) == (ref["n_cand3"], ref["n_int3"])
    assert (got["n_cand2"], got["n_int2"]) == (lj["n_cand2"], lj["n_int2"])
    assert got["e3"] == pytest.approx(ref["e3"], rel=1e-10, abs=0)
    assert got["w3"] == pytest.approx(ref["w3"], rel=1e-10, abs=0)
    close(f * s, ref["f"])
    close(f2 * s, lj["f"])


@pytest.mark.parametrize("exp", [-140, -126, -66, 66, 125, 130])
def test_cells_pairs_and_histogram(atm3, exp):
    b1, x1, r1, _ = system(0)
    box, x, rc, s = system(exp)
    prm = oracle.params(b1, r1, 0.0)
    lj, cells = oracle.lj_cells(prm, x1, "fp64"), oracle.build_cells(prm, x1)
    with atm3.AtmSystem(box, x.shape[1], rc=rc, nu=0.0, lj_sigma=s) as c:
        c.set_state(x)
        c.build_cells()
        got = c.get_cells()
        c.rdf_accumulate(rc, 40)
        hist = c.rdf_get(40)
        r = c.compute_forces("3c08", "product", "fp64")
        f = c.get_forces("lj")
    for k in ("cell_of", "cell_start", "perm"):
        assert np.array_equal(np.asarray(got[k]).ravel(), np.asarray(cells[k]).ravel()), k
    assert np.array_equal(np.asarray(hist[0]).ravel().astype(np.int64),
                          np.asarray(oracle.rdf_counts(prm, x1, r1, 40)).ravel().astype(np.int64))
    assert (r["n_cand2"], r["n_int2"]) == (lj["n_cand2"], lj["n_int2"])
    close(f * s, lj["f"])
