"""The pair histogram's kernel where it can go wrong: replicas that share a CTA (a
CTA takes 16 molecules), the last CTA ragged, more molecules than a warp a molecule
(4,096 CTAs), one bin and the most, a range far below the cell edge.  Counts are
exactly the oracle's."""
import numpy as np
import pytest

import oracle

pytestmark = pytest.mark.gpu

RC, NU = 2.5, 0.073


@pytest.mark.parametrize("sizes,box,r_max,nbins", [
    ((60, 130, 7, 93), 8.0, 2.5, 250), ((1, 2, 300), 7.7, 2.4, 1), ((70001,), 61.5, 2.5, 1000),
    ((20000,), 30.0, 0.05, 64)])
def test_counts_equal_the_oracle(sizes, box, r_max, nbins):
    import torch
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_2510_21230_gb300 import atm3, build
    build.build()
    rng = np.random.default_rng(sum(sizes))
    xs = [rng.uniform(0, box, (3, n)) for n in sizes]
    with atm3.AtmSystem(np.full((len(sizes), 3), box), list(sizes), rc=RC, nu=NU) as s:
        s.set_state(np.ascontiguousarray(np.concatenate(xs, 1)))
        s.build_cells()
        s.rdf_accumulate(r_max, nbins)
        counts, samples = s.rdf_get(nbins)
    assert samples == 1
    for r, x in enumerate(xs):
        ref = oracle.rdf_counts(oracle.params([box] * 3, RC, NU), x, r_max, nbins)
        assert np.array_equal(np.asarray(counts).reshape(len(sizes), nbins)[r], ref), r
