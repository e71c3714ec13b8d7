"""Descriptors of small systems (a warp to a molecule) and of large ones (a
thread to a molecule) are the same bit for bit: a system alone and inside a
batch that is large enough for the other kernel, for molecule counts at the
edges of warps and blocks, sparse and crowded cells (more than 32 molecules)."""
import numpy as np
import pytest

from paper_2510_21230_gb300 import synth

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def atm3():
    import torch
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_2510_21230_gb300 import atm3 as m, build
    build.build()
    return m


@pytest.mark.parametrize("n,rho", [(1, 0.001), (33, 0.05), (127, 0.2), (1003, 0.8), (2000, 2.4)])
def test_same_descriptors(atm3, n, rho):
    a = synth.homogeneous(n, rho, 1.0, seed=n)
    b = synth.homogeneous(45000, 0.5, 1.0, seed=1)
    with atm3.AtmSystem(a["box"], n) as s:
        s.set_state(a["x"])
        s.build_cells()
        alone = s.surrogate_descriptors()
    with atm3.AtmSystem([a["box"], b["box"]], [n, b["n"]]) as s:
        s.set_state(np.concatenate([a["x"], b["x"]], axis=1))
        s.build_cells()
        batch = s.surrogate_descriptors()
    for x, y in zip(alone, batch):
        assert np.array_equal(x, y[:n])
    assert n < 2 or np.abs(alone[0]).max() > 0
