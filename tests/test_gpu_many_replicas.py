"""Reductions of many small replicas: an evaluation of 400 replicas of 130 molecules costs
less than two and a half times one system of as many (5.1 times while every thread of every
partial sum met an FP64 division, 16 cycles of the SM's pipe an instruction), and gives the
replicas' own sums."""
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


def test_cost_of_many_replicas(atm3):
    import torch

    def best(boxes, ns, x):
        with atm3.AtmSystem(boxes, ns, stream=torch.cuda.current_stream().cuda_stream) as s:
            s.set_state(x)
            s.build_cells()
            s.surrogate_set_model(synth.sur_params(7), np.zeros(32, np.float32), np.ones(32, np.float32))
            t = np.inf
            for _ in range(12):
                a, b = torch.cuda.Event(enable_timing=True), torch.cuda.Event(enable_timing=True)
                a.record()
                for _ in range(5):
                    s.compute_forces("3c08", "pair", "surrogate", sync=False)
                b.record()
                torch.cuda.synchronize()
                t = min(t, a.elapsed_time(b))
        return t

    cfg = [synth.homogeneous(130, 0.3, 1.0, seed=k) for k in range(400)]
    many = best([c["box"] for c in cfg], [c["n"] for c in cfg], np.concatenate([c["x"] for c in cfg], axis=1))
    one = synth.homogeneous(52000, 0.3, 1.0, seed=1)
    assert many < 2.5 * best(one["box"], one["n"], one["x"])


@pytest.mark.parametrize("trav,trunc,prec,rtol", [("3c08", "pair", "fp64", 1e-12), ("3c01", "pair", "fp64", 1e-12),
                                                  ("3c18", "pair", "fp32c", 1e-6), ("3c08", "product", "fp64", 1e-12)])
def test_sums_of_small_and_large_replicas(atm3, trav, trunc, prec, rtol):
    """Slices of up to 32 entries and of more take different trees."""
    cfg = [synth.homogeneous(n, 0.6, 1.0, seed=n) for n in (600, 2100, 3000)]
    alone = []
    for c in cfg:
        with atm3.AtmSystem(c["box"], c["n"]) as s:
            s.set_state(c["x"], c["v"])
            s.build_cells()
            alone.append(s.compute_forces(trav, trunc, prec))
    with atm3.AtmSystem([c["box"] for c in cfg], [c["n"] for c in cfg]) as s:
        s.set_state(np.concatenate([c["x"] for c in cfg], axis=1), np.concatenate([c["v"] for c in cfg], axis=1))
        s.build_cells()
        s.compute_forces(trav, trunc, prec)
        batch = s.results()
    for a, b in zip(alone, batch):
        for k in ("n_cand3", "n_int3", "n_cand2", "n_int2"):
            assert a[k] == b[k], k
        for k in ("e2", "e3", "w2", "w3", "ekin"):
            assert b[k] == pytest.approx(a[k], rel=rtol, abs=rtol * abs(a["e2"])), k
