"""FP64 graph steps while the units of the forward lists grow: beyond the rows that
were allocated (new buffers under a live graph), and beyond the 32 molecules a cell
that the lists can hold (during the steps).  Counts and states are those of steps
without a graph and of the oracle (1e-10 of every FP64 parity test)."""
import numpy as np
import pytest

import oracle

pytestmark = pytest.mark.gpu

RC = 2.5


@pytest.fixture(scope="module")
def atm3():
    import torch
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_2510_21230_gb300 import atm3 as m, build
    build.build()
    return m


def grid(lo, hi, per, rng, jitter=0.02):
    """Jittered points of a per[0] x per[1] x per[2] grid inside [lo, hi)."""
    g = np.stack(np.meshgrid(*[np.arange(k) for k in per], indexing="ij"), -1).reshape(-1, 3)
    h = (np.asarray(hi) - lo) / per
    return (lo + (g + 0.5 + rng.uniform(-jitter, jitter, g.shape)) * h).T


def run(atm3, box, states, steps, graph, **kw):
    out = []
    with atm3.AtmSystem(box, states[0][0].shape[1], rc=RC, **kw) as s:
        s.set_options(graph=graph)
        for x, v in states:
            s.set_state(x, v)
            r = s.step(steps, "3c08", "pair", "fp64")
            out.append((r, *s.get_state(), s.get_forces("total")))
    return out


def compare(got, ref):
    for (r, x, v, f), (r0, x0, v0, f0) in zip(got, ref):
        assert (r["n_cand3"], r["n_int3"], r["n_int2"]) == (r0["n_cand3"], r0["n_int3"], r0["n_int2"])
        assert r["e3"] == pytest.approx(r0["e3"], rel=1e-10)
        for a, b in ((x, x0), (v, v0), (f, f0)):
            assert np.all(np.abs(a - b) <= 1e-10 * (np.abs(b) + np.sqrt(np.mean(b ** 2))))


def test_rows_grow_under_a_live_graph(atm3):
    rng = np.random.default_rng(5)
    box = np.full(3, 4 * RC * 1.02)
    thin = grid(np.zeros(3), box, (6, 6, 6), rng)
    dense = grid(np.zeros(3), box * 0.55, (6, 6, 6), rng)      # the same molecules in fewer cells
    v = rng.normal(0.0, 0.5, thin.shape)
    states = [(thin, v), (dense, v), (thin, v), (dense, v)]
    kw = dict(nu=0.073, dt=0.0005)
    got = run(atm3, box, states, 5, True, **kw)
    compare(got, run(atm3, box, states, 5, False, **kw))
    for (r, x, _, f), (x0, v0) in zip(got, states):
        ref = oracle.md_run(oracle.params(box, RC, 0.073), x0, v0, 5, 0.0005, "3c08", "pair", "fp64")
        d = x - ref["x"]
        d -= box[:, None] * np.round(d / box[:, None])
        assert np.abs(d).max() <= 1e-10
        assert np.all(np.abs(f - ref["f"]) <= 1e-9 * (np.abs(ref["f"]) + np.sqrt(np.mean(ref["f"] ** 2))))


def test_a_cell_fills_beyond_32_during_graph_steps(atm3):
    rng = np.random.default_rng(6)
    w = RC * 1.02
    box = np.full(3, 4 * w)
    here = grid(np.array([w, w, w]), np.array([2 * w, 2 * w, 2 * w]), (3, 4, 2), rng)         # 24 that stay
    come = grid(np.array([0.5 * w, w, w]), np.array([0.99 * w, 2 * w, 2 * w]), (2, 4, 2), rng)  # 16 that come
    x = np.concatenate([here, come], axis=1)
    v = np.zeros_like(x)
    v[0, here.shape[1]:] = 100.0       # 0.2 a step: all of them inside within 7 steps
    kw = dict(nu=1e-9, lj_eps=0.0, dt=0.002)
    states = [(x, v), (x, v)]
    got = run(atm3, box, states, 7, True, **kw)
    compare(got, run(atm3, box, states, 7, False, **kw))
    ref = oracle.md_run(oracle.params(box, RC, 1e-9, 0.0), x, v, 7, 0.002, "3c08", "pair", "fp64")
    end = oracle.build_cells(oracle.params(box, RC, 1e-9, 0.0), ref["x"])
    assert np.diff(end["cell_start"]).max() > 32
    for r, xx, _, f in got:
        d = xx - ref["x"]
        d -= box[:, None] * np.round(d / box[:, None])
        assert np.abs(d).max() <= 1e-10
        assert np.all(np.abs(f - ref["f"]) <= 1e-9 * (np.abs(ref["f"]) + np.sqrt(np.mean(ref["f"] ** 2))))
