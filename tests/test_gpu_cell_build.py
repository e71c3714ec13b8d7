"""The cell build's quotients and orders where they can go wrong: coordinates on
the cell faces and a few units in the last place to either side of them, in the
last cell up to the box edge, zero (of either sign), subnormal, outside the box on
both sides, and cells of one to many more than 32 molecules.  Cells, starts and
orders are exactly those of float64 arithmetic."""
import numpy as np
import pytest

pytestmark = pytest.mark.gpu


def wrapped(x, L):
    t = x - np.floor(x / L) * L
    t = np.where(t < 0, t + L, t)
    t = np.where(t >= L, 0.0, t)
    return np.where((x >= 0) & (x < L), x, t)


@pytest.mark.parametrize("box,crowd", [((7.6, 7.6, 7.6), 1), ((9.1, 13.7, 77.3), 40), ((40.0, 25.3, 8.01), 200)])
def test_cells_are_exact(box, crowd):
    import torch
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_2510_21230_gb300 import atm3, build
    build.build()
    box = np.array(box)
    nc = np.floor(box / 2.5).astype(int)
    w = box / nc
    rng = np.random.default_rng(int(box.sum()))
    edge = []
    for d in range(3):
        vals = [0.0, -0.0, 5e-324, 1e-310, 1e-40, -1e-18, -box[d], 3.0 * box[d], -0.3 * box[d], 1.7 * box[d],
                np.nextafter(box[d], 0)]
        for k in range(nc[d] + 1):
            v = u = k * w[d]
            for _ in range(4):
                vals += [v, u]
                v, u = np.nextafter(v, np.inf), np.nextafter(u, -np.inf)
            vals += [k * w[d] * (1 + s * 2.0 ** -e) for s in (-1, 1) for e in (19, 20, 21, 22, 23, 24, 30)]
        edge.append(np.array(vals))
    m = max(len(e) for e in edge)
    x = np.stack([rng.permutation(np.resize(edge[d], m)) for d in range(3)])
    x = np.concatenate([x, rng.uniform(0, box[:, None], (3, 500)),
                        w[:, None] * (1 + 0.9 * rng.uniform(size=(3, crowd)))], 1)
    x = np.ascontiguousarray(x[:, rng.permutation(x.shape[1])])
    n = x.shape[1]
    with atm3.AtmSystem(box, n, rc=2.5, nu=0.073) as s:
        s.set_state(x)
        s.build_cells()
        got = s.get_cells()
    t = wrapped(x, box[:, None])
    c = np.minimum(np.floor(t / w[:, None]).astype(int), nc[:, None] - 1)
    cell = (c[2] * nc[1] + c[1]) * nc[0] + c[0]
    assert np.array_equal(got["ncell"], nc)
    assert np.array_equal(got["cell_of"], cell)
    assert np.array_equal(np.diff(got["cell_start"]), np.bincount(cell, minlength=int(np.prod(nc))))
    assert np.array_equal(got["perm"], np.argsort(cell, kind="stable"))
