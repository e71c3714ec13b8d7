"""Accuracy of the FP32C forces of 3c01, from positions whose cell-local coordinates and
displacements are FP32 numbers, so that nothing is lost before the triplet terms: rms
error against FP64 sums over rms force no larger than that of the owner kernel, which
evaluates canonical displacements and adds F_i with compensation (measured there, the
same positions; 2 % for the order of the additions)."""
import numpy as np
import pytest

pytestmark = pytest.mark.gpu

W, NCELL, RC, NU = 4.0, 4, 3.99, 0.073


@pytest.fixture(scope="module")
def atm3():
    import torch
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_2510_21230_gb300 import atm3 as m, build
    build.build()
    return m


def positions(n, seed):
    """n molecules at least 0.9 apart on multiples of 2^-22 (24 bits of a cell edge of 4)."""
    rng = np.random.default_rng(seed)
    box, x = W * NCELL, np.zeros((0, 3))
    while len(x) < n:
        t = np.floor(rng.uniform(0.0, box, 3) * 2 ** 22) / 2 ** 22
        d = x - t
        d -= box * np.round(d / box)
        if np.all((d * d).sum(1) > 0.81):
            x = np.vstack([x, t])
    return np.ascontiguousarray(x.T)


def owner_forces(x, trunc):
    """3c01's forces in FP64 and the owner visits."""
    box, n = W * NCELL, x.shape[1]
    cell = np.floor(x / W).astype(int)
    f, visits = np.zeros((3, n)), 0
    rc2, rc6 = RC ** 2, RC ** 6
    for p in range(n):
        o = (cell - cell[:, p:p + 1] + 1) % NCELL - 1        # cell offset, -1 .. 2
        near = np.all(o <= 1, axis=0)
        near[p] = False
        d = (x - cell * W) - (x[:, p:p + 1] - cell[:, p:p + 1] * W) + o * W
        d = d[:, near]
        a = (d * d).sum(0)
        if trunc == "pair":
            d, a = d[:, a < rc2], a[a < rc2]
        j, k = np.triu_indices(d.shape[1], 1)
        e = d[:, k] - d[:, j]
        c = (e * e).sum(0)
        keep = c < rc2 if trunc == "pair" else a[j] * a[k] * c < rc6
        dj, dk, e = (v[:, keep] for v in (d[:, j], d[:, k], e))
        a, b, c = ((v * v).sum(0) for v in (dj, dk, e))
        A, B, C = b + c - a, a + c - b, a + b - c
        q = 1.0 / np.sqrt(a * b * c)
        q2 = q * q
        nq5, K = NU * (q * q2) * q2, 1.5 + 0.9375 * (A * B * C * q2)
        ga = 2.0 * nq5 * (0.375 * (2.0 * a * A - B * C) - K * (b * c))
        gb = 2.0 * nq5 * (0.375 * (2.0 * b * B - A * C) - K * (a * c))
        f[:, p] = (ga * dj).sum(1) + (gb * dk).sum(1)
        visits += int(keep.sum())
    return f, visits


# (truncation, molecules): rms error of the owner kernel over the same twelve systems
OWNER = {("product", 320): 3.147e-7, ("pair", 900): 2.653e-7}


@pytest.mark.parametrize("trunc,n", sorted(OWNER))
def test_as_close_as_the_owner_kernel(atm3, trunc, n):
    errors = []
    for k in range(12):
        x = positions(n, 1000 * k + n)
        want, visits = owner_forces(x, trunc)
        with atm3.AtmSystem(np.full(3, W * NCELL), n, rc=RC, nu=NU) as s:
            s.set_state(x)
            s.build_cells()
            got = s.compute_forces("3c01", trunc, "fp32c")
            f = s.get_forces("atm")
        assert got["n_int3"] == visits
        errors.append(np.mean((f - want) ** 2) / np.mean(want ** 2))
    assert np.sqrt(np.mean(errors)) <= 1.02 * OWNER[trunc, n]
