"""FP64 forces and energies of triangles with one side short against the others: 64
triangles apart from each other, each a pair of molecules at 0.1 to 1e-3 of a length unit
and a third one within r_c, some across faces of cells and of the box.  Against the same
sums in extended precision within the 1e-10 of every parity test, of the largest force of
a triangle.  (Displacements of three roundings of lengths up to L = 41 leave 2e-11 at 1e-3;
a third side by cancellation, c = a + b - 2 d_j d_k, 1e-8.)"""
import numpy as np
import pytest

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


def triangles(gap):
    """box, and the molecules i, j, k of 64 triangles, every fourth cell per axis
    (so that no unit of cells meets two)."""
    w = RC * 1.013
    box = np.full(3, 16 * w)
    rng = np.random.default_rng(23)
    g = np.stack(np.meshgrid(*[np.arange(4)] * 3, indexing="ij"), -1).reshape(-1, 3).T
    unit = lambda m: (lambda v: v / np.sqrt((v * v).sum(0)))(rng.normal(size=(3, m)))
    i = (4 * g + rng.uniform(0.0, 1.0, g.shape)) * w
    j = i + rng.uniform(1.0, 2.3, 64) * unit(64)
    return box, [np.mod(v, box[:, None]) for v in (i, j, j + gap * unit(64))]


def extended(box, t):
    """Forces on i, j, k and energies in extended precision (u in r^2 form:
    nu q^3 (1 + 3 x y m q^2), q = (a b c)^(-1/2), x, y, m the dot products at the corners)."""
    T = np.longdouble

    def d(p, q):
        v, L = q.astype(T) - p.astype(T), box[:, None].astype(T)
        return np.where(v > L / 2, v - L, np.where(v < -L / 2, v + L, v))
    i, j, k = t
    dj, dk, e = d(i, j), d(i, k), d(j, k)
    dot = lambda u, v: (u * v).sum(0)
    a, b, c, x, y, m = dot(dj, dj), dot(dk, dk), dot(e, e), -dot(dj, e), dot(dk, e), dot(dj, dk)
    q2 = 1 / (a * b * c)
    q = np.sqrt(q2)
    p = x * y * m * q2
    q5 = 3 * T(NU) * q * q2 * q2
    ga = q5 * (a * y - x * m - (1 + 5 * p) * b * c)
    gb = q5 * (b * x - y * m - (1 + 5 * p) * a * c)
    gc = q5 * (c * m - x * y - (1 + 5 * p) * a * b)
    return [ga * dj + gb * dk, -ga * dj + gc * e, -gb * dk - gc * e], T(NU) * q * q2 * (1 + 3 * p)


@pytest.mark.parametrize("trav,trunc", [("3c01", "pair"), ("3c18", "pair"), ("3c08", "pair"), ("3c01", "product"),
                                        ("3c18", "product"), ("3c08", "product")])
@pytest.mark.parametrize("gap", [0.1, 1e-2, 1e-3])
def test_against_extended_precision(atm3, gap, trav, trunc):
    box, t = triangles(gap)
    want, u = extended(box, t)
    x = np.ascontiguousarray(np.concatenate(t, axis=1))
    with atm3.AtmSystem(box, x.shape[1], rc=RC, nu=NU) as s:
        s.set_state(x)
        s.build_cells()
        got = s.compute_forces(trav, trunc, "fp64")
        f = s.get_forces("atm").reshape(3, 3, 64)
    assert got["n_int3"] == 64 * (3 if trav == "3c01" else 1)
    assert abs(got["e3"] - float(u.sum())) <= 1e-10 * float(np.abs(u).sum())
    assert abs(got["w3"] - 9 * float(u.sum())) <= 9e-10 * float(np.abs(u).sum())
    largest = np.max([np.sqrt((v * v).sum(0)) for v in want], axis=0)
    for c in range(3):
        assert np.all(np.abs(f[:, c, :] - want[c]) <= 1e-10 * largest)
