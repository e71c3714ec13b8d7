"""Surrogate evaluations of liquids with three cells an axis, up to 4/3 r_c wide: their
cells hold more than 32 molecules here and there, and the descriptors of a molecule must not
fall back to a direct pass for that.  (Per molecule 1.5 times the time of cells of 13; the
direct pass took 2.6 times.)"""
import numpy as np
import pytest

from paper_2510_21230_gb300 import synth

pytestmark = pytest.mark.gpu


def test_cells_over_32_cost_less_than_twice_per_molecule():
    torch = pytest.importorskip("torch")
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_2510_21230_gb300 import atm3, build
    build.build()

    def per_molecule(n, rho):
        cfg = [synth.homogeneous(n, rho, 1.0, seed=k) for k in range(40)]
        x = np.concatenate([c["x"] for c in cfg], axis=1)
        with atm3.AtmSystem([c["box"] for c in cfg], [c["n"] for c in cfg],
                            stream=torch.cuda.current_stream().cuda_stream) as s:
            s.set_state(x)
            s.build_cells()
            occ = np.diff(s.get_cells()["cell_start"]).max()
            s.surrogate_set_model(synth.sur_params(7), np.zeros(32, np.float32), np.ones(32, np.float32))
            best = np.inf
            for _ in range(12):
                a, b = torch.cuda.Event(enable_timing=True), torch.cuda.Event(enable_timing=True)
                a.record()
                for _ in range(5):
                    s.compute_forces("3c08", "pair", "surrogate", sync=False)
                b.record()
                torch.cuda.synchronize()
                best = min(best, a.elapsed_time(b))
        return best / x.shape[1], occ

    wide, most = per_molecule(700, 0.85)
    narrow, few = per_molecule(864, 0.8)
    assert 32 < most <= 48 and few <= 32
    assert wide < 2.0 * narrow
