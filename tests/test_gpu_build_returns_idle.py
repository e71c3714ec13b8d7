"""atm_build_cells synchronises the stream: when it returns, the sort too is done.
(A million cells: their scan alone takes longer than the call's return.)"""
import numpy as np
import pytest

pytestmark = pytest.mark.gpu


def test_the_stream_is_idle_after_a_build():
    torch = pytest.importorskip("torch")
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_2510_21230_gb300 import atm3, build
    build.build()
    n, box = 1000000, np.array([250.1, 250.2, 250.3])
    x = np.random.default_rng(3).uniform(0.0, 1.0, (3, n)) * box[:, None]
    st = torch.cuda.Stream()
    with atm3.AtmSystem(box, n, rc=2.5, nu=0.073, stream=st.cuda_stream) as s:
        s.set_state(x)
        for _ in range(5):
            s.build_cells()
            assert st.query()
