"""Training batches drawn inside the tensor-core kernel: the loss of a step equals
the loss over the same rows handed in one by one.

The row of element b of step k is a fixed function of (seed, k, b), restated here.
Both sides run the same arithmetic on the same tiles, and the loss is summed in
double precision, so they agree to the FP32 rounding of its scale (1e-6).  Batch
sizes: one sample, both sides of a tile's 128, one past the tiles that run at a
time, and ragged ones."""
import numpy as np
import pytest

from paper_2510_21230_gb300 import synth

pytestmark = pytest.mark.gpu

M64 = (1 << 64) - 1


def _mix(z):
    z = ((z ^ (z >> 30)) * 0xBF58476D1CE4E5B9) & M64
    z = ((z ^ (z >> 27)) * 0x94D049BB133111EB) & M64
    return z ^ (z >> 31)


def _rows(seed, step, batch, n):
    z = _mix((seed + 0x9E3779B97F4A7C15 * (step + 1)) & M64)
    return [_mix((z + 0x9E3779B97F4A7C15 * (b + 1)) & M64) % n for b in range(batch)]


@pytest.mark.parametrize("n,batch", [(1537, 1), (1537, 127), (1537, 128), (1537, 129), (1537, 300), (1537, 1000),
                                     (1537, 152 * 128 + 1), (20000, 152 * 128 + 1)])
def test_sampled_batch_equals_its_rows(n, batch):
    import torch
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_2510_21230_gb300 import atm3, build
    build.build()
    seed = 5
    P = synth.sur_params(61)
    mean = np.linspace(-0.5, 0.5, 32).astype(np.float32)
    scale = np.linspace(0.7, 1.5, 32).astype(np.float32)
    D, V, T = synth.sur_rows(n, 62, mean, scale)
    T = np.asarray(T, dtype=np.float32).reshape(n, 3)
    # a batch of all rows or more is the data set itself
    idx = np.array(_rows(seed, 0, batch, n)) if batch < n else np.arange(n)
    with atm3.AtmSystem(10.0, 1, rc=2.5, nu=0.073) as s:
        s.surrogate_set_model(P, mean, scale)
        s.surrogate_add_rows(D, V, T)
        _, s2 = s.surrogate_dataset()
        want, _ = s.surrogate_loss_grad(np.asarray(D).reshape(n, -1)[idx], np.asarray(V).reshape(n, -1)[idx],
                                        T[idx], s2)
        got = s.surrogate_train(1, batch=batch, lr=1e-3, seed=seed)[0]
    assert abs(got - want) <= 1e-6 * want, (batch, got, want)
