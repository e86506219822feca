"""FP32 gradient on a grid with more rows of tiles than a launch grid has blocks in y."""
import numpy as np
import pytest

import workloads as W

pytestmark = pytest.mark.gpu


def test_more_than_65535_rows_of_tiles():
    import torch
    from paper_2404_01035_gb300 import Simulation
    n, copies = 64, 8200   # 524800 rows, 65600 tiles of 8
    p = W.adjoint_well_2d(n=64)
    small = p.copy(nx=4, ny=n)
    y = np.arange(n) + 0.5
    phi = np.zeros((2, 1, n, 4))
    phi[0] = 0.5 * (1.0 + 0.6 * np.sin(2 * np.pi * y / n))[None, :, None]
    phi[1] = 1.0 - phi[0]
    mu = np.full((1, 1, n, 4), 1.634)
    grads = []
    for reps in (1, copies):
        q = small.copy(ny=n * reps, phi0=None, mu0=None)
        sim = Simulation(q, dtype="f32")
        sim.enable_checkpoints(3)
        f = lambda a: torch.tensor(np.tile(a, (1, 1, reps, 1)), device="cuda", dtype=torch.float32)  # noqa: E731
        sim.set_fields(f(phi), f(mu))
        sim.step(5)
        g = sim.grad(f(phi - 0.3), None)
        grads.append([np.asarray(v.cpu() if hasattr(v, "cpu") else v, dtype=np.float64) for v in g])
        sim.close()
    # a periodic repetition: the fields' gradients repeat, the parameters' add up
    a, b = grads
    assert np.abs(a[0]).max() > 0
    assert np.allclose(b[0], copies * a[0], rtol=1e-4, atol=1e-4 * copies * np.abs(a[0]).max())
    for k in (1, 2):
        t = np.tile(a[k], (1, 1, copies, 1))
        assert np.abs(b[k] - t).max() <= 1e-4 * np.abs(t).max()   # (forward steps of another kernel: a few roundings a step)
