"""Batched runs at the edges of the 128-cell strips and of the 32-cell segments,
for each strip height and by units: every simulation matches its own single run."""
import numpy as np
import pytest

import workloads as W

pytestmark = pytest.mark.gpu

STEPS = 6
# per step, values up to 1 (phi) and 2 (mu) rounded a handful of times in
# either order: 4 half-units of 2 in FP32 (2^-24 each, times 2) a step
TOL = STEPS * 4 * 2 * 2.0 ** -24


@pytest.mark.parametrize("tile", [4, 8, 16, 0])   # 0: few cells in all, stepped by units
def test_strip_edges(tile):
    from paper_2404_01035_gb300 import Simulation
    from paper_2404_01035_gb300.batch import Batch
    probs = []
    for i, (nx, ny, bc) in enumerate([(1, 40, [3, 3, 3]), (40, 1, [1, 1, 3]), (31, 17, [3, 1, 3]), (32, 16, [1, 3, 3]),
                                      (64, 15, [3, 3, 3]), (127, 9, [1, 1, 3]), (128, 8, [3, 3, 3]), (129, 7, [1, 3, 3]),
                                      (256, 33, [1, 1, 3]), (260, 31, [3, 3, 3])] +
                                     ([(1111, 400, [3, 1, 3])] if tile else [])):
        probs.append(W.small_multiphase(n=8, dim=2, N=2, NM=1, nx=nx, ny=ny, bc=bc, seed=nx + ny).copy(V=0.0))
    phi = []
    for p in probs:   # stripes of one phase, 75 cells wide, with boundaries of 15 cells
        x, y = np.arange(p.nx)[None, :], np.arange(p.ny)[:, None]
        t = np.mod((x + 0.4 * y + 4.0 * np.sin(y / 9.0)) / 75.0, 2)
        f = np.clip(5.0 * (0.6 - np.abs(np.mod(t + 1.0, 2.0) - 1.0)), 0.0, 1.0)[None]
        phi.append(np.stack([f, 1.0 - f]))
    b = Batch(probs)
    b.set_tile(tile or 8)
    for i, p in enumerate(probs):
        b.set_fields(i, phi[i], p.mu0)
    b.step(STEPS)
    b.sync()
    for i, p in enumerate(probs):
        sim = Simulation(p, dtype="f32")
        sim.set_fields(phi[i], p.mu0)
        sim.step(STEPS)
        want = sim.get_fields()
        sim.close()
        got = b.get_fields(i)
        assert np.abs(got[0] - want[0]).max() <= TOL and np.abs(got[1] - want[1]).max() <= TOL, i
    b.close()
