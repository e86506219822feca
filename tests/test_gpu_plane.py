"""The launch a larger binary 2-D FP32 context starts with (bulk strips, then the
listed segments) against the fused kernel, over the forms it takes."""
import numpy as np
import pytest

import workloads as W

pytestmark = pytest.mark.gpu

STEPS = 5
# per step, values up to 1 (phi) and 2 (mu) rounded a handful of times in
# either order: 4 half-units of 2 in FP32 (2^-24 each, times 2) a step
TOL = STEPS * 4 * 2 * 2.0 ** -24


@pytest.mark.parametrize("nx,ny", [(1, 300100), (31, 9700), (33, 9101), (131, 2300), (160, 1900), (516, 583),
                                   (2052, 150), (2050, 151), (9999, 31), (300100, 1)])
@pytest.mark.parametrize("kind", ["obstacle", "well", "noise", "rotated"])
def test_split_equals_fused(nx, ny, kind):
    N = 2
    from paper_2404_01035_gb300 import Simulation
    p = W.small_multiphase(n=8, dim=2, N=N, NM=N - 1, nx=nx, ny=ny, rotate=kind == "rotated",
                           potential="well" if kind == "well" else "obstacle",
                           bc=[1, 3, 3] if kind == "well" else None if kind == "noise" else [3, 1, 3], seed=nx + 3 * ny)
    if kind == "noise":
        p = p.copy(noise_amp=0.05, noise_seed=3)
    # (far along y the profile's temperature would otherwise leave the model's range)
    p = p.copy(G=p.G * 16.0 / max(ny, 16))
    # stripes of one phase, 75 cells wide, with boundaries of 15 cells
    x, y = np.arange(nx)[None, :], np.arange(ny)[:, None]
    t = np.mod((x + 0.4 * y + 4.0 * np.sin(y / 9.0)) / 75.0, N)
    phi = np.stack([np.clip(5.0 * (0.6 - np.abs(np.mod(t - a + 0.5 * N, N) - 0.5 * N)), 0.0, 1.0) for a in range(N)])
    phi = (phi / phi.sum(0))[:, None]
    out = []
    for split in (1, 0):
        sim = Simulation(p, dtype="f32")
        sim.set_launch([i for i, t in enumerate(sim.tiles()) if t[2] == split][0], 0)
        sim.set_fields(phi, p.mu0)
        sim.step(1 if kind == "noise" else STEPS)   # noise depends on whether a phase is exactly 0
        out.append(sim.get_fields())
        sim.sync()
        sim.close()
    assert np.abs(out[0][0] - out[1][0]).max() <= TOL
    assert np.abs(out[0][1] - out[1][1]).max() <= TOL
