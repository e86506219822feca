"""The launch a 3-D FP32 context starts with (the split step) against the fused
kernel, over the forms it takes."""
import numpy as np
import pytest

import workloads as W

pytestmark = pytest.mark.gpu

STEPS = 5
# per step, values up to 1 (phi) and 2 (mu) rounded a handful of times in
# either order: 4 half-units of 2 in FP32 (2^-24 each, times 2) a step
TOL = STEPS * 4 * 2 * 2.0 ** -24


@pytest.mark.parametrize("nx,ny,nz", [(1, 5, 40), (33, 1, 9), (7, 9, 1), (130, 7, 5), (64, 12, 11)])
@pytest.mark.parametrize("N,kind", [(2, "well"), (2, "noise"), (3, "rotated"), (3, "gamma3")])
def test_default_equals_fused(nx, ny, nz, N, kind):
    from paper_2404_01035_gb300 import Simulation
    p = W.small_multiphase(n=8, dim=3, N=N, NM=N - 1, nx=nx, ny=ny, nz=nz, rotate=kind == "rotated",
                           potential="well" if kind == "well" else "obstacle", gamma3=0.4 if kind == "gamma3" else 0.0,
                           bc=[1, 3, 3] if kind == "well" else None, seed=nx + 3 * nz)
    if kind == "noise":
        p = p.copy(noise_amp=0.05, noise_seed=3)
    out = []
    for fused in (False, True):
        sim = Simulation(p, dtype="f32")
        tiles = sim.tiles()
        assert tiles[sim.launch()[0]][2] == 1
        if fused:
            sim.set_launch([i for i, t in enumerate(tiles) if t[2] == 0][0], 0)
        sim.set_fields(p.phi0, p.mu0)
        sim.step(1 if kind == "noise" else STEPS)   # noise depends on whether a phase is exactly 0
        out.append(sim.get_fields())
        sim.sync()
        sim.close()
    assert np.abs(out[0][0] - out[1][0]).max() <= TOL
    assert np.abs(out[0][1] - out[1][1]).max() <= TOL
