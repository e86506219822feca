"""The one-gamma row kernel of the split step with many phases against the
general path (the fused kernel, which evaluates every pair)."""
import numpy as np
import pytest

import workloads as W

pytestmark = pytest.mark.gpu

# (one step with phi noise: its amplitude depends on whether a phase is exactly 0)
STEPS = 5
# per step, values up to 1 (phi) and 2 (mu) rounded a handful of times in
# either order: 4 half-units of 2 in FP32 (2^-24 each, times 2) a step
TOL = STEPS * 4 * 2 * 2.0 ** -24


def _run(prob, split, steps):
    from paper_2404_01035_gb300 import Simulation
    sim = Simulation(prob, dtype="f32")
    tiles = sim.tiles()
    sim.set_launch([i for i, t in enumerate(tiles) if t[2] == int(split)][0], 0)
    sim.set_fields(prob.phi0, prob.mu0)
    sim.step(steps)
    out = sim.get_fields()
    sim.sync()
    sim.close()
    return out


@pytest.mark.parametrize("nx,ny,nz", [(31, 5, 7), (64, 9, 8), (33, 6, 40), (161, 4, 5), (1, 9, 12)])
@pytest.mark.parametrize("kind", ["rotated", "plain_aniso", "isotropic_well", "grain_growth", "noise"])
def test_rows_equal_the_pair_form(nx, ny, nz, kind):
    p = W.small_multiphase(n=8, dim=3, N=8, NM=1, nx=nx, ny=ny, nz=nz, aniso=kind in ("rotated", "plain_aniso", "noise"),
                           rotate=kind == "rotated", potential="well" if kind == "isotropic_well" else "obstacle",
                           bc=[3, 1, 3] if kind == "rotated" else None, seed=nx + nz)
    p.gamma = 0.9 * (np.ones((8, 8)) - np.eye(8))
    p = p.copy(dt=0.5 * p.dt)
    if kind == "rotated":   # some pairs only, as grains in liquid
        p.delta[:4, :4] = 0.0
    if kind == "grain_growth":
        p = p.copy(grain_growth=1, delta=np.zeros((8, 8)))
    if kind == "noise":
        p = p.copy(noise_amp=0.05, noise_seed=3)
    steps = 1 if kind == "noise" else STEPS
    a, b = _run(p, True, steps), _run(p, False, steps)
    assert np.abs(b[0] - p.phi0).max() > 10 * TOL   # the state moved
    assert np.abs(a[0] - b[0]).max() <= TOL
    assert np.abs(a[1] - b[1]).max() <= TOL
