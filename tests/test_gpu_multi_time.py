"""Steps of a small 2-D grid in a pulled temperature gradient: the time of each step
is rounded the same however the steps are spread over calls, checkpoints and
restarts."""
import numpy as np
import pytest

import workloads as W

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("dtype", ["f32", "f64"])
def test_any_split_of_the_steps_gives_the_same_bits(dtype):
    from paper_2404_01035_gb300 import Simulation
    p = W.small_multiphase(n=8, dim=2, N=3, NM=2, nx=40, ny=33, seed=5)
    p = p.copy(G=0.03, V=7.0, z0=0.0, T0=p.T_ref, dt=0.37 * p.dt)   # T - T_ref = -G V t at the origin
    out = []
    for parts in ([60], [1] * 60, [7, 13, 40], "restart"):
        sim = Simulation(p, dtype=dtype, t0=0.1)
        sim.set_fields(p.phi0, p.mu0)
        if parts == "restart":
            sim.step(23)
            blob = sim.checkpoint()
            sim.step(9)
            sim.restore(blob)
            sim.step(37)
        else:
            for n in parts:
                sim.step(n)
        out.append(sim.get_fields())
        sim.close()
    for o in out[1:]:
        assert np.array_equal(out[0][0], o[0]) and np.array_equal(out[0][1], o[1])
