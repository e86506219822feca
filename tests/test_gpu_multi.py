"""The persistent multi-step launch of small 2-D grids: any split of the steps
over calls gives the same bits, and the result agrees with the grid stepped one
launch at a time (as it is with diagnostics after every step: same kernel; the
FP64 oracle fixes the values)."""
import numpy as np
import pytest

import oracle
import workloads as W

pytestmark = pytest.mark.gpu


def _run(p, dtype, parts, diag_every=0):
    from paper_2404_01035_gb300 import Simulation
    sim = Simulation(p, dtype=dtype)
    sim.set_fields(p.phi0, p.mu0)
    sim.set_diag_every(diag_every)
    for n in parts:
        sim.step(n)
    out = sim.get_fields()
    sim.sync()
    assert sim.time()[0] == sum(parts)
    sim.close()
    return out


@pytest.mark.parametrize("nx,ny", [(1, 1), (1, 40), (31, 3), (32, 9), (33, 1), (65, 70), (160, 130)])
@pytest.mark.parametrize("N,bc", [(2, [3, 3, 3]), (2, [1, 3, 3]), (3, [3, 1, 3])])
def test_split_of_the_steps_and_the_oracle(nx, ny, N, bc):
    p = W.small_multiphase(n=8, dim=2, N=N, NM=N - 1, nx=nx, ny=ny, rotate=True, bc=bc, seed=nx + ny)
    whole = _run(p, "f64", [23])
    for parts, every in (([1] * 23, 0), ([7, 16], 0), ([23], 5)):
        part = _run(p, "f64", parts, every)
        assert np.array_equal(whole[0], part[0]) and np.array_equal(whole[1], part[1])
    o = oracle.run(p, p.phi0, p.mu0, 23)
    assert max(np.abs(whole[0] - o[0]).max(), np.abs(whole[1] - o[1]).max()) <= 1e-10


@pytest.mark.parametrize("nx,ny", [(283, 282), (284, 283)])   # on either side of the FP32 limit
def test_both_sides_of_the_size_rule(nx, ny):
    p = W.binary_problem("edge", nx, ny=ny, delta=0.03, Delta=0.2, R=9.0)
    g = _run(p, "f32", [11, 9])
    o = oracle.run(p, p.phi0, p.mu0, 20)
    assert max(np.abs(g[0] - o[0]).max(), np.abs(g[1] - o[1]).max()) <= 1e-4
