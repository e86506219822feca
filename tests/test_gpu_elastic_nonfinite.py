"""An eigenstrain that is not a number makes the state non-finite, whichever phase
holds it; it is not taken for no eigenstrain."""
import numpy as np
import pytest

import workloads as W

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("phase", [0, 1])
@pytest.mark.parametrize("dtype", ["f32", "f64"])
def test_nan_eigenstrain_is_reported(phase, dtype):
    from paper_2404_01035_gb300 import Simulation
    from paper_2404_01035_gb300._binding import MSError
    p = W.small_multiphase(n=16, dim=3, N=2, NM=1, bc=[3, 3, 3], seed=6)
    C = np.zeros((6, 6))
    C[:3, :3] = 0.6
    C[range(3), range(3)] = 1.0
    C[range(3, 6), range(3, 6)] = 0.4
    eig = np.zeros((2, 3, 3))
    eig[phase] = np.nan * np.eye(3)
    sim = Simulation(p, dtype=dtype, elastic_C=C, eigenstrain=eig)
    sim.set_fields(p.phi0, p.mu0)
    sim.step(2)
    with pytest.raises(MSError, match="non-finite"):
        sim.diag()
    sim.close()
